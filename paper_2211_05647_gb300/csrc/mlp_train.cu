// mlp_train.cu -- loss and gradient of the closure network on the tensor
// cores: a cluster of four CTAs per 128-row tile of the batch (batches of many
// tiles: one CTA) runs the forward pass and the whole backward pass of its tile on mma.sync BF16 tiles with FP32
// accumulation, and writes the tile's gradient; a second kernel sums the tiles'
// gradients in a fixed order.
//
// Loss L = mean_b (y_b - t_b)^2.  Backward, straight through the forward's BF16
// roundings (h1 and W2 as the forward's MMAs used them):
//   dy_b = 2 (y_b - t_b) / B                      (rows past the batch: 0)
//   dW3 = h2^T dy, db3 = sum dy                    (column sums, FP32)
//   dz2 = (dy w3^T) * GELU'(z2), db2 = colsum dz2
//   dW2 = h1^T dz2                                 MMA, M = K = N = 128 (K over the tile's rows)
//   dh1 = dz2 W2^T, dz1 = dh1 * GELU'(z1)          MMA, K = 128
//   dW1 = x^T dz1, db1 = colsum dz1                MMA, M = 32 (17 used), K over the rows
// dz2 and dz1 enter the MMAs rounded to BF16; z1, z2 and the column sums stay
// FP32.  The transposed operands (h1^T, x^T as A; dz2, dz1 as B over rows)
// are read with ldmatrix .trans from the row-major tiles.
//
// A minibatch of 4096 rows is 32 tiles: one CTA a tile left four fifths of the SMs
// idle and each tile a serial chain of 29 us, half of it the conversion of the
// weights and the gather of the rows.  Now
//  * a CTA of the cluster takes 32 rows through the row-wise phases (a warp 16 rows
//    x 32 columns), hands its h1, dz2 and dz1 to the others through distributed
//    shared memory, and forms a quarter of dW2 (by k) and of dW1 (by n), each over
//    all 128 rows.  Every sum keeps its order: the accumulation of an MMA
//    over the tile's rows, y over a row's columns, a column over a warp's sixteen rows and
//    then over the eight groups of them;
//  * the weights reach it as BF16 images in the layout of its shared memory and the
//    rows as BF16 tiles, prepared outside: in training by the kernel that applies the
//    previous minibatch's gradient, which holds every new weight anyway, and in blocks
//    of its own copies the next minibatch's rows and finds the places of the one after
//    that in the epoch's permutation (a walk of a few microseconds, off the path).
// Two launches a minibatch of 4096: 35.9 -> 12.8 us.  Bound by the latency of the
// phases (the contractions are 0.2 us of the tensor cores).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "cp_async.cuh"
#include "mlp_tc.cuh"
#include "shuffle.cuh"

namespace cg = cooperative_groups;

namespace fp {

constexpr int kTrainStride = kMlpNParams + 1;   // per tile: the packed gradient, then the tile's loss sum
constexpr int kTrainCtas = 4;                   // CTAs a tile
constexpr int kTrainRows = kMlpRows / kTrainCtas;   // rows a CTA takes through the row-wise phases
constexpr int kTrainCols = kMlpH / kTrainCtas;      // hidden units whose dW2 rows / dW1 columns it forms
constexpr int kLdS = kTrainCols + 8;            // padded pitch of a 32-column slice

// BF16 operands of the parameters, as the tile kernel's shared memory holds them
struct alignas(16) TrainWeights {
    __nv_bfloat16 w1t[kMlpH][kLd1];    // w1t[n][k] = W1[k][n] (k >= 17 zero): B of layer 1
    __nv_bfloat16 w2t[kMlpH][kLd2];    // w2t[n][k] = W2[k][n]: B of layer 2
    __nv_bfloat16 w2n[kMlpH][kLd2];    // w2n[k][n] = W2[k][n]: B of dh1 = dz2 W2^T
};
// one tile's inputs (cols >= 17 zero, rows past the batch zero)
struct alignas(16) TrainTile {
    __nv_bfloat16 x[kMlpRows][kLd1];
};

struct MlpTrainSmem {
    TrainWeights w;
    TrainTile t;
    __nv_bfloat16 h1[kTrainRows][kLd2];       // h1 of the CTA's rows
    __nv_bfloat16 h1s[kMlpRows][kLdS];        // h1 of every row, the CTA's 32 columns
    __nv_bfloat16 dz2[kMlpRows][kLd2];        // dz2 of every row
    __nv_bfloat16 dz1s[kMlpRows][kLdS];       // dz1 of every row, the CTA's 32 columns
    float yt[kTrainRows][4][17];              // y's terms of a row by lane of the quad and column tile
    float y[kTrainRows];
    float b1[kMlpH], b2[kMlpH], w3[kMlpH];
    float colsum[3][8][kMlpH];                // per 16 rows: dW3, db2, db1 partial column sums (first CTA's is used)
    float loss[8], dyb[8];
    float b3;
};

// workspace after the tiles' gradients: the weights, the tiles' rows, their targets, and two minibatches' sample
// indices
struct TrainWs {
    float *grad;
    TrainWeights *w;
    TrainTile *x;
    float *t;
    int64_t *src[2];
};
size_t train_align(size_t b) { return (b + 255) & ~(size_t)255; }
size_t train_ws_bytes(int64_t tiles)
{
    return train_align((size_t)tiles * kTrainStride * sizeof(float)) + train_align(sizeof(TrainWeights)) +
           (size_t)tiles * (sizeof(TrainTile) + kMlpRows * (sizeof(float) + 2 * sizeof(int64_t))) + 256;
}
TrainWs train_ws(void *workspace, int64_t tiles)
{
    char *p = reinterpret_cast<char *>(((uintptr_t)workspace + 255) & ~(uintptr_t)255);
    TrainWs w{};
    w.grad = reinterpret_cast<float *>(p);
    p += train_align((size_t)tiles * kTrainStride * sizeof(float));
    w.w = reinterpret_cast<TrainWeights *>(p);
    p += train_align(sizeof(TrainWeights));
    w.x = reinterpret_cast<TrainTile *>(p);
    p += (size_t)tiles * sizeof(TrainTile);
    w.src[0] = reinterpret_cast<int64_t *>(p);
    w.src[1] = w.src[0] + tiles * kMlpRows;
    w.t = reinterpret_cast<float *>(w.src[1] + tiles * kMlpRows);
    return w;
}

// the BF16 operands parameter i appears in
__device__ __forceinline__ void put_weight(TrainWeights *w, int i, float v)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    if (i < kOffB1) {
        w->w1t[i % kMlpH][i / kMlpH] = b;
    } else if (i >= kOffW2 && i < kOffB2) {
        const int q = i - kOffW2, k = q / kMlpH, n = q % kMlpH;
        w->w2t[n][k] = b;
        w->w2n[k][n] = b;
    }
}

// row r of the batch (B rows, padded to whole tiles) -> its tile: sample src (r past the batch: zeros).  Eight
// threads a row, five columns each.
__device__ __forceinline__ void put_row(const TrainWs &ws, const float *__restrict__ X, const float *__restrict__ T,
                                        int64_t B, int64_t r, int part, int64_t src)
{
    __nv_bfloat16 *o = ws.x[r / kMlpRows].x[r % kMlpRows];
#pragma unroll
    for (int q = 0; q < kLd1 / 8; ++q) {
        const int k = part * (kLd1 / 8) + q;
        o[k] = __float2bfloat16_rn(k < kMlpIn && r < B ? X[src * kMlpIn + k] : 0.0f);
    }
    if (part == 0) ws.t[r] = r < B ? T[src] : 0.0f;
}

// Blocks of 256 threads: the parameters', then 32 rows each, then the places of 256 rows each.
constexpr int kParamBlocks = (kMlpNParams + 1 + 255) / 256;
unsigned copy_blocks(int64_t tiles) { return (unsigned)(tiles * kMlpRows / 32); }
unsigned place_blocks(int64_t tiles) { return (unsigned)((tiles * kMlpRows + 255) / 256); }

// the first minibatch: BF16 weights, its rows (with use_perm samples perm(row)) and, when there is a second, the
// places of that one's rows
__global__ void __launch_bounds__(256) k_mlp_train_prepare(const float *__restrict__ P, const float *__restrict__ X,
                                                           const float *__restrict__ T, int64_t B, int64_t padded,
                                                           unsigned copies, TrainWs ws, Perm perm, int use_perm)
{
    pdl_enter();
    const unsigned b = blockIdx.x;
    if (b < kParamBlocks) {
        const int i = b * 256 + threadIdx.x;
        if (i < kMlpNParams) put_weight(ws.w, i, P[i]);
        for (int q = i; q < kMlpH * (kLd1 - kMlpIn); q += kParamBlocks * 256)   // w1t's unused columns
            ws.w->w1t[q / (kLd1 - kMlpIn)][kMlpIn + q % (kLd1 - kMlpIn)] = __float2bfloat16_rn(0.0f);
    } else if (b < kParamBlocks + copies) {
        const int64_t r = (int64_t)(b - kParamBlocks) * 32 + (threadIdx.x >> 3);
        put_row(ws, X, T, B, r, (int)(threadIdx.x & 7),
                use_perm && r < B ? (int64_t)perm_index((uint64_t)r, perm) : r);
    } else {
        const int64_t r = (int64_t)(b - kParamBlocks - copies) * 256 + threadIdx.x;
        if (r < B) ws.src[1][r] = (int64_t)perm_index((uint64_t)(B + r), perm);
    }
}

__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], const __nv_bfloat16 *row)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(row)));
}

// Sum of the two rows a thread holds for fragment column pair (c0, c1), then
// over the 8 row groups of the warp (lanes with equal t); lanes 0..3 store.
__device__ __forceinline__ void warp_colsum(float *dst, int col, float v0, float v1, int lane)
{
#pragma unroll
    for (int off = 4; off < 32; off <<= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, off);
        v1 += __shfl_xor_sync(0xffffffffu, v1, off);
    }
    if (lane < 4) {
        dst[col] = v0;
        dst[col + 1] = v1;
    }
}

// a tile's sums over its eight 16-row groups: dW3, db2, db1; db3 and the loss
__device__ __forceinline__ void tile_colsums(const float (*colsum)[8][kMlpH], const float *loss, const float *dyb,
                                             float *out, int tid)
{
    if (tid < kMlpH) {
        float a = 0.0f, b = 0.0f, c = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            a += colsum[0][w][tid];
            b += colsum[1][w][tid];
            c += colsum[2][w][tid];
        }
        out[kOffW3 + tid] = a;
        out[kOffB2 + tid] = b;
        out[kOffB1 + tid] = c;
    }
    if (tid == 0) {
        float l = 0.0f, d = 0.0f;
        for (int w = 0; w < 8; ++w) {
            l += loss[w];
            d += dyb[w];
        }
        out[kOffB3] = d;
        out[kMlpNParams] = l;
    }
}

// One 128-row tile per cluster of kTrainCtas CTAs (256 threads each) of a batch of B rows; writes
// ws.grad[tile][0 .. kMlpNParams) = the tile's gradient contribution and [kMlpNParams] = its sum of squared
// residuals / B.
__global__ void __cluster_dims__(kTrainCtas, 1, 1) __launch_bounds__(256, 1)
    k_mlp_train_tile(const float *__restrict__ P, TrainWs ws, int64_t B)
{
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    MlpTrainSmem &s = *reinterpret_cast<MlpTrainSmem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int rank = (int)cluster.block_rank();
    const int64_t tile = blockIdx.x / kTrainCtas;
    const int rg = warp >> 2, cgp = warp & 3;      // the warp's 16 rows and 32 columns in the row-wise phases
    const int l0 = rg * 16;                        // first row, of the CTA's
    const int r0 = rank * kTrainRows + l0;         // and of the tile's
    const int grp = rank * 2 + rg;                 // 16-row group of the tile
    float *out = ws.grad + tile * kTrainStride;
    MlpTrainSmem *peer[kTrainCtas];
#pragma unroll
    for (int c = 0; c < kTrainCtas; ++c) peer[c] = cluster.map_shared_rank(&s, c);
    MlpTrainSmem *const slice = cluster.map_shared_rank(&s, cgp);   // the CTA that takes this warp's columns

    cluster.barrier_arrive();   // started: the others may write this CTA's shared memory (waited for below)
    pdl_enter();
    // ---- weights and the input tile, as prepared (W2's second copy, needed last, as a group of its own)
    const unsigned char *gw = reinterpret_cast<const unsigned char *>(ws.w);
    const unsigned char *gx = reinterpret_cast<const unsigned char *>(ws.x + tile);
    for (int i = tid; i < (int)(sizeof(TrainTile) / 16); i += 256)
        cpa16(reinterpret_cast<unsigned char *>(&s.t) + 16 * i, gx + 16 * i);
    constexpr int kFirst = (int)(offsetof(TrainWeights, w2n) / 16);
    for (int i = tid; i < kFirst; i += 256) cpa16(reinterpret_cast<unsigned char *>(&s.w) + 16 * i, gw + 16 * i);
    cpa_commit();
    for (int i = kFirst + tid; i < (int)(sizeof(TrainWeights) / 16); i += 256)
        cpa16(reinterpret_cast<unsigned char *>(&s.w) + 16 * i, gw + 16 * i);
    cpa_commit();
    const int64_t row = tile * kMlpRows + r0 + g;   // the thread's rows: row and row + 8
    const float ta = row < B ? ws.t[row] : 0.0f, tb = row + 8 < B ? ws.t[row + 8] : 0.0f;
    for (int i = tid; i < kMlpH; i += 256) {
        s.b1[i] = P[kOffB1 + i];
        s.b2[i] = P[kOffB2 + i];
        s.w3[i] = P[kOffW3 + i];
    }
    if (tid == 0) s.b3 = P[kOffB3];
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();            // the first copies of every thread have landed
    cluster.barrier_wait();

    // ---- forward, layer 1: h1 = gelu(z1) -> shared (BF16); z1 is formed again, bit for bit, where
    //      GELU'(z1) is needed, rather than kept in registers
    uint32_t xa[2][4];   // the warp's rows of x as A fragments (K = 32: two k steps)
#pragma unroll
    for (int ks = 0; ks < kMlpK1 / 16; ++ks) {
        xa[ks][0] = ld_b32(&s.t.x[r0 + g][ks * 16 + 2 * t]);
        xa[ks][1] = ld_b32(&s.t.x[r0 + g + 8][ks * 16 + 2 * t]);
        xa[ks][2] = ld_b32(&s.t.x[r0 + g][ks * 16 + 2 * t + 8]);
        xa[ks][3] = ld_b32(&s.t.x[r0 + g + 8][ks * 16 + 2 * t + 8]);
    }
    auto z1_tile = [&](int nt, float (&z)[4]) {
        z[0] = z[1] = z[2] = z[3] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kMlpK1 / 16; ++ks)
            mma_bf16_16816(z, xa[ks], ld_b32(&s.w.w1t[nt * 8 + g][ks * 16 + 2 * t]),
                           ld_b32(&s.w.w1t[nt * 8 + g][ks * 16 + 2 * t + 8]));
        const int col = nt * 8 + 2 * t;
        z[0] += s.b1[col];
        z[1] += s.b1[col + 1];
        z[2] += s.b1[col];
        z[3] += s.b1[col + 1];
    };
    const int nt0 = cgp * 4;   // the warp's column tiles
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float z[4];
        z1_tile(nt0 + q, z);
        const int col = (nt0 + q) * 8 + 2 * t, cs = q * 8 + 2 * t;
        const uint32_t lo = pack_bf16(gelu_f(z[0]), gelu_f(z[1])), hi = pack_bf16(gelu_f(z[2]), gelu_f(z[3]));
        *reinterpret_cast<uint32_t *>(&s.h1[l0 + g][col]) = lo;
        *reinterpret_cast<uint32_t *>(&s.h1[l0 + g + 8][col]) = hi;
        *reinterpret_cast<uint32_t *>(&slice->h1s[r0 + g][cs]) = lo;       // whose dW2 rows these columns are
        *reinterpret_cast<uint32_t *>(&slice->h1s[r0 + g + 8][cs]) = hi;
    }
    __syncthreads();

    // ---- forward, layer 2 (the warp's rows and columns) and the terms of y
    float z2[4][4];
#pragma unroll
    for (int q = 0; q < 4; ++q) z2[q][0] = z2[q][1] = z2[q][2] = z2[q][3] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < kMlpH / 16; ++ks) {
        uint32_t a[4];
        a[0] = ld_b32(&s.h1[l0 + g][ks * 16 + 2 * t]);
        a[1] = ld_b32(&s.h1[l0 + g + 8][ks * 16 + 2 * t]);
        a[2] = ld_b32(&s.h1[l0 + g][ks * 16 + 2 * t + 8]);
        a[3] = ld_b32(&s.h1[l0 + g + 8][ks * 16 + 2 * t + 8]);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            mma_bf16_16816(z2[q], a, ld_b32(&s.w.w2t[(nt0 + q) * 8 + g][ks * 16 + 2 * t]),
                           ld_b32(&s.w.w2t[(nt0 + q) * 8 + g][ks * 16 + 2 * t + 8]));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int col = (nt0 + q) * 8 + 2 * t;
        z2[q][0] += s.b2[col];
        z2[q][1] += s.b2[col + 1];
        z2[q][2] += s.b2[col];
        z2[q][3] += s.b2[col + 1];
        s.yt[l0 + g][t][nt0 + q] = gelu_f(z2[q][0]) * s.w3[col] + gelu_f(z2[q][1]) * s.w3[col + 1];
        s.yt[l0 + g + 8][t][nt0 + q] = gelu_f(z2[q][2]) * s.w3[col] + gelu_f(z2[q][3]) * s.w3[col + 1];
    }
    __syncthreads();
    if (tid < 4 * kTrainRows) {   // four threads a row: its columns in order, then across the quad
        const int row = tid >> 2;
        float y = 0.0f;
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) y += s.yt[row][t][nt];
        y += __shfl_xor_sync(0xffffffffu, y, 1);
        y += __shfl_xor_sync(0xffffffffu, y, 2);
        if (t == 0) s.y[row] = y;
    }
    __syncthreads();
    const float e0 = row < B ? s.y[l0 + g] + s.b3 - ta : 0.0f;
    const float e1 = row + 8 < B ? s.y[l0 + g + 8] + s.b3 - tb : 0.0f;
    const float dy0 = 2.0f * e0 / (float)B, dy1 = 2.0f * e1 / (float)B;

    // ---- dW3 = h2^T dy, dz2 = dy w3 GELU'(z2) (-> every CTA's shared memory, BF16), db2 = colsum dz2
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int col = (nt0 + q) * 8 + 2 * t;
        warp_colsum(peer[0]->colsum[0][grp], col, gelu_f(z2[q][0]) * dy0 + gelu_f(z2[q][2]) * dy1,
                    gelu_f(z2[q][1]) * dy0 + gelu_f(z2[q][3]) * dy1, lane);
        const float d00 = dy0 * s.w3[col] * gelu_grad_f(z2[q][0]);
        const float d01 = dy0 * s.w3[col + 1] * gelu_grad_f(z2[q][1]);
        const float d10 = dy1 * s.w3[col] * gelu_grad_f(z2[q][2]);
        const float d11 = dy1 * s.w3[col + 1] * gelu_grad_f(z2[q][3]);
        warp_colsum(peer[0]->colsum[1][grp], col, d00 + d10, d01 + d11, lane);
        const uint32_t lo = pack_bf16(d00, d01), hi = pack_bf16(d10, d11);
#pragma unroll
        for (int c = 0; c < kTrainCtas; ++c) {
            *reinterpret_cast<uint32_t *>(&peer[c]->dz2[r0 + g][col]) = lo;
            *reinterpret_cast<uint32_t *>(&peer[c]->dz2[r0 + g + 8][col]) = hi;
        }
    }
    if (cgp == 0) {
        float l = e0 * e0 + e1 * e1, d = dy0 + dy1;
        if (t != 0) l = d = 0.0f;   // every lane of a quad holds the same two rows
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, off);
            d += __shfl_xor_sync(0xffffffffu, d, off);
        }
        if (lane == 0) {
            peer[0]->loss[grp] = l / (float)B;
            peer[0]->dyb[grp] = d;
        }
    }
    cpa_wait_all();   // W2's second copy, with the barrier
    cluster.sync();   // h1 slices and dz2 of every row are here

    // ---- dh1 = dz2 W2^T for the warp's rows and columns, dz1 = dh1 GELU'(z1) (-> the CTA whose columns these are)
    {
        float dh[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) dh[q][0] = dh[q][1] = dh[q][2] = dh[q][3] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kMlpH / 16; ++ks) {
            uint32_t a[4];
            a[0] = ld_b32(&s.dz2[r0 + g][ks * 16 + 2 * t]);
            a[1] = ld_b32(&s.dz2[r0 + g + 8][ks * 16 + 2 * t]);
            a[2] = ld_b32(&s.dz2[r0 + g][ks * 16 + 2 * t + 8]);
            a[3] = ld_b32(&s.dz2[r0 + g + 8][ks * 16 + 2 * t + 8]);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                mma_bf16_16816(dh[q], a, ld_b32(&s.w.w2n[(nt0 + q) * 8 + g][ks * 16 + 2 * t]),
                               ld_b32(&s.w.w2n[(nt0 + q) * 8 + g][ks * 16 + 2 * t + 8]));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int col = (nt0 + q) * 8 + 2 * t, cs = q * 8 + 2 * t;
            float z[4];
            z1_tile(nt0 + q, z);
            const float d00 = dh[q][0] * gelu_grad_f(z[0]), d01 = dh[q][1] * gelu_grad_f(z[1]);
            const float d10 = dh[q][2] * gelu_grad_f(z[2]), d11 = dh[q][3] * gelu_grad_f(z[3]);
            warp_colsum(peer[0]->colsum[2][grp], col, d00 + d10, d01 + d11, lane);
            *reinterpret_cast<uint32_t *>(&slice->dz1s[r0 + g][cs]) = pack_bf16(d00, d01);
            *reinterpret_cast<uint32_t *>(&slice->dz1s[r0 + g + 8][cs]) = pack_bf16(d10, d11);
        }
    }
    // arrive now, wait after dW2, which needs none of it (the last exchange: a CTA may leave after the wait)
    cluster.barrier_arrive();

    const int q3 = lane >> 3, rr = lane & 7;
    // ---- dW2[k][n] = sum_b h1[b][k] dz2[b][n] for the CTA's 32 k: warp (rg, cgp) forms 16 of them x 32 n
    {
        float acc[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kMlpRows / 16; ++ks) {
            const int b0 = ks * 16;
            uint32_t a[4];   // A(k, b) = h1[b][k]: blocks (b lo/hi) x (k lo/hi) in the a0..a3 order
            ldsm_x4_trans(a, &s.h1s[b0 + ((q3 >> 1) << 3) + rr][rg * 16 + ((q3 & 1) << 3)]);
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                uint32_t bq[4];   // B(b, n) = dz2[b][n]: (nt, b lo), (nt, b hi), (nt + 1, b lo), (nt + 1, b hi)
                ldsm_x4_trans(bq, &s.dz2[b0 + ((q3 & 1) << 3) + rr][(nt0 + q + (q3 >> 1)) * 8]);
                mma_bf16_16816(acc[q], a, bq[0], bq[1]);
                mma_bf16_16816(acc[q + 1], a, bq[2], bq[3]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int col = (nt0 + q) * 8 + 2 * t;
            float *o = out + kOffW2 + (rank * kTrainCols + rg * 16 + g) * kMlpH + col;
            *reinterpret_cast<float2 *>(o) = make_float2(acc[q][0], acc[q][1]);
            *reinterpret_cast<float2 *>(o + 8 * kMlpH) = make_float2(acc[q][2], acc[q][3]);
        }
    }
    cluster.barrier_wait();   // dz1 slices and every column sum are here

    // ---- dW1[k][n] = sum_b x[b][k] dz1[b][n] (k < 17) for the CTA's 32 n: warp (rg, cgp) forms the 16-row block
    //      k in [16 rg, +16) for one n tile
    {
        float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int ks = 0; ks < kMlpRows / 16; ++ks) {
            const int b0 = ks * 16;
            uint32_t a[4], bq[4];
            ldsm_x4_trans(a, &s.t.x[b0 + ((q3 >> 1) << 3) + rr][rg * 16 + ((q3 & 1) << 3)]);
            // the n tile in both halves of the load: (b lo), (b hi) twice
            ldsm_x4_trans(bq, &s.dz1s[b0 + ((q3 & 1) << 3) + rr][cgp * 8]);
            mma_bf16_16816(acc, a, bq[0], bq[1]);
        }
        const int col = rank * kTrainCols + cgp * 8 + 2 * t;
        const int k_lo = rg * 16 + g, k_hi = k_lo + 8;
        if (k_lo < kMlpIn)
            *reinterpret_cast<float2 *>(out + kOffW1 + k_lo * kMlpH + col) = make_float2(acc[0], acc[1]);
        if (k_hi < kMlpIn)
            *reinterpret_cast<float2 *>(out + kOffW1 + k_hi * kMlpH + col) = make_float2(acc[2], acc[3]);
    }

    // ---- column sums over the 16-row groups: dW3, db2, db1; db3 and the loss
    if (rank == 0) tile_colsums(s.colsum, s.loss, s.dyb, out, tid);
}

// The same for batches of more tiles than a wave of clusters takes (launch_train_tile): one tile a CTA, a warp its 16
// rows through every phase, nothing exchanged between CTAs.  The values are the cluster's, sum for sum.  Bound by the
// tile's phases as the cluster is (262 144 rows, 2048 tiles: 0.35 ms a minibatch, 80 TFLOP/s).
struct MlpTrainSmem1 {
    TrainWeights w;
    TrainTile t;
    __nv_bfloat16 h1[kMlpRows][kLd2];     // h1, later dz1 (once dW2 is formed)
    __nv_bfloat16 dz2[kMlpRows][kLd2];
    float b1[kMlpH], b2[kMlpH], w3[kMlpH];
    float colsum[3][8][kMlpH];            // per warp: dW3, db2, db1 partial column sums
    float loss[8], dyb[8];
    float b3;
};

__global__ void __launch_bounds__(256, 1) k_mlp_train_tile1(const float *__restrict__ P, TrainWs ws, int64_t B)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    MlpTrainSmem1 &s = *reinterpret_cast<MlpTrainSmem1 *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int r0 = warp * 16;
    const int64_t tile = blockIdx.x;
    float *out = ws.grad + tile * kTrainStride;

    pdl_enter();
    const unsigned char *gw = reinterpret_cast<const unsigned char *>(ws.w);
    const unsigned char *gx = reinterpret_cast<const unsigned char *>(ws.x + tile);
    for (int i = tid; i < (int)(sizeof(TrainTile) / 16); i += 256)
        cpa16(reinterpret_cast<unsigned char *>(&s.t) + 16 * i, gx + 16 * i);
    for (int i = tid; i < (int)(sizeof(TrainWeights) / 16); i += 256)
        cpa16(reinterpret_cast<unsigned char *>(&s.w) + 16 * i, gw + 16 * i);
    cpa_commit();
    const int64_t row = tile * kMlpRows + r0 + g;   // the thread's rows: row and row + 8
    const float ta = row < B ? ws.t[row] : 0.0f, tb = row + 8 < B ? ws.t[row + 8] : 0.0f;
    for (int i = tid; i < kMlpH; i += 256) {
        s.b1[i] = P[kOffB1 + i];
        s.b2[i] = P[kOffB2 + i];
        s.w3[i] = P[kOffW3 + i];
    }
    if (tid == 0) s.b3 = P[kOffB3];
    cpa_wait_all();
    __syncthreads();

    // ---- forward, layer 1: h1 = gelu(z1) -> shared (BF16)
    uint32_t xa[2][4];   // the warp's rows of x as A fragments (K = 32: two k steps)
#pragma unroll
    for (int ks = 0; ks < kMlpK1 / 16; ++ks) {
        xa[ks][0] = ld_b32(&s.t.x[r0 + g][ks * 16 + 2 * t]);
        xa[ks][1] = ld_b32(&s.t.x[r0 + g + 8][ks * 16 + 2 * t]);
        xa[ks][2] = ld_b32(&s.t.x[r0 + g][ks * 16 + 2 * t + 8]);
        xa[ks][3] = ld_b32(&s.t.x[r0 + g + 8][ks * 16 + 2 * t + 8]);
    }
    auto z1_tile = [&](int nt, float (&z)[4]) {
        z[0] = z[1] = z[2] = z[3] = 0.0f;
#pragma unroll
        for (int ks = 0; ks < kMlpK1 / 16; ++ks)
            mma_bf16_16816(z, xa[ks], ld_b32(&s.w.w1t[nt * 8 + g][ks * 16 + 2 * t]),
                           ld_b32(&s.w.w1t[nt * 8 + g][ks * 16 + 2 * t + 8]));
        const int col = nt * 8 + 2 * t;
        z[0] += s.b1[col];
        z[1] += s.b1[col + 1];
        z[2] += s.b1[col];
        z[3] += s.b1[col + 1];
    };
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) {
        float z[4];
        z1_tile(nt, z);
        const int col = nt * 8 + 2 * t;
        *reinterpret_cast<uint32_t *>(&s.h1[r0 + g][col]) = pack_bf16(gelu_f(z[0]), gelu_f(z[1]));
        *reinterpret_cast<uint32_t *>(&s.h1[r0 + g + 8][col]) = pack_bf16(gelu_f(z[2]), gelu_f(z[3]));
    }
    __syncwarp();

    // ---- forward, layer 2 (the warp's own rows of h1) and the output y
    float z2[16][4];
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) z2[nt][0] = z2[nt][1] = z2[nt][2] = z2[nt][3] = 0.0f;
#pragma unroll 2
    for (int ks = 0; ks < kMlpH / 16; ++ks) {
        uint32_t a[4];
        a[0] = ld_b32(&s.h1[r0 + g][ks * 16 + 2 * t]);
        a[1] = ld_b32(&s.h1[r0 + g + 8][ks * 16 + 2 * t]);
        a[2] = ld_b32(&s.h1[r0 + g][ks * 16 + 2 * t + 8]);
        a[3] = ld_b32(&s.h1[r0 + g + 8][ks * 16 + 2 * t + 8]);
#pragma unroll
        for (int nt = 0; nt < 16; ++nt)
            mma_bf16_16816(z2[nt], a, ld_b32(&s.w.w2t[nt * 8 + g][ks * 16 + 2 * t]),
                           ld_b32(&s.w.w2t[nt * 8 + g][ks * 16 + 2 * t + 8]));
    }
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) {
        const int col = nt * 8 + 2 * t;
        z2[nt][0] += s.b2[col];
        z2[nt][1] += s.b2[col + 1];
        z2[nt][2] += s.b2[col];
        z2[nt][3] += s.b2[col + 1];
        y0 += gelu_f(z2[nt][0]) * s.w3[col] + gelu_f(z2[nt][1]) * s.w3[col + 1];
        y1 += gelu_f(z2[nt][2]) * s.w3[col] + gelu_f(z2[nt][3]) * s.w3[col + 1];
    }
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    const float e0 = row < B ? y0 + s.b3 - ta : 0.0f;
    const float e1 = row + 8 < B ? y1 + s.b3 - tb : 0.0f;
    const float dy0 = 2.0f * e0 / (float)B, dy1 = 2.0f * e1 / (float)B;

    // ---- dW3 = h2^T dy, dz2 = dy w3 GELU'(z2) (-> shared, BF16), db2 = colsum dz2
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) {
        const int col = nt * 8 + 2 * t;
        warp_colsum(s.colsum[0][warp], col, gelu_f(z2[nt][0]) * dy0 + gelu_f(z2[nt][2]) * dy1,
                    gelu_f(z2[nt][1]) * dy0 + gelu_f(z2[nt][3]) * dy1, lane);
        const float d00 = dy0 * s.w3[col] * gelu_grad_f(z2[nt][0]);
        const float d01 = dy0 * s.w3[col + 1] * gelu_grad_f(z2[nt][1]);
        const float d10 = dy1 * s.w3[col] * gelu_grad_f(z2[nt][2]);
        const float d11 = dy1 * s.w3[col + 1] * gelu_grad_f(z2[nt][3]);
        warp_colsum(s.colsum[1][warp], col, d00 + d10, d01 + d11, lane);
        *reinterpret_cast<uint32_t *>(&s.dz2[r0 + g][col]) = pack_bf16(d00, d01);
        *reinterpret_cast<uint32_t *>(&s.dz2[r0 + g + 8][col]) = pack_bf16(d10, d11);
    }
    {
        float l = e0 * e0 + e1 * e1, d = dy0 + dy1;
        if (t != 0) l = d = 0.0f;   // every lane of a quad holds the same two rows
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            l += __shfl_xor_sync(0xffffffffu, l, off);
            d += __shfl_xor_sync(0xffffffffu, d, off);
        }
        if (lane == 0) {
            s.loss[warp] = l / (float)B;
            s.dyb[warp] = d;
        }
    }
    __syncthreads();

    const int q3 = lane >> 3, rr = lane & 7;
    // ---- dW2[k][n] = sum_b h1[b][k] dz2[b][n]: the warp forms rows k in [16 warp, +16)
    {
        float acc[16][4];
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.0f;
#pragma unroll 2
        for (int ks = 0; ks < kMlpRows / 16; ++ks) {
            const int b0 = ks * 16;
            uint32_t a[4];   // A(k, b) = h1[b][k]: blocks (b lo/hi) x (k lo/hi) in the a0..a3 order
            ldsm_x4_trans(a, &s.h1[b0 + ((q3 >> 1) << 3) + rr][r0 + ((q3 & 1) << 3)]);
#pragma unroll
            for (int nt = 0; nt < 16; nt += 2) {
                uint32_t bq[4];   // B(b, n) = dz2[b][n]: (nt, b lo), (nt, b hi), (nt + 1, b lo), (nt + 1, b hi)
                ldsm_x4_trans(bq, &s.dz2[b0 + ((q3 & 1) << 3) + rr][(nt + (q3 >> 1)) * 8]);
                mma_bf16_16816(acc[nt], a, bq[0], bq[1]);
                mma_bf16_16816(acc[nt + 1], a, bq[2], bq[3]);
            }
        }
#pragma unroll
        for (int nt = 0; nt < 16; ++nt) {
            const int col = nt * 8 + 2 * t;
            float *o = out + kOffW2 + (r0 + g) * kMlpH + col;
            *reinterpret_cast<float2 *>(o) = make_float2(acc[nt][0], acc[nt][1]);
            *reinterpret_cast<float2 *>(o + 8 * kMlpH) = make_float2(acc[nt][2], acc[nt][3]);
        }
    }

    // ---- dh1 = dz2 W2^T for the warp's own rows, dz1 = dh1 GELU'(z1)
    float dh[16][4];
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) dh[nt][0] = dh[nt][1] = dh[nt][2] = dh[nt][3] = 0.0f;
#pragma unroll 2
    for (int ks = 0; ks < kMlpH / 16; ++ks) {
        uint32_t a[4];
        a[0] = ld_b32(&s.dz2[r0 + g][ks * 16 + 2 * t]);
        a[1] = ld_b32(&s.dz2[r0 + g + 8][ks * 16 + 2 * t]);
        a[2] = ld_b32(&s.dz2[r0 + g][ks * 16 + 2 * t + 8]);
        a[3] = ld_b32(&s.dz2[r0 + g + 8][ks * 16 + 2 * t + 8]);
#pragma unroll
        for (int nt = 0; nt < 16; ++nt)
            mma_bf16_16816(dh[nt], a, ld_b32(&s.w.w2n[nt * 8 + g][ks * 16 + 2 * t]),
                           ld_b32(&s.w.w2n[nt * 8 + g][ks * 16 + 2 * t + 8]));
    }
    __syncthreads();   // every warp has read h1 (dW2) before dz1 takes its place
#pragma unroll
    for (int nt = 0; nt < 16; ++nt) {
        const int col = nt * 8 + 2 * t;
        float z[4];
        z1_tile(nt, z);
        const float d00 = dh[nt][0] * gelu_grad_f(z[0]), d01 = dh[nt][1] * gelu_grad_f(z[1]);
        const float d10 = dh[nt][2] * gelu_grad_f(z[2]), d11 = dh[nt][3] * gelu_grad_f(z[3]);
        warp_colsum(s.colsum[2][warp], col, d00 + d10, d01 + d11, lane);
        *reinterpret_cast<uint32_t *>(&s.h1[r0 + g][col]) = pack_bf16(d00, d01);
        *reinterpret_cast<uint32_t *>(&s.h1[r0 + g + 8][col]) = pack_bf16(d10, d11);
    }
    __syncthreads();

    // ---- dW1[k][n] = sum_b x[b][k] dz1[b][n] (k < 17): the warp forms the 16-row block k in [16 (warp & 1), +16) for
    //      the n tiles [4 (warp >> 1), +4)
    {
        const int mt = warp & 1, n0 = (warp >> 1) * 4;
        float acc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;
#pragma unroll 2
        for (int ks = 0; ks < kMlpRows / 16; ++ks) {
            const int b0 = ks * 16;
            uint32_t a[4];
            ldsm_x4_trans(a, &s.t.x[b0 + ((q3 >> 1) << 3) + rr][mt * 16 + ((q3 & 1) << 3)]);
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                uint32_t bq[4];
                ldsm_x4_trans(bq, &s.h1[b0 + ((q3 & 1) << 3) + rr][(n0 + j + (q3 >> 1)) * 8]);
                mma_bf16_16816(acc[j], a, bq[0], bq[1]);
                mma_bf16_16816(acc[j + 1], a, bq[2], bq[3]);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int col = (n0 + j) * 8 + 2 * t;
            const int k_lo = mt * 16 + g, k_hi = k_lo + 8;
            if (k_lo < kMlpIn)
                *reinterpret_cast<float2 *>(out + kOffW1 + k_lo * kMlpH + col) = make_float2(acc[j][0], acc[j][1]);
            if (k_hi < kMlpIn)
                *reinterpret_cast<float2 *>(out + kOffW1 + k_hi * kMlpH + col) = make_float2(acc[j][2], acc[j][3]);
        }
    }

    tile_colsums(s.colsum, s.loss, s.dyb, out, tid);
}

// grad[i] = sum over tiles (in tile order) of ws[tile][i]; loss = sum of ws[tile][kMlpNParams]
__device__ __forceinline__ float tile_sum(const float *__restrict__ ws, int ntiles, int i)
{
    float a = 0.0f;
#pragma unroll 16
    for (int q = 0; q < ntiles; ++q) a += ws[(int64_t)q * kTrainStride + i];
    return a;
}

__global__ void __launch_bounds__(256) k_mlp_train_reduce(const float *__restrict__ ws, int ntiles,
                                                          float *__restrict__ grad, float *__restrict__ loss)
{
    pdl_enter();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i > kMlpNParams) return;
    const float a = tile_sum(ws, ntiles, i);
    if (i < kMlpNParams) grad[i] = a;
    else *loss = a;
}

// the same sum per parameter followed by its Adam step (step count t: c1, c2), and the minibatch's loss
// added to *loss_acc times loss_scale; the new weights' BF16 operands.  Blocks past the parameters' copy the rows of
// the next minibatch (places in `next`), those past them find the places of the one after that (rows first .. of
// the permuted order) for `after`.
__global__ void __launch_bounds__(256)
    k_mlp_train_reduce_adam(TrainWs ws, int ntiles, float *__restrict__ P, float *__restrict__ m,
                            float *__restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2,
                            double *__restrict__ loss_acc, double loss_scale, const float *__restrict__ X,
                            const float *__restrict__ T, int64_t B, unsigned copies, const int64_t *next,
                            int64_t *after, Perm perm, int64_t first)
{
    const unsigned b = blockIdx.x;
    if (b >= kParamBlocks + copies) {   // its buffer was last read two launches ago
        const int64_t r = (int64_t)(b - kParamBlocks - copies) * 256 + threadIdx.x;
        const int64_t at = r < B ? (int64_t)perm_index((uint64_t)(first + r), perm) : 0;
        pdl_enter();
        if (r < B) after[r] = at;
        return;
    }
    pdl_enter();
    if (b >= kParamBlocks) {
        const int64_t r = (int64_t)(b - kParamBlocks) * 32 + (threadIdx.x >> 3);
        put_row(ws, X, T, B, r, (int)(threadIdx.x & 7), r < B ? next[r] : 0);
        return;
    }
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i > kMlpNParams) return;
    const float a = tile_sum(ws.grad, ntiles, i);
    if (i < kMlpNParams) {
        adam_update(P, m, v, i, a, lr, b1, b2, eps, c1, c2);
        put_weight(ws.w, i, P[i]);
    } else {
        *loss_acc += (double)a * loss_scale;
    }
}

// places: the places of the second minibatch's rows too
cudaError_t launch_train_prepare(cudaStream_t st, const float *P, const float *X, const float *T, int64_t B,
                                 const TrainWs &ws, int64_t tiles, const Perm *perm, bool places)
{
    const unsigned copies = copy_blocks(tiles);
    return launch_pdl(k_mlp_train_prepare, dim3(kParamBlocks + copies + (places ? place_blocks(tiles) : 0u)), dim3(256),
                      0, st, P, X, T, B, tiles * kMlpRows, copies, ws, perm ? *perm : Perm{}, perm ? 1 : 0);
}

// A cluster takes a tile in some 11 us, a CTA in some 20, on a quarter of the SMs: the clusters are ahead while one wave
// of them does (us a minibatch of an epoch, clusters / CTAs: 32 tiles 18.2 / 25.2, 48 27.4 / 28.1, 64 28.3 / 27.8,
// 76 36.9 / 30.8, 128 43.4 / 29.9, 512 138 / 87.9, 2048 556 / 352).
cudaError_t launch_train_tile(cudaStream_t st, const float *P, int64_t B, const TrainWs &ws, int64_t tiles)
{
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool clusters = 8 * tiles <= 3 * sms;
    const size_t smem = clusters ? sizeof(MlpTrainSmem) : sizeof(MlpTrainSmem1);
    auto kern = clusters ? k_mlp_train_tile : k_mlp_train_tile1;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(kern, dim3((unsigned)tiles * (clusters ? kTrainCtas : 1)), dim3(256), smem, st, P, ws, B);
}

}  // namespace fp

using namespace fp;

extern "C" {

size_t fdtd_mlp_workspace_bytes(int64_t batch)
{
    if (batch < 1) return 0;
    const int64_t tiles = (batch + kMlpRows - 1) / kMlpRows;
    return train_ws_bytes(tiles);
}

int fdtd_mlp_loss_grad(const float *params, const float *x, const float *target, int64_t batch, float *grad,
                       float *loss, void *workspace, size_t workspace_bytes, void *stream)
{
    if (!params || !x || !target || !grad || !loss || !workspace || batch < 1)
        return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_loss_grad: bad argument");
    if (workspace_bytes < fdtd_mlp_workspace_bytes(batch))
        return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_loss_grad: workspace too small");
    const int64_t tiles = (batch + kMlpRows - 1) / kMlpRows;
    if (tiles > (1 << 24)) return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_loss_grad: batch too large");
    cudaStream_t st = (cudaStream_t)stream;
    const TrainWs ws = train_ws(workspace, tiles);
    cudaError_t e = launch_train_prepare(st, params, x, target, batch, ws, tiles, nullptr, false);
    if (e == cudaSuccess) e = launch_train_tile(st, params, batch, ws, tiles);
    if (e == cudaSuccess)
        e = launch_pdl(k_mlp_train_reduce, dim3(kParamBlocks), dim3(256), 0, st, (const float *)ws.grad, (int)tiles,
                       grad, loss);
    if (e != cudaSuccess) return fp_set_global_error(FDTD_ERR_CUDA, cudaGetErrorString(e));
    return FDTD_OK;
}

size_t fdtd_mlp_train_workspace_bytes(int64_t batch) { return fdtd_mlp_workspace_bytes(batch); }

int fdtd_mlp_train_epoch(float *params, float *grad, float *m, float *v, const float *x, const float *t, int64_t n,
                         int64_t batch, uint64_t seed, int64_t epoch, int64_t iter0, int64_t total_iters, double lr,
                         double beta1, double beta2, double eps, double *loss_mean, void *workspace,
                         size_t workspace_bytes, void *stream)
{
    (void)grad;   // the fused reduction applies each tile-summed gradient directly
    if (!params || !m || !v || !x || !t || !loss_mean || !workspace || batch < 1 || n < batch ||
        n > (int64_t)1 << 40 || epoch < 0 || iter0 < 0 || total_iters < 1 || !(lr > 0) || !std::isfinite(lr))
        return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_train_epoch: bad argument (need n >= batch >= 1)");
    if (workspace_bytes < fdtd_mlp_train_workspace_bytes(batch))
        return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_train_epoch: workspace too small");
    const int64_t tiles = (batch + kMlpRows - 1) / kMlpRows;
    if (tiles > (1 << 24)) return fp_set_global_error(FDTD_ERR_INVAL, "fdtd_mlp_train_epoch: batch too large");
    cudaStream_t st = (cudaStream_t)stream;
    const TrainWs ws = train_ws(workspace, tiles);
    cudaError_t e = cudaMemsetAsync(loss_mean, 0, sizeof(double), st);
    if (e != cudaSuccess) return fp_set_global_error(FDTD_ERR_CUDA, cudaGetErrorString(e));
    const int64_t nb = n / batch;   // the ragged tail of the permuted order is left out this epoch
    const Perm p = make_perm(n, seed, epoch);
    e = launch_train_prepare(st, params, x, t, batch, ws, tiles, &p, nb > 1);
    for (int64_t b = 0; b < nb && e == cudaSuccess; ++b) {
        e = launch_train_tile(st, params, batch, ws, tiles);
        if (e != cudaSuccess) break;
        const int64_t it = iter0 + b;
        const double lr_t = lr * 0.5 * (1.0 + std::cos(kPi * (double)std::min(it, total_iters) / (double)total_iters));
        const double c1 = 1.0 - std::pow(beta1, (double)(it + 1)), c2 = 1.0 - std::pow(beta2, (double)(it + 1));
        const unsigned copies = b + 1 < nb ? copy_blocks(tiles) : 0u, places = b + 2 < nb ? place_blocks(tiles) : 0u;
        e = launch_pdl(k_mlp_train_reduce_adam, dim3(kParamBlocks + copies + places), dim3(256), 0, st, ws, (int)tiles,
                       params, m, v, (float)lr_t, (float)beta1, (float)beta2, (float)eps, (float)c1, (float)c2,
                       loss_mean, 1.0 / (double)nb, x, t, batch, copies, (const int64_t *)ws.src[(b + 1) & 1],
                       ws.src[b & 1], p, (b + 2) * batch);
    }
    if (e != cudaSuccess) return fp_set_global_error(FDTD_ERR_CUDA, cudaGetErrorString(e));
    return FDTD_OK;
}

}  // extern "C"
