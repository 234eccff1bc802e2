// nn.cu -- BF16 tensor-core kernels and the U-Net of the learned warm start.
//
// The network predicts, for each strain increment of a 2D specimen, the
// displacement the plain damped relaxation would add after the affine load
// step (inputs: phase map, current non-affine displacement, strain
// increment). It is trained on increments the method itself generates, and
// its prediction only moves the starting point of the relaxation, which then
// runs to the same force-residual tolerance as without it.
//
// Convolutions are implicit GEMMs on the 5th-generation tensor cores (BF16
// operands staged by TMA, FP32 accumulators in tensor memory; conv_tc.cu):
//   forward   M = pixels, N = Cout, K = taps x Cin (bias + ReLU epilogue)
//   dgrad     the forward kernel with 180-degree rotated, transposed weights
//   wgrad     M = taps x Cin, N = Cout, K = pixels, split over pixel patches,
//             partial tiles folded in a fixed order (deterministic)
// Everything else (pooling, upsampling, head, loss, Adam, data preparation)
// is plain elementwise or fixed-order reduction kernels.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "../../include/lsm_nn.h"
#include "nn_internal.h"
#include "nvtx_range.h"

namespace lsm {
namespace nn {

// The kernels between the convolutions move activations of 16 to 64 MB that
// mostly stay in L2, so what bounds them is the number of bytes a thread has
// in flight: every thread handles eight channels as one 16-byte access (all
// channel counts are multiples of 32, all slice offsets multiples of 8), and
// the reductions over pixels run beside a pass that reads the tensor anyway.

__device__ __forceinline__ uint4 ld8(const bf16 *p) { return *reinterpret_cast<const uint4 *>(p); }
__device__ __forceinline__ void st8(bf16 *p, const uint4 &v) { *reinterpret_cast<uint4 *>(p) = v; }
__device__ __forceinline__ unsigned word(const uint4 &v, int w) { return w == 0 ? v.x : w == 1 ? v.y : w == 2 ? v.z : v.w; }
// channel 2 w + h of eight packed ones
__device__ __forceinline__ float ch(const uint4 &v, int w, int h)
{
    return __uint_as_float(h ? word(v, w) & 0xffff0000u : word(v, w) << 16);
}
__device__ __forceinline__ unsigned pack2(float lo, float hi)
{
    return (unsigned)__bfloat16_as_ushort(__float2bfloat16(lo)) |
           (unsigned)__bfloat16_as_ushort(__float2bfloat16(hi)) << 16;
}
// the two channels of a gradient word where the activation's are positive, else 0
__device__ __forceinline__ unsigned relu_mask(unsigned g, unsigned a)
{
    return (__uint_as_float(a << 16) > 0.0f ? g & 0xffffu : 0u) |
           (__uint_as_float(a & 0xffff0000u) > 0.0f ? g & 0xffff0000u : 0u);
}
__device__ __forceinline__ void add2(float *acc, unsigned g)
{
    acc[0] += __uint_as_float(g << 16);
    acc[1] += __uint_as_float(g & 0xffff0000u);
}

// Pixel reductions: a block of 256 threads covers 32 channels (blockIdx.y) as
// 64 pixels x 4 groups of eight; it strides over the pixels and leaves one
// partial sum per channel, folded in a fixed order by k_fold_cols.
constexpr int RED_PIX = 64;
constexpr int RED_BLOCKS = 1216;  // 8 blocks on each of 152 SMs

static dim3 red_grid(int64_t M, int C)
{
    const int chunks = C / 32;
    const int64_t most = RED_BLOCKS / chunks > 1 ? RED_BLOCKS / chunks : 1;
    return dim3((unsigned)std::min<int64_t>((M + RED_PIX - 1) / RED_PIX, most), (unsigned)chunks);
}

// Sum of v over the warp's eight pixels (lanes of one channel group differ in bits 2 to 4).
__device__ __forceinline__ float pix_sum(float v)
{
    v += __shfl_xor_sync(0xffffffffu, v, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

// The block's sums of its 32 channels, to part[blockIdx.x][C].
__device__ __forceinline__ void red_store(const float acc[8], int C, float *__restrict__ part)
{
    __shared__ float sh[8][32];
    const int t = threadIdx.x;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const float v = pix_sum(acc[k]);
        if ((t & 31) < 4) sh[t >> 5][(t & 3) * 8 + k] = v;
    }
    __syncthreads();
    if (t < 32) {
        float s = sh[0][t];
#pragma unroll
        for (int w = 1; w < 8; w++) s += sh[w][t];
        part[(int64_t)blockIdx.x * C + blockIdx.y * 32 + t] = s;
    }
}

// Column sums of partial rows, for several segments in one launch: a block
// folds 32 columns with 32 row lanes (rows l, l + 32, ... in order, then the
// lanes in order).
struct FoldSeg {
    const float *part;
    float *out;
    int stride, cols, rows, first;  // row stride; columns; rows; first block
    float scale;
};
constexpr int MAX_SEG = 16;
struct FoldTab {
    FoldSeg s[MAX_SEG];
    int n = 0, blocks = 0;
    void add(const float *part, int stride, int cols, int rows, float scale, float *out)
    {
        s[n++] = FoldSeg{part, out, stride, cols, rows, blocks, scale};
        blocks += (cols + 31) / 32;
    }
};

__global__ void __launch_bounds__(1024) k_fold_cols(const __grid_constant__ FoldTab tab)
{
    __shared__ float sh[32][33];
    int q = 0;
    while (q + 1 < tab.n && (int)blockIdx.x >= tab.s[q + 1].first) q++;
    const FoldSeg &g = tab.s[q];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5, c = ((int)blockIdx.x - g.first) * 32 + lane;
    float s = 0.0f;
    if (c < g.cols) {
#pragma unroll 8
        for (int r = row; r < g.rows; r += 32) s += g.part[(int64_t)r * g.stride + c];
    }
    sh[row][lane] = s;
    __syncthreads();
    if (row == 0 && c < g.cols) {
        s = sh[0][lane];
#pragma unroll
        for (int l = 1; l < 32; l++) s += sh[l][lane];
        g.out[c] = s * g.scale;
    }
}

// Column sums of grad[M][C] (rows g_cs apart) as partial rows of C.
__global__ void __launch_bounds__(256) k_bias_part(const bf16 *__restrict__ grad, int g_cs, int C, int64_t M,
                                                   float *__restrict__ part)
{
    const int t = threadIdx.x, c = blockIdx.y * 32 + (t & 3) * 8;
    float acc[8] = {};
#pragma unroll 4
    for (int64_t m = (int64_t)blockIdx.x * RED_PIX + (t >> 2); m < M; m += (int64_t)gridDim.x * RED_PIX) {
        const uint4 g = ld8(grad + m * g_cs + c);
#pragma unroll
        for (int w = 0; w < 4; w++) add2(acc + 2 * w, word(g, w));
    }
    red_store(acc, C, part);
}

// Bias gradient of a convolution called by itself. The scratch holds at least
// 32 C floats (the caller's weight partials: C rows of taps x Cin >= 32).
cudaError_t bias_grad(const bf16 *grad, int g_cs, int C, int64_t M, float *db, float *scratch, size_t scratch_floats,
                      cudaStream_t st)
{
    dim3 grid = red_grid(M, C);
    grid.x = (unsigned)std::min<size_t>(grid.x, scratch_floats / C);
    k_bias_part<<<grid, 256, 0, st>>>(grad, g_cs, C, M, scratch);
    FoldTab tab;
    tab.add(scratch, C, C, (int)grid.x, 1.0f, db);
    k_fold_cols<<<tab.blocks, 1024, 0, st>>>(tab);
    return cudaGetLastError();
}

// Wr[ci][tap'][co] = W[co][taps - 1 - tap'][ci] for every convolution that
// passes a gradient on, in one launch: a block transposes one 32 x 32 tile of
// one tap through shared memory. (One launch per convolution, reading along
// co with a stride of a whole weight row, took 45 us for the 13; the pass
// moves 7.8 MB.)
struct RotSeg {
    int64_t off;
    int Cout, Cin, first;
};
struct RotTab {
    RotSeg s[MAX_SEG];
    int n = 0, blocks = 0;
};

__global__ void __launch_bounds__(256) k_rotate(const __grid_constant__ RotTab tab, const bf16 *__restrict__ W,
                                                bf16 *__restrict__ Wr)
{
    __shared__ bf16 sh[32][34];
    int q = 0;
    while (q + 1 < tab.n && (int)blockIdx.x >= tab.s[q + 1].first) q++;
    const int Cout = tab.s[q].Cout, Cin = tab.s[q].Cin;
    const int64_t off = tab.s[q].off;
    const int i = (int)blockIdx.x - tab.s[q].first, nci = Cin / 32, tap = i % 9, r = i / 9;
    const int ci0 = (r % nci) * 32, co0 = (r / nci) * 32, lane = threadIdx.x & 31, y = threadIdx.x >> 5;
#pragma unroll
    for (int j = y; j < 32; j += 8) sh[j][lane] = W[off + ((int64_t)(co0 + j) * 9 + 8 - tap) * Cin + ci0 + lane];
    __syncthreads();
#pragma unroll
    for (int j = y; j < 32; j += 8) Wr[off + ((int64_t)(ci0 + j) * 9 + tap) * Cout + co0 + lane] = sh[lane][j];
}

// ------------------------------------------------------- small kernels

// grad *= (act > 0) on a channel slice (grad dense C, act with a stride), and
// the masked gradient's channel sums, the bias gradient of the convolution
// that made act: 15 us at 524,288 pixels x 32 (one element a thread took 52 us,
// the bias sums 50 us more).
__global__ void __launch_bounds__(256) k_relu_bwd(bf16 *__restrict__ grad, int C, const bf16 *__restrict__ act,
                                                  int a_cs, int64_t M, float *__restrict__ part)
{
    const int t = threadIdx.x, c = blockIdx.y * 32 + (t & 3) * 8;
    float acc[8] = {};
#pragma unroll 2
    for (int64_t m = (int64_t)blockIdx.x * RED_PIX + (t >> 2); m < M; m += (int64_t)gridDim.x * RED_PIX) {
        uint4 g = ld8(grad + m * C + c);
        const uint4 a = ld8(act + m * a_cs + c);
        g = make_uint4(relu_mask(g.x, a.x), relu_mask(g.y, a.y), relu_mask(g.z, a.z), relu_mask(g.w, a.w));
        st8(grad + m * C + c, g);
#pragma unroll
        for (int w = 0; w < 4; w++) add2(acc + 2 * w, word(g, w));
    }
    red_store(acc, C, part);
}

// 2x2 max pool: out[b,y,x,c] = max over the window of in (channel slice)
__global__ void k_pool_fwd(const bf16 *__restrict__ in, int in_cs, bf16 *__restrict__ out, int C, int B, int H, int Wd)
{
    const unsigned Ho = H / 2, Wo = Wd / 2, G = C / 8;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= B * Ho * Wo * G) return;
    const unsigned c = (i % G) * 8, p = i / G, x = p % Wo, by = p / Wo;  // by = b Ho + y
    const bf16 *src = in + ((int64_t)2 * by * Wd + 2 * x) * in_cs + c;
    const uint4 v0 = ld8(src), v1 = ld8(src + in_cs), v2 = ld8(src + (int64_t)Wd * in_cs),
                v3 = ld8(src + (int64_t)(Wd + 1) * in_cs);
    unsigned o[4];
#pragma unroll
    for (int w = 0; w < 4; w++) {
        float m[2];
#pragma unroll
        for (int h = 0; h < 2; h++)
            m[h] = fmaxf(fmaxf(fmaxf(fmaxf(-INFINITY, ch(v0, w, h)), ch(v1, w, h)), ch(v2, w, h)), ch(v3, w, h));
        o[w] = pack2(m[0], m[1]);
    }
    st8(out + (int64_t)p * C + c, make_uint4(o[0], o[1], o[2], o[3]));
}

// Gradient of pool and skip at an encoder output: the pool's, routed to the
// first maximum of each window, plus the skip connection's (channel slice of
// a concat gradient), masked by the output's ReLU, to a dense [B][H][Wd][C]
// gradient, and its channel sums (the bias gradient). A thread takes a whole
// window, so that each tensor is read once: at 8 x 256 x 256 x 32 36 us; the
// pool's pass alone took 149 us with a thread per element, the ReLU's and the
// bias sums' 103 us more.
__global__ void __launch_bounds__(256) k_pool_bwd(const bf16 *__restrict__ gout, const bf16 *__restrict__ in,
                                                  int in_cs, const bf16 *__restrict__ gskip, int s_cs,
                                                  bf16 *__restrict__ gin, int C, int B, int H, int Wd,
                                                  float *__restrict__ part)
{
    const unsigned Wo = Wd / 2, M = (unsigned)B * (H / 2) * Wo;
    const int t = threadIdx.x, c = blockIdx.y * 32 + (t & 3) * 8;
    float acc[8] = {};
    for (unsigned p = blockIdx.x * RED_PIX + (t >> 2); p < M; p += gridDim.x * RED_PIX) {
        const unsigned x = p % Wo, by = p / Wo;
        const int64_t p0 = (int64_t)2 * by * Wd + 2 * x;  // the window's first pixel
        const uint4 go = ld8(gout + (int64_t)p * C + c);
        uint4 v[4], sk[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int64_t pq = p0 + (q >> 1) * Wd + (q & 1);
            v[q] = ld8(in + pq * in_cs + c);
            sk[q] = ld8(gskip + pq * s_cs + c);
        }
        unsigned o[4][4];
#pragma unroll
        for (int w = 0; w < 4; w++) {
            float g[4][2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                float mx = -INFINITY;
                int arg = 0;
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (ch(v[q], w, h) > mx) {
                        mx = ch(v[q], w, h);
                        arg = q;
                    }
#pragma unroll
                for (int q = 0; q < 4; q++) g[q][h] = (arg == q ? ch(go, w, h) : 0.0f) + ch(sk[q], w, h);
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                o[q][w] = relu_mask(pack2(g[q][0], g[q][1]), word(v[q], w));
                add2(acc + 2 * w, o[q][w]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
            st8(gin + (p0 + (q >> 1) * Wd + (q & 1)) * C + c, make_uint4(o[q][0], o[q][1], o[q][2], o[q][3]));
    }
    red_store(acc, C, part);
}

// nearest x2 upsampling into a channel slice of a concat tensor, a thread per
// input pixel and eight channels (84 MB at 8 x 256 x 256 x 64: 12 us, 173 us
// with a thread per output element)
__global__ void k_up_fwd(const bf16 *__restrict__ in, int C, bf16 *__restrict__ out, int out_cs, int B, int Hin,
                         int Win)
{
    const unsigned G = C / 8, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (unsigned)B * Hin * Win * G) return;
    const unsigned c = (i % G) * 8, p = i / G, x = p % Win, by = p / Win;
    const uint4 v = ld8(in + (int64_t)p * C + c);
    bf16 *dst = out + ((int64_t)4 * by * Win + 2 * x) * out_cs + c;
    const int64_t row = (int64_t)2 * Win * out_cs;
    st8(dst, v);
    st8(dst + out_cs, v);
    st8(dst + row, v);
    st8(dst + row + out_cs, v);
}

// Gradient of nearest upsampling (sum of the 2x2 block of a concat-gradient
// slice), masked by the ReLU of the upsampled activation, and its channel sums.
__global__ void __launch_bounds__(256) k_up_bwd(const bf16 *__restrict__ g, int g_cs, const bf16 *__restrict__ act,
                                                bf16 *__restrict__ gin, int C, int B, int Hin, int Win,
                                                float *__restrict__ part)
{
    const unsigned M = (unsigned)B * Hin * Win;
    const int t = threadIdx.x, c = blockIdx.y * 32 + (t & 3) * 8;
    float acc[8] = {};
    for (unsigned p = blockIdx.x * RED_PIX + (t >> 2); p < M; p += gridDim.x * RED_PIX) {
        const unsigned x = p % Win, by = p / Win;
        const bf16 *src = g + ((int64_t)4 * by * Win + 2 * x) * g_cs + c;
        const int64_t row = (int64_t)2 * Win * g_cs;
        const uint4 v0 = ld8(src), v1 = ld8(src + g_cs), v2 = ld8(src + row), v3 = ld8(src + row + g_cs);
        const uint4 a = ld8(act + (int64_t)p * C + c);
        unsigned o[4];
#pragma unroll
        for (int w = 0; w < 4; w++) {
            float s[2];
#pragma unroll
            for (int h = 0; h < 2; h++) s[h] = 0.0f + ch(v0, w, h) + ch(v1, w, h) + ch(v2, w, h) + ch(v3, w, h);
            o[w] = relu_mask(pack2(s[0], s[1]), word(a, w));
            add2(acc + 2 * w, o[w]);
        }
        st8(gin + (int64_t)p * C + c, make_uint4(o[0], o[1], o[2], o[3]));
    }
    red_store(acc, C, part);
}

constexpr int HEAD_C = 32;

// head: out[m][j] = b[j] + sum_c W[j][c] act[m][c], two outputs, FP32
__global__ void __launch_bounds__(256) k_head_fwd(const bf16 *__restrict__ act, const float *__restrict__ W,
                                                  const float *__restrict__ b, float2 *__restrict__ out, int64_t M)
{
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    uint4 v[HEAD_C / 8];
#pragma unroll
    for (int q = 0; q < HEAD_C / 8; q++) v[q] = ld8(act + m * HEAD_C + 8 * q);
    float s0 = b[0], s1 = b[1];
#pragma unroll
    for (int c = 0; c < HEAD_C; c++) {
        const float a = ch(v[c >> 3], (c & 7) >> 1, c & 1);
        s0 = fmaf(W[c], a, s0);
        s1 = fmaf(W[HEAD_C + c], a, s1);
    }
    out[m] = make_float2(s0, s1);
}

// Loss and head backward in one pass over the prediction, the target and the
// head's input: with d = pred - target, the loss terms d^2 and the output
// gradient g = 2 d / count; the gradient of the head's input gact[m][c] =
// sum_j W[j][c] g[m][j], masked by its ReLU; and per block the sums of
// g act (64), g (2), d^2 (1), to part[blockIdx.x][67], and of gact, to
// bpart[blockIdx.x][32]. It was four kernels, of which the weight sums (66
// threads a block, 4,096 pixels one after the other) took 893 us and the
// single-thread sum of the loss 84 us at 524,288 pixels; now 27 us for
// the 75 MB.
constexpr int HEAD_COLS = 2 * HEAD_C + 3;

__global__ void __launch_bounds__(256) k_head_bwd(const float2 *__restrict__ pred, const float *__restrict__ tgt,
                                                  const float *__restrict__ W, const bf16 *__restrict__ act,
                                                  bf16 *__restrict__ gact, int64_t M, float *__restrict__ part,
                                                  float *__restrict__ bpart)
{
    __shared__ float sh[8][2 * HEAD_C + 12];
    const int t = threadIdx.x, lane = t & 31, c = (t & 3) * 8;
    float w0[8], w1[8], a0[8] = {}, a1[8] = {}, ab[8] = {}, ag0 = 0.0f, ag1 = 0.0f, al = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        w0[k] = W[c + k];
        w1[k] = W[HEAD_C + c + k];
    }
    const float cnt = (float)(2 * M);
#pragma unroll 2
    for (int64_t m = (int64_t)blockIdx.x * RED_PIX + (t >> 2); m < M; m += (int64_t)gridDim.x * RED_PIX) {
        const float2 pr = pred[m];
        const uint4 a = ld8(act + m * HEAD_C + c);
        const float d0 = pr.x - tgt[2 * m], d1 = pr.y - tgt[2 * m + 1];
        const float g0 = 2.0f * d0 / cnt, g1 = 2.0f * d1 / cnt;
        al += d0 * d0;
        al += d1 * d1;
        ag0 += g0;
        ag1 += g1;
        unsigned o[4];
#pragma unroll
        for (int w = 0; w < 4; w++) {
            float v[2];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int k = 2 * w + h;
                const float x = ch(a, w, h);
                a0[k] += g0 * x;
                a1[k] += g1 * x;
                v[h] = w0[k] * g0 + w1[k] * g1;
            }
            o[w] = relu_mask(pack2(v[0], v[1]), word(a, w));
            add2(ab + 2 * w, o[w]);
        }
        st8(gact + m * HEAD_C + c, make_uint4(o[0], o[1], o[2], o[3]));
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const float s0 = pix_sum(a0[k]), s1 = pix_sum(a1[k]);
        if (lane < 4) {
            sh[t >> 5][c + k] = s0;
            sh[t >> 5][HEAD_C + c + k] = s1;
        }
    }
    // every channel group has summed the same g and d^2: group 0's go out
    const float s0 = pix_sum(ag0), s1 = pix_sum(ag1), sl = pix_sum(al);
    if (lane == 0) {
        sh[t >> 5][2 * HEAD_C] = s0;
        sh[t >> 5][2 * HEAD_C + 1] = s1;
        sh[t >> 5][2 * HEAD_C + 2] = sl;
    }
    __syncthreads();
    if (t < HEAD_COLS) {
        float s = sh[0][t];
#pragma unroll
        for (int w = 1; w < 8; w++) s += sh[w][t];
        part[(int64_t)blockIdx.x * HEAD_COLS + t] = s;
    }
    red_store(ab, HEAD_C, bpart);
}

// Adam on FP32 master parameters, refreshing the BF16 copies of the conv
// weights (bf_off < 0: the parameter has no BF16 copy).
__global__ void k_adam(float *__restrict__ w, const float *__restrict__ g, float *__restrict__ m1,
                       float *__restrict__ m2, int64_t n, float lr, float b1, float b2, float eps, float c1, float c2,
                       bf16 *__restrict__ wb, const int64_t *__restrict__ bfmap)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.0f - b1) * gi;
    const float v = b2 * m2[i] + (1.0f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = v;
    const float wi = w[i] - lr * (a / c1) / (sqrtf(v / c2) + eps);
    w[i] = wi;
    const int64_t j = bfmap[i];
    if (j >= 0) wb[j] = __float2bfloat16(wi);
}

__global__ void k_to_bf16(const float *__restrict__ w, bf16 *__restrict__ wb, const int64_t *__restrict__ bfmap,
                          int64_t n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t j = bfmap[i];
    if (j >= 0) wb[j] = __float2bfloat16(w[i]);
}

// ----------------------------------------------------- data preparation

// Network input (NHWC, 32 channels, 7 used):
//   0     phase - 1.5
//   1, 2  current non-affine displacement per unit strain: (u_x - eps (X - xc),
//         u_y) / (eps W a / 2), 0 before any load
//   3     strain increment / 1e-3
//   4     current strain / 0.1
//   5, 6  position (X - xc) / (W a / 2), (Y - yc) / (H a / 2)
// In the elastic range every increment relaxes by the same field per unit
// strain, so channels 1-2 carry most of the answer after the first increment;
// the position channels let the network place global fields (the lateral
// contraction) that the phase map alone cannot locate.
__global__ void k_prep_input(const uint8_t *__restrict__ phase, const float *__restrict__ u, const float *__restrict__ eps,
                             float deps, int S, int H, int Wd, float a, float de_scale, bf16 *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t HW = (int64_t)H * Wd;
    if (i >= S * HW) return;
    const int s = (int)(i / HW);
    const int64_t g = i - s * HW;
    const int x = (int)(g % Wd), y = (int)(g / Wd);
    const float hx = 0.5f * (Wd - 1) * a, hy = 0.5f * (H - 1) * a;
    const float e = eps[s];
    const float ux = u[(2 * s) * HW + g] - e * (x * a - hx), uy = u[(2 * s + 1) * HW + g];
    const float us = e * 0.5f * Wd * a;
    bf16 *o = out + i * 32;
    o[0] = __float2bfloat16((float)phase[i] - 1.5f);
    o[1] = __float2bfloat16(e > 0.0f ? ux / us : 0.0f);
    o[2] = __float2bfloat16(e > 0.0f ? uy / us : 0.0f);
    o[3] = __float2bfloat16(deps / de_scale);
    o[4] = __float2bfloat16(e / 0.1f);
    o[5] = __float2bfloat16((x * a - hx) / (0.5f * Wd * a));
    o[6] = __float2bfloat16((y * a - hy) / (0.5f * H * a));
    for (int c = 7; c < 32; c++) o[c] = __float2bfloat16(0.0f);
}

// Training target: the relaxation's displacement after the affine load step,
// (u_relaxed - u_loaded) / (deps * w_scale), NHWC with 2 channels.
__global__ void k_prep_target(const float *__restrict__ u_loaded, const float *__restrict__ u_relaxed, float deps,
                              float w_scale, int S, int64_t HW, float *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S * HW) return;
    const int s = (int)(i / HW);
    const int64_t g = i - s * HW;
    for (int c = 0; c < 2; c++)
        out[2 * i + c] = (u_relaxed[(2 * s + c) * HW + g] - u_loaded[(2 * s + c) * HW + g]) / (deps * w_scale);
}

// Prediction -> displacement increment [S][2][H][W]
__global__ void k_pred_to_du(const float *__restrict__ pred, float deps, float w_scale, int S, int64_t HW,
                             float *__restrict__ du)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= S * HW) return;
    const int s = (int)(i / HW);
    const int64_t g = i - s * HW;
    for (int c = 0; c < 2; c++) du[(2 * s + c) * HW + g] = pred[2 * i + c] * deps * w_scale;
}

// ------------------------------------------------------------- the U-Net

struct Conv {
    int Cin, Cout, taps;
    int64_t w_off, b_off, wb_off;  // offsets in params (FP32) and in the BF16 weight copy
};

static inline unsigned nblk(int64_t n) { return (unsigned)((n + 255) / 256); }

struct UNet {
    int H = 0, W = 0, maxB = 0;
    uint64_t seed = 0;
    cudaStream_t st = nullptr;
    bool own_stream = false;
    std::string err;
    std::vector<Conv> convs;  // e1a e1 e2a e2 e3a e3 e4a e4 d3a d3 d2a d2 d1a d1
    int64_t head_w = 0, head_b = 0;
    int64_t nparam = 0, nbf = 0;
    float *P = nullptr, *G = nullptr, *M1 = nullptr, *M2 = nullptr;
    bf16 *WB = nullptr, *WR = nullptr;  // BF16 weights, the same rotated (at the same offsets)
    int64_t *bfmap = nullptr;
    int64_t step = 0;
    // activations (NHWC bf16); the encoder outputs e1, e2, e3 live in the
    // skip slices of the decoder's concat tensors
    bf16 *e1a = nullptr, *d1c = nullptr;                 // 32; concat 96 = [up d2 0..63 | e1 64..95]
    bf16 *p1 = nullptr, *e2a = nullptr, *d2c = nullptr;  // 32 @H/2; 64; concat 192 = [up d3 | e2 128..191]
    bf16 *p2 = nullptr, *e3a = nullptr, *d3c = nullptr;  // 64 @H/4; 128; concat 384 = [up e4 | e3 256..383]
    bf16 *p3 = nullptr, *e4a = nullptr, *e4 = nullptr;   // 128 @H/8; 256; 256
    bf16 *d3a = nullptr, *d3 = nullptr, *d2a = nullptr, *d2 = nullptr, *d1a = nullptr, *d1 = nullptr;
    const bf16 *xin = nullptr;  // the last forward's input (kept for the first conv's wgrad)
    float *out = nullptr;
    bf16 *gd1c = nullptr, *gd2c = nullptr, *gd3c = nullptr;  // gradients of the concat tensors
    bf16 *ta = nullptr, *tb = nullptr;                       // gradient ping-pong (L1 x 32 each)
    float *ws = nullptr;  // wgrad scratch
    size_t ws_floats = 0;
    float *bpart = nullptr, *hpart = nullptr;  // partial rows: RED_BLOCKS x 32 per convolution; the head's
    float *loss = nullptr;
};

static const int NCONV = 14;

static void unet_free(UNet &u)
{
    void *ptrs[] = {u.P,   u.G,   u.M1,  u.M2,  u.WB,  u.WR,  u.bfmap, u.e1a, u.d1c,  u.p1,   u.e2a,
                    u.d2c, u.p2,  u.e3a, u.d3c, u.p3,  u.e4a, u.e4,    u.d3a, u.d3,   u.d2a,  u.d2,
                    u.d1a, u.d1,  u.out, u.gd1c, u.gd2c, u.gd3c, u.ta, u.tb, u.ws, u.bpart, u.hpart, u.loss};
    for (void *p : ptrs)
        if (p) cudaFree(p);
}

#define NN_TRY(x)                             \
    do {                                      \
        cudaError_t e_ = (x);                 \
        if (e_ != cudaSuccess) return e_;     \
    } while (0)

template <typename T>
static cudaError_t nalloc(T **p, size_t n)
{
    return cudaMalloc((void **)p, (n ? n : 1) * sizeof(T));
}

static cudaError_t unet_setup(UNet &u)
{
    // conv list: (Cin, Cout); every conv is 3x3, pad 1, bias + ReLU
    const int spec[NCONV][2] = {{32, 32},  {32, 32},   {32, 64},  {64, 64},  {64, 128}, {128, 128}, {128, 256},
                                {256, 256}, {384, 128}, {128, 128}, {192, 64}, {64, 64},  {96, 32},   {32, 32}};
    int64_t off = 0, boff = 0;
    for (int q = 0; q < NCONV; q++) {
        Conv c{spec[q][0], spec[q][1], 9, 0, 0, 0};
        c.w_off = off;
        off += (int64_t)c.Cout * 9 * c.Cin;
        c.b_off = off;
        off += c.Cout;
        c.wb_off = boff;
        boff += (int64_t)c.Cout * 9 * c.Cin;
        u.convs.push_back(c);
    }
    u.head_w = off;
    off += 2 * 32;
    u.head_b = off;
    off += 2;
    u.nparam = off;
    u.nbf = boff;
    // He-normal init (seeded), zero biases; the first conv sees 4 real channels
    std::vector<float> P(u.nparam, 0.0f);
    std::vector<int64_t> map(u.nparam, -1);
    std::mt19937_64 rng(u.seed);
    for (int q = 0; q < NCONV; q++) {
        const Conv &c = u.convs[q];
        const int fan_in = 9 * (q == 0 ? 7 : c.Cin);
        std::normal_distribution<float> nd(0.0f, std::sqrt(2.0f / fan_in));
        for (int64_t i = 0; i < (int64_t)c.Cout * 9 * c.Cin; i++) {
            const int ci = (int)(i % c.Cin);
            P[c.w_off + i] = (q == 0 && ci >= 7) ? 0.0f : nd(rng);
            map[c.w_off + i] = c.wb_off + i;
        }
    }
    {
        std::normal_distribution<float> nd(0.0f, 0.1f * std::sqrt(1.0f / 32));
        for (int i = 0; i < 64; i++) P[u.head_w + i] = nd(rng);
    }
    const int B = u.maxB, H = u.H, W = u.W;
    const int64_t L1 = (int64_t)B * H * W, L2 = L1 / 4, L3 = L1 / 16, L4 = L1 / 64;
    NN_TRY(nalloc(&u.P, u.nparam));
    NN_TRY(nalloc(&u.G, u.nparam));
    NN_TRY(nalloc(&u.M1, u.nparam));
    NN_TRY(nalloc(&u.M2, u.nparam));
    NN_TRY(nalloc(&u.bfmap, u.nparam));
    NN_TRY(nalloc(&u.WB, u.nbf));
    NN_TRY(nalloc(&u.WR, u.nbf));
    NN_TRY(nalloc(&u.e1a, L1 * 32));
    NN_TRY(nalloc(&u.d1c, L1 * 96));
    NN_TRY(nalloc(&u.p1, L2 * 32));
    NN_TRY(nalloc(&u.e2a, L2 * 64));
    NN_TRY(nalloc(&u.d2c, L2 * 192));
    NN_TRY(nalloc(&u.p2, L3 * 64));
    NN_TRY(nalloc(&u.e3a, L3 * 128));
    NN_TRY(nalloc(&u.d3c, L3 * 384));
    NN_TRY(nalloc(&u.p3, L4 * 128));
    NN_TRY(nalloc(&u.e4a, L4 * 256));
    NN_TRY(nalloc(&u.e4, L4 * 256));
    NN_TRY(nalloc(&u.d3a, L3 * 128));
    NN_TRY(nalloc(&u.d3, L3 * 128));
    NN_TRY(nalloc(&u.d2a, L2 * 64));
    NN_TRY(nalloc(&u.d2, L2 * 64));
    NN_TRY(nalloc(&u.d1a, L1 * 32));
    NN_TRY(nalloc(&u.d1, L1 * 32));
    NN_TRY(nalloc(&u.out, L1 * 2));
    NN_TRY(nalloc(&u.gd1c, L1 * 96));
    NN_TRY(nalloc(&u.gd2c, L2 * 192));
    NN_TRY(nalloc(&u.gd3c, L3 * 384));
    NN_TRY(nalloc(&u.ta, L1 * 32));
    NN_TRY(nalloc(&u.tb, L1 * 32));
    u.ws_floats = 16u << 20;  // 64 MiB of split partials
    NN_TRY(nalloc(&u.ws, u.ws_floats));
    NN_TRY(nalloc(&u.bpart, (size_t)NCONV * RED_BLOCKS * 32));
    NN_TRY(nalloc(&u.hpart, (size_t)RED_BLOCKS * HEAD_COLS));
    NN_TRY(nalloc(&u.loss, 1));
    NN_TRY(cudaMemcpyAsync(u.P, P.data(), u.nparam * 4, cudaMemcpyHostToDevice, u.st));
    NN_TRY(cudaMemcpyAsync(u.bfmap, map.data(), u.nparam * 8, cudaMemcpyHostToDevice, u.st));
    NN_TRY(cudaMemsetAsync(u.M1, 0, u.nparam * 4, u.st));
    NN_TRY(cudaMemsetAsync(u.M2, 0, u.nparam * 4, u.st));
    NN_TRY(cudaMemsetAsync(u.G, 0, u.nparam * 4, u.st));
    k_to_bf16<<<nblk(u.nparam), 256, 0, u.st>>>(u.P, u.WB, u.bfmap, u.nparam);
    NN_TRY(cudaStreamSynchronize(u.st));
    return cudaGetLastError();
}

static cudaError_t conv_f(UNet &u, int q, const bf16 *in, int in_cs, int in_c0, bf16 *out, int out_cs, int out_c0,
                          int B, int H, int W)
{
    const Conv &c = u.convs[q];
    return conv_fwd(in, in_cs, in_c0, c.Cin, u.WB + c.wb_off, u.P + c.b_off, out, out_cs, out_c0, c.Cout, B, H, W, 9,
                    true, u.st);
}

static cudaError_t unet_forward(UNet &u, int B, const bf16 *x0)
{
    const int H = u.H, W = u.W, H2 = H / 2, W2 = W / 2, H3 = H / 4, W3 = W / 4, H4 = H / 8, W4 = W / 8;
    const int64_t L1 = (int64_t)B * H * W, L2 = L1 / 4, L3 = L1 / 16, L4 = L1 / 64;
    u.xin = x0;
    NN_TRY(conv_f(u, 0, x0, 32, 0, u.e1a, 32, 0, B, H, W));
    NN_TRY(conv_f(u, 1, u.e1a, 32, 0, u.d1c, 96, 64, B, H, W));  // e1 -> skip slice
    k_pool_fwd<<<nblk(L2 * 32 / 8), 256, 0, u.st>>>(u.d1c + 64, 96, u.p1, 32, B, H, W);
    NN_TRY(conv_f(u, 2, u.p1, 32, 0, u.e2a, 64, 0, B, H2, W2));
    NN_TRY(conv_f(u, 3, u.e2a, 64, 0, u.d2c, 192, 128, B, H2, W2));  // e2
    k_pool_fwd<<<nblk(L3 * 64 / 8), 256, 0, u.st>>>(u.d2c + 128, 192, u.p2, 64, B, H2, W2);
    NN_TRY(conv_f(u, 4, u.p2, 64, 0, u.e3a, 128, 0, B, H3, W3));
    NN_TRY(conv_f(u, 5, u.e3a, 128, 0, u.d3c, 384, 256, B, H3, W3));  // e3
    k_pool_fwd<<<nblk(L4 * 128 / 8), 256, 0, u.st>>>(u.d3c + 256, 384, u.p3, 128, B, H3, W3);
    NN_TRY(conv_f(u, 6, u.p3, 128, 0, u.e4a, 256, 0, B, H4, W4));
    NN_TRY(conv_f(u, 7, u.e4a, 256, 0, u.e4, 256, 0, B, H4, W4));
    k_up_fwd<<<nblk(L4 * 256 / 8), 256, 0, u.st>>>(u.e4, 256, u.d3c, 384, B, H4, W4);
    NN_TRY(conv_f(u, 8, u.d3c, 384, 0, u.d3a, 128, 0, B, H3, W3));
    NN_TRY(conv_f(u, 9, u.d3a, 128, 0, u.d3, 128, 0, B, H3, W3));
    k_up_fwd<<<nblk(L3 * 128 / 8), 256, 0, u.st>>>(u.d3, 128, u.d2c, 192, B, H3, W3);
    NN_TRY(conv_f(u, 10, u.d2c, 192, 0, u.d2a, 64, 0, B, H2, W2));
    NN_TRY(conv_f(u, 11, u.d2a, 64, 0, u.d2, 64, 0, B, H2, W2));
    k_up_fwd<<<nblk(L2 * 64 / 8), 256, 0, u.st>>>(u.d2, 64, u.d1c, 96, B, H2, W2);
    NN_TRY(conv_f(u, 12, u.d1c, 96, 0, u.d1a, 32, 0, B, H, W));
    NN_TRY(conv_f(u, 13, u.d1a, 32, 0, u.d1, 32, 0, B, H, W));
    k_head_fwd<<<nblk(L1), 256, 0, u.st>>>(u.d1, u.P + u.head_w, u.P + u.head_b, (float2 *)u.out, L1);
    return cudaGetLastError();
}

// Backward of conv q: gpre = gradient at its output (already masked by its
// ReLU); writes dW into G and, if gin != nullptr, the dense input gradient.
// (db is summed by the pass that made gpre.)
static cudaError_t conv_b(UNet &u, int q, const bf16 *gpre, const bf16 *in, int in_cs, int in_c0, bf16 *gin, int B,
                          int H, int W)
{
    const Conv &c = u.convs[q];
    NN_TRY(conv_wgrad(gpre, c.Cout, c.Cout, in, in_cs, in_c0, c.Cin, B, H, W, 9, u.G + c.w_off, nullptr, u.ws,
                      u.ws_floats, u.st));
    if (gin)
        NN_TRY(conv_fwd(gpre, c.Cout, 0, c.Cout, u.WR + c.wb_off, nullptr, gin, c.Cin, 0, c.Cin, B, H, W, 9, false,
                        u.st));
    return cudaSuccess;
}

// The partial rows of conv q's bias gradient (RED_BLOCKS x 32 floats each:
// red_grid gives C / 32 times that many blocks fewer), and their fold.
static float *bias_rows(UNet &u, int q, dim3 grid, FoldTab &tab)
{
    float *part = u.bpart + (int64_t)q * RED_BLOCKS * 32;
    const Conv &c = u.convs[q];
    tab.add(part, c.Cout, c.Cout, (int)grid.x, 1.0f, u.G + c.b_off);
    return part;
}

// ReLU backward at conv q's output act
static void relu_b(UNet &u, int q, bf16 *g, const bf16 *act, int64_t M, FoldTab &tab)
{
    const int C = u.convs[q].Cout;
    const dim3 grid = red_grid(M, C);
    k_relu_bwd<<<grid, 256, 0, u.st>>>(g, C, act, C, M, bias_rows(u, q, grid, tab));
}

// Upsampling and ReLU backward at conv q's output act [B][H][W]
static void up_b(UNet &u, int q, const bf16 *g, int g_cs, const bf16 *act, bf16 *gin, int B, int H, int W, FoldTab &tab)
{
    const int C = u.convs[q].Cout;
    const dim3 grid = red_grid((int64_t)B * H * W, C);
    k_up_bwd<<<grid, 256, 0, u.st>>>(g, g_cs, act, gin, C, B, H, W, bias_rows(u, q, grid, tab));
}

// Pool, skip and ReLU backward at conv q's output, the skip slice of a concat tensor
static void pool_b(UNet &u, int q, const bf16 *gout, const bf16 *act, const bf16 *gskip, int cs, bf16 *gin, int B,
                   int H, int W, FoldTab &tab)
{
    const int C = u.convs[q].Cout;
    const dim3 grid = red_grid((int64_t)B * (H / 2) * (W / 2), C);
    k_pool_bwd<<<grid, 256, 0, u.st>>>(gout, act, cs, gskip, cs, gin, C, B, H, W, bias_rows(u, q, grid, tab));
}

// Mean squared error against target and its gradient w.r.t. every
// parameter, into G (the loss goes to u.loss).
static cudaError_t unet_backward(UNet &u, int B, const float *target)
{
    const int H = u.H, W = u.W, H2 = H / 2, W2 = W / 2, H3 = H / 4, W3 = W / 4, H4 = H / 8, W4 = W / 8;
    const int64_t L1 = (int64_t)B * H * W, L2 = L1 / 4, L3 = L1 / 16, L4 = L1 / 64;
    FoldTab tab;
    {
        RotTab rot;
        for (int q = 1; q < NCONV; q++) {  // conv 0 passes no gradient on
            const Conv &c = u.convs[q];
            rot.s[rot.n++] = RotSeg{c.wb_off, c.Cout, c.Cin, rot.blocks};
            rot.blocks += (c.Cout / 32) * (c.Cin / 32) * 9;
        }
        k_rotate<<<rot.blocks, 256, 0, u.st>>>(rot, u.WB, u.WR);
    }
    {  // loss, head weights and bias (contiguous in P), and the masked gradient of d1
        const dim3 grid = red_grid(L1, HEAD_C);
        k_head_bwd<<<grid.x, 256, 0, u.st>>>((const float2 *)u.out, target, u.P + u.head_w, u.d1, u.ta, L1, u.hpart,
                                             bias_rows(u, 13, grid, tab));
        tab.add(u.hpart, HEAD_COLS, HEAD_COLS - 1, (int)grid.x, 1.0f, u.G + u.head_w);
        tab.add(u.hpart + HEAD_COLS - 1, HEAD_COLS, 1, (int)grid.x, 1.0f / (float)(2 * L1), u.loss);
    }
    // decoder
    NN_TRY(conv_b(u, 13, u.ta, u.d1a, 32, 0, u.tb, B, H, W));
    relu_b(u, 12, u.tb, u.d1a, L1, tab);
    NN_TRY(conv_b(u, 12, u.tb, u.d1c, 96, 0, u.gd1c, B, H, W));
    up_b(u, 11, u.gd1c, 96, u.d2, u.ta, B, H2, W2, tab);
    NN_TRY(conv_b(u, 11, u.ta, u.d2a, 64, 0, u.tb, B, H2, W2));
    relu_b(u, 10, u.tb, u.d2a, L2, tab);
    NN_TRY(conv_b(u, 10, u.tb, u.d2c, 192, 0, u.gd2c, B, H2, W2));
    up_b(u, 9, u.gd2c, 192, u.d3, u.ta, B, H3, W3, tab);
    NN_TRY(conv_b(u, 9, u.ta, u.d3a, 128, 0, u.tb, B, H3, W3));
    relu_b(u, 8, u.tb, u.d3a, L3, tab);
    NN_TRY(conv_b(u, 8, u.tb, u.d3c, 384, 0, u.gd3c, B, H3, W3));
    up_b(u, 7, u.gd3c, 384, u.e4, u.ta, B, H4, W4, tab);
    // bottleneck
    NN_TRY(conv_b(u, 7, u.ta, u.e4a, 256, 0, u.tb, B, H4, W4));
    relu_b(u, 6, u.tb, u.e4a, L4, tab);
    NN_TRY(conv_b(u, 6, u.tb, u.p3, 128, 0, u.ta, B, H4, W4));
    // encoder level 3
    pool_b(u, 5, u.ta, u.d3c + 256, u.gd3c + 256, 384, u.tb, B, H3, W3, tab);
    NN_TRY(conv_b(u, 5, u.tb, u.e3a, 128, 0, u.ta, B, H3, W3));
    relu_b(u, 4, u.ta, u.e3a, L3, tab);
    NN_TRY(conv_b(u, 4, u.ta, u.p2, 64, 0, u.tb, B, H3, W3));
    // level 2
    pool_b(u, 3, u.tb, u.d2c + 128, u.gd2c + 128, 192, u.ta, B, H2, W2, tab);
    NN_TRY(conv_b(u, 3, u.ta, u.e2a, 64, 0, u.tb, B, H2, W2));
    relu_b(u, 2, u.tb, u.e2a, L2, tab);
    NN_TRY(conv_b(u, 2, u.tb, u.p1, 32, 0, u.ta, B, H2, W2));
    // level 1
    pool_b(u, 1, u.ta, u.d1c + 64, u.gd1c + 64, 96, u.tb, B, H, W, tab);
    NN_TRY(conv_b(u, 1, u.tb, u.e1a, 32, 0, u.ta, B, H, W));
    relu_b(u, 0, u.ta, u.e1a, L1, tab);
    NN_TRY(conv_b(u, 0, u.ta, u.xin, 32, 0, nullptr, B, H, W));
    k_fold_cols<<<tab.blocks, 1024, 0, u.st>>>(tab);
    return cudaGetLastError();
}

static cudaError_t unet_adam(UNet &u, float lr)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    u.step += 1;
    const float c1 = 1.0f - std::pow(b1, (float)u.step), c2 = 1.0f - std::pow(b2, (float)u.step);
    k_adam<<<nblk(u.nparam), 256, 0, u.st>>>(u.P, u.G, u.M1, u.M2, u.nparam, lr, b1, b2, eps, c1, c2, u.WB, u.bfmap);
    return cudaGetLastError();
}

}  // namespace nn
}  // namespace lsm

// =================================================================== C ABI

struct lsm_unet : public lsm::nn::UNet {};

namespace {
thread_local std::string g_nn_err;

lsm_status nfail(lsm_unet *u, lsm_status st, const std::string &m)
{
    if (u)
        u->err = m;
    else
        g_nn_err = m;
    return st;
}

lsm_status ncuda(lsm_unet *u, cudaError_t e, const char *where)
{
    return nfail(u, e == cudaErrorMemoryAllocation ? LSM_ENOMEM : LSM_ECUDA,
                 std::string(where) + ": " + cudaGetErrorString(e));
}

bool batch_ok(lsm_unet *u, int32_t b) { return u && b >= 1 && b <= u->maxB; }
}  // namespace

extern "C" {

lsm_status lsm_unet_create(int32_t height, int32_t width, int32_t max_batch, uint64_t seed, void *stream,
                           lsm_unet **out)
{
    if (!out) return nfail(nullptr, LSM_EINVAL, "out is required");
    *out = nullptr;
    if (height < 8 || width < 8 || height % 8 || width % 8 || max_batch < 1)
        return nfail(nullptr, LSM_EINVAL, "height and width must be multiples of 8 (>= 8), max_batch >= 1");
    if ((int64_t)height * width * max_batch > ((int64_t)1 << 26))
        return nfail(nullptr, LSM_EINVAL, "height * width * max_batch above 2^26 pixels");
    lsm_unet *u = new (std::nothrow) lsm_unet();
    if (!u) return nfail(nullptr, LSM_ENOMEM, "host allocation failed");
    u->H = height;
    u->W = width;
    u->maxB = max_batch;
    u->seed = seed;
    if (stream) {
        u->st = (cudaStream_t)stream;
    } else {
        if (cudaStreamCreateWithFlags(&u->st, cudaStreamNonBlocking) != cudaSuccess) {
            delete u;
            return nfail(nullptr, LSM_ECUDA, "stream create failed");
        }
        u->own_stream = true;
    }
    cudaGetLastError();
    cudaError_t e = lsm::nn::unet_setup(*u);
    if (e != cudaSuccess) {
        lsm::nn::unet_free(*u);
        if (u->own_stream) cudaStreamDestroy(u->st);
        delete u;
        return nfail(nullptr, e == cudaErrorMemoryAllocation ? LSM_ENOMEM : LSM_ECUDA,
                     std::string("unet setup: ") + cudaGetErrorString(e));
    }
    *out = u;
    return LSM_OK;
}

void lsm_unet_destroy(lsm_unet *u)
{
    if (!u) return;
    cudaStreamSynchronize(u->st);
    lsm::nn::unet_free(*u);
    if (u->own_stream) cudaStreamDestroy(u->st);
    delete u;
}

const char *lsm_unet_last_error(const lsm_unet *u) { return u ? u->err.c_str() : g_nn_err.c_str(); }

lsm_status lsm_unet_param_count(lsm_unet *u, int64_t *n)
{
    if (!u || !n) return nfail(u, LSM_EINVAL, "null argument");
    *n = u->nparam;
    return LSM_OK;
}

lsm_status lsm_unet_get_params(lsm_unet *u, float *host, int64_t n)
{
    if (!u || !host || n != u->nparam) return nfail(u, LSM_EINVAL, "need a host buffer of param_count floats");
    cudaError_t e = cudaMemcpyAsync(host, u->P, n * 4, cudaMemcpyDeviceToHost, u->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
    return e == cudaSuccess ? LSM_OK : ncuda(u, e, "get_params");
}

lsm_status lsm_unet_set_params(lsm_unet *u, const float *host, int64_t n)
{
    if (!u || !host || n != u->nparam) return nfail(u, LSM_EINVAL, "need a host buffer of param_count floats");
    cudaError_t e = cudaMemcpyAsync(u->P, host, n * 4, cudaMemcpyHostToDevice, u->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(u->M1, 0, n * 4, u->st);
    if (e == cudaSuccess) e = cudaMemsetAsync(u->M2, 0, n * 4, u->st);
    if (e == cudaSuccess) {
        lsm::nn::k_to_bf16<<<lsm::nn::nblk(n), 256, 0, u->st>>>(u->P, u->WB, u->bfmap, n);
        e = cudaStreamSynchronize(u->st);
    }
    u->step = 0;
    return e == cudaSuccess ? LSM_OK : ncuda(u, e, "set_params");
}

lsm_status lsm_unet_forward(lsm_unet *u, const void *in, float *out, int32_t batch)
{
    lsm::NvtxRange nvtx_("lsm_unet_forward");
    if (!batch_ok(u, batch) || !in || !out) return nfail(u, LSM_EINVAL, "bad arguments");
    cudaError_t e = lsm::nn::unet_forward(*u, batch, (const lsm::nn::bf16 *)in);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(out, u->out, (size_t)batch * u->H * u->W * 2 * 4, cudaMemcpyDeviceToDevice, u->st);
    return e == cudaSuccess ? LSM_OK : ncuda(u, e, "forward");
}

// LSM_ETIMEOUT if a tensor-core convolution gave up a bounded wait
static lsm_status conv_status(lsm_unet *u, cudaStream_t st = nullptr)
{
    bool t = false;
    const cudaError_t e = lsm::nn::conv_timeout(&t, u ? u->st : st);
    if (e != cudaSuccess) return ncuda(u, e, "convolution status");
    return t ? nfail(u, LSM_ETIMEOUT, "a tensor-core convolution gave up waiting for its MMAs") : LSM_OK;
}

lsm_status lsm_unet_gradients(lsm_unet *u, const void *in, const float *target, int32_t batch, float *loss,
                              float *grad)
{
    lsm::NvtxRange nvtx_("lsm_unet_gradients");
    if (!batch_ok(u, batch) || !in || !target) return nfail(u, LSM_EINVAL, "bad arguments");
    cudaError_t e = lsm::nn::unet_forward(*u, batch, (const lsm::nn::bf16 *)in);
    if (e == cudaSuccess) e = lsm::nn::unet_backward(*u, batch, target);
    if (e == cudaSuccess && loss) e = cudaMemcpyAsync(loss, u->loss, 4, cudaMemcpyDeviceToHost, u->st);
    if (e == cudaSuccess && grad) e = cudaMemcpyAsync(grad, u->G, u->nparam * 4, cudaMemcpyDeviceToHost, u->st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
    if (e != cudaSuccess) return ncuda(u, e, "gradients");
    return conv_status(u);
}

lsm_status lsm_unet_train_step(lsm_unet *u, const void *in, const float *target, int32_t batch, float lr, float *loss)
{
    lsm::NvtxRange nvtx_("lsm_unet_train_step");
    if (!batch_ok(u, batch) || !in || !target || !(lr > 0)) return nfail(u, LSM_EINVAL, "bad arguments");
    cudaError_t e = lsm::nn::unet_forward(*u, batch, (const lsm::nn::bf16 *)in);
    if (e == cudaSuccess) e = lsm::nn::unet_backward(*u, batch, target);
    if (e == cudaSuccess) e = lsm::nn::unet_adam(*u, lr);
    if (e == cudaSuccess && loss) {
        e = cudaMemcpyAsync(loss, u->loss, 4, cudaMemcpyDeviceToHost, u->st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
        if (e == cudaSuccess) return conv_status(u);
    }
    return e == cudaSuccess ? LSM_OK : ncuda(u, e, "train_step");
}

lsm_status lsm_unet_prepare_input(const uint8_t *phase, const float *u, const float *eps, float deps, int32_t S,
                                  int32_t H, int32_t W, double a, void *in, void *stream)
{
    lsm::NvtxRange nvtx_("lsm_unet_prepare_input");
    if (!phase || !u || !eps || !in || S < 1 || H < 1 || W < 1 || !(deps != 0.0f))
        return nfail(nullptr, LSM_EINVAL, "prepare_input: bad arguments");
    const int64_t n = (int64_t)S * H * W;
    const float de_scale = 1e-3f;
    lsm::nn::k_prep_input<<<lsm::nn::nblk(n), 256, 0, (cudaStream_t)stream>>>(
        phase, u, eps, deps, S, H, W, (float)a, de_scale, (lsm::nn::bf16 *)in);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LSM_OK : nfail(nullptr, LSM_ECUDA, cudaGetErrorString(e));
}

lsm_status lsm_unet_prepare_target(const float *u_loaded, const float *u_relaxed, float deps, int32_t S, int32_t H,
                                   int32_t W, double a, float *target, void *stream)
{
    if (!u_loaded || !u_relaxed || !target || S < 1 || !(deps != 0.0f))
        return nfail(nullptr, LSM_EINVAL, "prepare_target: bad arguments");
    const int64_t HW = (int64_t)H * W;
    lsm::nn::k_prep_target<<<lsm::nn::nblk(S * HW), 256, 0, (cudaStream_t)stream>>>(
        u_loaded, u_relaxed, deps, (float)(0.5 * W * a), S, HW, target);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LSM_OK : nfail(nullptr, LSM_ECUDA, cudaGetErrorString(e));
}

lsm_status lsm_unet_prediction_to_displacement(const float *pred, float deps, int32_t S, int32_t H, int32_t W,
                                               double a, float *du, void *stream)
{
    if (!pred || !du || S < 1) return nfail(nullptr, LSM_EINVAL, "prediction_to_displacement: bad arguments");
    const int64_t HW = (int64_t)H * W;
    lsm::nn::k_pred_to_du<<<lsm::nn::nblk(S * HW), 256, 0, (cudaStream_t)stream>>>(pred, deps, (float)(0.5 * W * a),
                                                                                  S, HW, du);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LSM_OK : nfail(nullptr, LSM_ECUDA, cudaGetErrorString(e));
}

lsm_status lsm_nn_conv_forward(const void *in, int32_t in_cs, int32_t in_c0, int32_t Cin, const void *W,
                               const float *bias, void *out, int32_t out_cs, int32_t out_c0, int32_t Cout, int32_t B,
                               int32_t H, int32_t Wd, int32_t taps, int32_t relu, void *stream)
{
    if (!in || !W || !out || (taps != 1 && taps != 9)) return nfail(nullptr, LSM_EINVAL, "conv_forward: bad arguments");
    const cudaError_t e = lsm::nn::conv_fwd((const lsm::nn::bf16 *)in, in_cs, in_c0, Cin, (const lsm::nn::bf16 *)W,
                                            bias, (lsm::nn::bf16 *)out, out_cs, out_c0, Cout, B, H, Wd, taps, relu != 0,
                                            (cudaStream_t)stream);
    if (e != cudaSuccess)
        return nfail(nullptr, e == cudaErrorInvalidValue ? LSM_EINVAL : LSM_ECUDA,
                     std::string("conv_forward: ") + cudaGetErrorString(e));
    return conv_status(nullptr, (cudaStream_t)stream);
}

lsm_status lsm_nn_set_wait_limit(int32_t polls, void *stream)
{
    const cudaError_t e = lsm::nn::conv_set_wait_limit(polls, (cudaStream_t)stream);
    if (e != cudaSuccess) return nfail(nullptr, LSM_ECUDA, std::string("set_wait_limit: ") + cudaGetErrorString(e));
    return LSM_OK;
}

lsm_status lsm_nn_conv_wgrad(const void *grad, int32_t Cout, const void *in, int32_t in_cs, int32_t in_c0, int32_t Cin,
                             int32_t B, int32_t H, int32_t Wd, int32_t taps, float *dW, float *db, float *scratch,
                             int64_t scratch_floats, void *stream)
{
    if (!grad || !in || !dW || !scratch || (taps != 1 && taps != 9))
        return nfail(nullptr, LSM_EINVAL, "conv_wgrad: bad arguments");
    const cudaError_t e = lsm::nn::conv_wgrad((const lsm::nn::bf16 *)grad, Cout, Cout, (const lsm::nn::bf16 *)in, in_cs,
                                              in_c0, Cin, B, H, Wd, taps, dW, db, scratch, (size_t)scratch_floats,
                                              (cudaStream_t)stream);
    return e == cudaSuccess ? LSM_OK : nfail(nullptr, LSM_EINVAL, std::string("conv_wgrad: ") + cudaGetErrorString(e));
}

}  // extern "C"
