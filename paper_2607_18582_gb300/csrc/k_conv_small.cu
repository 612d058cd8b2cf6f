// Direct convolution for layers whose per-row input fits in shared memory (the
// LeNet-5 convolutions): a block stages whole zero-padded input rows and the layer's
// weights in shared memory, and each thread computes whole 2x2 pooling windows.  The receptive-field offsets are compile-time
// constants, so the inner loop is loads with immediate offsets and FMAs.
//
// Arithmetic: every output element is the same fp32 chain as in k_stage_simt, i.e.
// acc = fma(x_k, w_k, acc) over k = (ky, kx, ci) ascending from +0 (zero-padding taps
// give x = 0), then + bias; the post-ops are the same helpers.  The two kernels give
// identical bits, so which one runs a layer does not change any result.
#include <algorithm>

#include "common.cuh"
#include "device_util.cuh"

namespace mure {

struct ConvSmallParams {
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T; int R;
    int iw;
    const float *Wt;  // [K][OC]
    const float *b;
    int act1;
    float *z; int64_t z_stride;
    float *y; int64_t y_stride;
    Overlay ov;       // mutated channels of the input rows (ov.patch null: none)
};

// The row part of a block, shared by the kernels below: where each of its rows' inputs are and
// whose mutant the row is.
struct SmallRows {
    const float *src[32];
    int g[32];
};

__device__ __forceinline__ void small_rows(const ConvSmallParams &p, SmallRows &sr, int64_t row0, int nrows)
{
    if ((int)threadIdx.x < nrows) {
        const int64_t row = row0 + threadIdx.x;
        sr.src[threadIdx.x] = p.x + (p.x_per_input ? (p.t0 + row % p.T) : row) * p.x_stride;
        sr.g[threadIdx.x] = (int)(row / p.T);
    }
    __syncthreads();
}

// The mutants' channels of the staged input rows (line floats per staged pixel row, IC per pixel,
// the image at (oy0, ox0)).
template <int IC>
__device__ __forceinline__ void small_overlay(const ConvSmallParams &p, const SmallRows &sr, int64_t row0, int nrows,
                                              float *xs, int tile, int line, int oy0, int ox0)
{
    const int per_row = p.ov.kmax * p.ov.cells;
    for (int i = threadIdx.x; i < nrows * per_row; i += blockDim.x) {
        const int rl = i / per_row, rem = i - rl * per_row, q = rem / p.ov.cells, c = rem - q * p.ov.cells;
        const int g = sr.g[rl];
        if (q >= p.ov.n_neurons[g]) continue;
        const int j = p.ov.ids[p.ov.neuron_off[g] + q];
        const int py = c / p.iw, px = c - py * p.iw;
        xs[rl * tile + (py + oy0) * line + (px + ox0) * IC + j] = p.ov.patch[(row0 + rl) * p.ov.row_stride + q * p.ov.cells + c];
    }
    __syncthreads();
}

// 5 x 5, 1 -> 6 channels, pad 2, on 28 x 28, pooled (LeNet's first layer).  A thread takes two
// neighbouring pooling windows: their 6 x 8 input field sits in registers (24 8-byte loads) and
// each tap's six weights serve 48 FMAs (a window per thread, reading its inputs tap by tap, was
// bound by its shared-memory loads, 10 for 24 FMAs: 1.08 ms for 109,000 rows, now 0.78).  16 rows of 98 pairs per block
// of 224 threads, seven rounds each; the staged lines are 36 floats, the image from column 4,
// so that rows are staged in 16-byte pieces.
constexpr int kC1Rows = 16, kC1Threads = 224, kC1Line = 36, kC1Tile = 32 * kC1Line;

__global__ void __launch_bounds__(kC1Threads, 2) k_conv1_pairs(const ConvSmallParams p)
{
    extern __shared__ __align__(16) float sm[];
    float *ws = sm;              // [25][8]
    float *xs = sm + 25 * 8;     // [rows][32][36]
    __shared__ SmallRows sr;
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * kC1Rows;
    const int nrows = (int)(p.R - row0 < kC1Rows ? p.R - row0 : kC1Rows);
    small_rows(p, sr, row0, nrows);
    for (int i = tid; i < 200; i += kC1Threads) ws[i] = (i & 7) < 6 ? __ldg(p.Wt + (i >> 3) * 6 + (i & 7)) : 0.f;
    // whole lines of nine 16-byte pieces: zero borders, the image's seven pieces between
#pragma unroll 4
    for (int i = tid; i < nrows * 288; i += kC1Threads) {
        const int rl = i / 288, e = i - rl * 288, y = e / 9, c = e - y * 9;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (y >= 2 && y < 30 && c >= 1 && c < 8)
            v = __ldg(reinterpret_cast<const float4 *>(sr.src[rl] + (y - 2) * 28) + c - 1);
        reinterpret_cast<float4 *>(xs)[i] = v;
    }
    __syncthreads();
    if (p.ov.patch) small_overlay<1>(p, sr, row0, nrows, xs, kC1Tile, kC1Line, 2, 4);
    for (int pr = tid; pr < nrows * 98; pr += kC1Threads) {
        const int rl = pr / 98, w = pr - rl * 98, py = w / 7, pp = w - py * 7;
        // inputs (2 py - 2 .. + 3, 4 pp - 2 .. + 5), staged from column 4 pp + 2
        const float *xt = xs + rl * kC1Tile + 2 * py * kC1Line + 4 * pp + 2;
        float x[6][8];
#pragma unroll
        for (int i = 0; i < 6; ++i)
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
                const float2 v = *reinterpret_cast<const float2 *>(xt + i * kC1Line + j);
                x[i][j] = v.x;
                x[i][j + 1] = v.y;
            }
        float acc[2][4][6];   // output row, column, channel
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int n = 0; n < 6; ++n) acc[d][c][n] = 0.f;
#pragma unroll
        for (int ky = 0; ky < 5; ++ky)
#pragma unroll
            for (int kx = 0; kx < 5; ++kx) {
                const float4 wa = *reinterpret_cast<const float4 *>(ws + (ky * 5 + kx) * 8);
                const float2 wb = *reinterpret_cast<const float2 *>(ws + (ky * 5 + kx) * 8 + 4);
                const float wv[6] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y};
#pragma unroll
                for (int d = 0; d < 2; ++d)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
#pragma unroll
                        for (int n = 0; n < 6; ++n) acc[d][c][n] = fmaf(x[ky + d][kx + c], wv[n], acc[d][c][n]);
            }
        const int64_t row = row0 + rl;
        float out[2][6];
#pragma unroll
        for (int n = 0; n < 6; ++n) {
            const float bias = __ldg(p.b + n);
            float v[2][4];
#pragma unroll
            for (int d = 0; d < 2; ++d)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[d][c] = acc[d][c][n] + bias;
            if (p.z) {
#pragma unroll
                for (int d = 0; d < 2; ++d)
                    *reinterpret_cast<float4 *>(p.z + row * p.z_stride + n * 784 + (2 * py + d) * 28 + 4 * pp) =
                        make_float4(v[d][0], v[d][1], v[d][2], v[d][3]);
            }
#pragma unroll
            for (int d = 0; d < 2; ++d)
#pragma unroll
                for (int c = 0; c < 4; ++c) v[d][c] = act_apply(p.act1, v[d][c]);
            out[0][n] = max4_first(v[0][0], v[0][1], v[1][0], v[1][1]);
            out[1][n] = max4_first(v[0][2], v[0][3], v[1][2], v[1][3]);
        }
        float4 *y = reinterpret_cast<float4 *>(p.y + row * p.y_stride + (py * 14 + 2 * pp) * 6);
        y[0] = make_float4(out[0][0], out[0][1], out[0][2], out[0][3]);
        y[1] = make_float4(out[0][4], out[0][5], out[1][0], out[1][1]);
        y[2] = make_float4(out[1][2], out[1][3], out[1][4], out[1][5]);
    }
}

// The other geometry, 5 x 5, 6 -> 16 channels, no padding, on 14 x 14, pooled (LeNet's second layer):
// a thread takes four output channels of a pooling window, two rows of 25 windows per block.
constexpr int kC2K = 5 * 5 * 6, kC2Oc = 16, kC2Line = 14 * 6, kC2Tile = 14 * kC2Line, kC2Rows = 2, kC2Threads = kC2Rows * 25 * 4;

__global__ void __launch_bounds__(256, 3) k_conv_small(const ConvSmallParams p)
{
    extern __shared__ __align__(16) float sm[];
    float *ws = sm;                  // [150][16]
    float *xs = sm + kC2K * kC2Oc;   // [rows][14][14][6]
    __shared__ SmallRows sr;
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * kC2Rows;
    const int nrows = (int)(p.R - row0 < kC2Rows ? p.R - row0 : kC2Rows);
    small_rows(p, sr, row0, nrows);
    for (int i = tid; i < kC2K * kC2Oc; i += kC2Threads) ws[i] = __ldg(p.Wt + i);
    // whole rows (their stride is a multiple of four) in 16-byte copies, several in flight
#pragma unroll 4
    for (int i = tid; i < nrows * (kC2Tile / 4); i += kC2Threads) {
        const int rl = i / (kC2Tile / 4), e = i - rl * (kC2Tile / 4);
        reinterpret_cast<float4 *>(xs)[i] = __ldg(reinterpret_cast<const float4 *>(sr.src[rl]) + e);
    }
    __syncthreads();
    if (p.ov.patch) small_overlay<6>(p, sr, row0, nrows, xs, kC2Tile, kC2Line, 0, 0);

    const int rl = tid / 100, cell = tid % 100 / 4, n0 = tid % 4 * 4;
    if (rl >= nrows) return;
    const int64_t row = row0 + rl;
    const int py = cell / 5, px = cell % 5;
    const float *xt = xs + rl * kC2Tile;
    int base[4];   // the window's positions
#pragma unroll
    for (int s = 0; s < 4; ++s) base[s] = (2 * py + (s >> 1)) * kC2Line + (2 * px + (s & 1)) * 6;
    float acc[4][4];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int n = 0; n < 4; ++n) acc[s][n] = 0.f;
#pragma unroll 1
    for (int ky = 0; ky < 5; ++ky)
#pragma unroll
        for (int kx = 0; kx < 5; ++kx)
#pragma unroll
            for (int ci = 0; ci < 6; ++ci) {
                const int k = (ky * 5 + kx) * 6 + ci;
                float w[4];
#pragma unroll
                for (int n = 0; n < 4; ++n) w[n] = ws[k * kC2Oc + n0 + n];
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    const float a = xt[base[s] + ky * kC2Line + kx * 6 + ci];
#pragma unroll
                    for (int n = 0; n < 4; ++n) acc[s][n] = fmaf(a, w[n], acc[s][n]);
                }
            }
#pragma unroll
    for (int nn = 0; nn < 4; ++nn) {
        const int n = n0 + nn;
        const float bias = __ldg(p.b + n);
        float v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const float zz = acc[s][nn] + bias;
            if (p.z) p.z[row * p.z_stride + n * 100 + (2 * py + (s >> 1)) * 10 + 2 * px + (s & 1)] = zz;
            v[s] = act_apply(p.act1, zz);
        }
        p.y[row * p.y_stride + cell * kC2Oc + n] = max4_first(v[0], v[1], v[2], v[3]);
    }
}

// Which layers the shared-memory kernel takes: stride 1, no residual add or GAP, and
// one of the compiled geometries.
int conv_small_variant(const Stage &S)
{
    if (S.kind != MURE_NODE_CONV2D || S.stride != 1 || S.has_add || S.gap) return 0;
    if (S.kh == 5 && S.kw == 5 && S.ic == 6 && S.oc == 16 && S.pad == 0 && S.ih == 14 && S.iw == 14 && S.pool) return 1;
    if (S.kh == 5 && S.kw == 5 && S.ic == 1 && S.oc == 6 && S.pad == 2 && S.ih == 28 && S.iw == 28 && S.pool) return 2;
    return 0;
}

int launch_conv_small(const Stage &S, Src x, RowMap rm, float *z_out, int64_t z_stride, float *y_out,
                      int64_t y_stride, cudaStream_t s, const Overlay *ov)
{
    if (rm.R <= 0) return 0;
    ConvSmallParams p{};
    if (ov) p.ov = *ov;
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.R = rm.R;
    p.iw = S.iw;
    p.Wt = S.Wt; p.b = S.b; p.act1 = S.act1;
    p.z = z_out; p.z_stride = z_stride;
    p.y = y_out; p.y_stride = y_stride;
    auto go = [&](auto kern, int rows, int threads, int floats) {
        const int smem = floats * (int)sizeof(float);
        allow_dynamic_smem(kern, smem);
        kern<<<(unsigned)((rm.R + rows - 1) / rows), threads, smem, s>>>(p);
    };
    if (S.variant == 1) go(k_conv_small, kC2Rows, kC2Threads, kC2K * kC2Oc + kC2Rows * kC2Tile);
    else go(k_conv1_pairs, kC1Rows, kC1Threads, 25 * 8 + kC1Rows * kC1Tile);
    return 1;
}

}  // namespace mure

// ------------------------------------------------ GF / WS delta, small layers --
//
// For the geometries above, the GF / WS correction sum_k e_k x_k of every output
// position is a one-channel convolution of the layer input with the mutant's patch
// vector e.  A block takes one mutant and several inputs: e and the zero-padded input
// tiles sit in shared memory and the taps are unrolled, in the generic kernel's order
// (k = (ky, kx, ci) ascending, fma chain from +0; a padding tap adds e * 0, which
// leaves the chain unchanged), so both kernels give the same bits.

namespace mure {

struct PatchDotParams {
    const float *z; int64_t z_stride; int z_per_input;   // channel-major [oc][oh*ow]
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T; int G;
    int ih, iw, oh, ow, act1;
    const int32_t *op, *n_neurons, *ids;
    const int64_t *neuron_off, *patch_off;
    const int32_t *dslot; int64_t n_dslot; int32_t dslot_g0;   // the batch's GF / WS slots
    const float *e_all;
    float *out; int64_t out_stride;
    int cells, rows_per_block;
    int oc;
};

template <int KH, int KW, int IC, int WP, int HP, int PAD, bool POOL, int KMAX>
__global__ void __launch_bounds__(256) k_patch_dot(const PatchDotParams p)
{
    constexpr int K = KH * KW * IC;
    constexpr int TILE = HP * WP * IC;
    extern __shared__ __align__(16) float sm[];
    const int g = blockIdx.x;
    const int op = p.op[g];
    if (op != MURE_OP_GF && op != MURE_OP_WS) return;
    const int k = min(p.n_neurons[g], KMAX);
    if (k <= 0) return;
    float *es = sm;               // [k][K]
    float *xs = sm + KMAX * K;    // [rows_per_block][TILE]
    const int tl0 = blockIdx.y * p.rows_per_block;
    const int nr = min(p.rows_per_block, p.T - tl0);
    const float *e = p.e_all + p.patch_off[g];
    for (int i = threadIdx.x; i < k * K; i += blockDim.x) es[i] = __ldg(e + i);
    for (int i = threadIdx.x; i < nr * TILE; i += blockDim.x) {
        const int rl = i / TILE, el = i - rl * TILE;
        const int ci = el % IC, pix = el / IC, px = pix % WP, py = pix / WP;
        const int iy = py - PAD, ix = px - PAD;
        const int64_t tl = tl0 + rl;
        float v = 0.f;
        if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
            v = __ldg(p.x + (p.x_per_input ? p.t0 + tl : (int64_t)g * p.T + tl) * p.x_stride + (iy * p.iw + ix) * IC + ci);
        xs[i] = v;
    }
    __syncthreads();
    const int32_t *ids = p.ids + p.neuron_off[g];
    const int per_row = k * p.cells;
    for (int it = threadIdx.x; it < nr * per_row; it += blockDim.x) {
        const int rl = it / per_row, rem = it - rl * per_row, q = rem / p.cells, c = rem - q * p.cells;
        const int64_t tl = tl0 + rl;
        const int64_t r = (int64_t)g * p.T + tl, t = p.t0 + tl;
        const int j = ids[q];
        const float *zr = p.z + (p.z_per_input ? t : r) * p.z_stride + (int64_t)j * (p.oh * p.ow);
        const float *xt = xs + rl * TILE;
        const float *eq = es + q * K;
        const int pw = POOL ? p.ow / 2 : p.ow;
        const int cy = c / pw, cx = c - cy * pw;
        float v4[4];
#pragma unroll
        for (int s = 0; s < (POOL ? 4 : 1); ++s) {
            const int oy = POOL ? 2 * cy + (s >> 1) : cy, ox = POOL ? 2 * cx + (s & 1) : cx;
            const float *xw = xt + (oy * WP + ox) * IC;
            float acc = 0.f;
#pragma unroll
            for (int ky = 0; ky < KH; ++ky)
#pragma unroll
                for (int kx = 0; kx < KW; ++kx)
#pragma unroll
                    for (int ci = 0; ci < IC; ++ci)
                        acc = fmaf(eq[(ky * KW + kx) * IC + ci], xw[(ky * WP + kx) * IC + ci], acc);
            v4[s] = act_apply(p.act1, zr[oy * p.ow + ox] + acc);
        }
        p.out[r * p.out_stride + q * p.cells + c] = POOL ? max4_first(v4[0], v4[1], v4[2], v4[3]) : v4[0];
    }
}

// The same values in memoized mode, one input per block: the input's padded map and
// its pre-activation maps are staged once, and every GF / WS slot of the batch (the
// mutants share the inputs) is computed from there, SMAX slots' filters at a time
// (EG: the filters are read through L1 instead of being staged).  A
// thread takes CW output cells (pooling windows: 4 CW positions) for SG slots: each
// filter tap costs 4 CW + SG shared loads (the slot loads are warp broadcasts) for
// 4 CW SG FMAs.  Every sum is the same ascending fp32 chain as in k_patch_dot, so the
// two kernels agree bit for bit.
template <int KH, int KW, int IC, int WP, int HP, int PAD, bool POOL, int CW, int SG, int SMAX, int NT, bool EG = false>
__global__ void __launch_bounds__(NT) k_patch_dot_in(const PatchDotParams p)
{
    constexpr int K = KH * KW * IC;
    constexpr int TILE = HP * WP * IC;
    constexpr int NPOS = POOL ? 4 : 1;
    constexpr int NP = CW * NPOS;          // positions per thread
    extern __shared__ __align__(16) float sm[];
    const int P = p.oh * p.ow;
    float *xs = sm;                       // [TILE] zero-padded input map
    float *es = xs + TILE;                // [SMAX][K] filter deltas (EG: read through L1 instead)
    float *zsm = es + (EG ? 0 : SMAX * K);   // [oc][P] pre-activation maps
    __shared__ int sl_g[SMAX], sl_q[SMAX], sl_j[SMAX];
    const int tl = blockIdx.x;
    const int64_t t = p.t0 + tl;
    const float *xin = p.x + t * p.x_stride;
    for (int i = threadIdx.x; i < TILE; i += NT) {
        const int ci = i % IC, pix = i / IC, px = pix % WP, py = pix / WP;
        const int iy = py - PAD, ix = px - PAD;
        xs[i] = ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw) ? __ldg(xin + (iy * p.iw + ix) * IC + ci)
                                                                                  : 0.f;
    }
    const float *zin = p.z + t * p.z_stride;
    for (int i = threadIdx.x; i < p.oc * P; i += NT) zsm[i] = __ldg(zin + i);
    const int pw = POOL ? p.ow / 2 : p.ow;
    const int chunks = (p.cells + CW - 1) / CW;
    // the batch's GF / WS slots (listed by the host), SMAX at a time
    for (int64_t s0 = 0; s0 < p.n_dslot; s0 += SMAX) {
        const int ns = (int)(p.n_dslot - s0 < SMAX ? p.n_dslot - s0 : SMAX);
        __syncthreads();
        for (int i = threadIdx.x; i < ns; i += NT) {
            const int g = p.dslot[2 * (s0 + i)] - p.dslot_g0, q = p.dslot[2 * (s0 + i) + 1];
            sl_g[i] = g;
            sl_q[i] = q;
            sl_j[i] = p.ids[p.neuron_off[g] + q];
        }
        __syncthreads();
        if (!EG) {
            for (int i = threadIdx.x; i < ns * K; i += NT) {
                const int sl = i / K, kk = i - sl * K;
                es[i] = __ldg(p.e_all + p.patch_off[sl_g[sl]] + (int64_t)sl_q[sl] * K + kk);
            }
            __syncthreads();
        }
        const int groups = (ns + SG - 1) / SG;
        for (int it = threadIdx.x; it < groups * chunks; it += NT) {
            const int sg = it / chunks, ch = it - sg * chunks;
            const int nsg = min(SG, ns - sg * SG);
            int off[NP];
#pragma unroll
            for (int w = 0; w < CW; ++w) {
                const int c = min(ch * CW + w, p.cells - 1);   // a chunk past the last cell repeats it
                const int cy = c / pw, cx = c - cy * pw;
#pragma unroll
                for (int s2 = 0; s2 < NPOS; ++s2) {
                    const int oy = POOL ? 2 * cy + (s2 >> 1) : cy, ox = POOL ? 2 * cx + (s2 & 1) : cx;
                    off[w * NPOS + s2] = (oy * WP + ox) * IC;
                }
            }
            const float *e0 = es + sg * SG * K;
            const float *eg[SG];
            if (EG) {
#pragma unroll
                for (int a = 0; a < SG; ++a) {
                    const int sl = sg * SG + (a < nsg ? a : 0);
                    eg[a] = p.e_all + p.patch_off[sl_g[sl]] + (int64_t)sl_q[sl] * K;
                }
            }
            float acc[SG][NP];
#pragma unroll
            for (int a = 0; a < SG; ++a)
#pragma unroll
                for (int q2 = 0; q2 < NP; ++q2) acc[a][q2] = 0.f;
#pragma unroll 1
            for (int ky = 0; ky < KH; ++ky)
#pragma unroll
                for (int kx = 0; kx < KW; ++kx)
#pragma unroll
                    for (int ci = 0; ci < IC; ++ci) {
                        const int kk = (ky * KW + kx) * IC + ci, xo = (ky * WP + kx) * IC + ci;
                        float xv[NP];
#pragma unroll
                        for (int q2 = 0; q2 < NP; ++q2) xv[q2] = xs[off[q2] + xo];
#pragma unroll
                        for (int a = 0; a < SG; ++a) {
                            const float ev = EG ? __ldg(eg[a] + kk) : e0[(a < nsg ? a : 0) * K + kk];
#pragma unroll
                            for (int q2 = 0; q2 < NP; ++q2) acc[a][q2] = fmaf(ev, xv[q2], acc[a][q2]);
                        }
                    }
#pragma unroll
            for (int a = 0; a < SG; ++a) {
                if (a >= nsg) break;
                const int sl = sg * SG + a;
                const float *zr = zsm + sl_j[sl] * P;
                float *orow = p.out + ((int64_t)sl_g[sl] * p.T + tl) * p.out_stride + sl_q[sl] * p.cells;
#pragma unroll
                for (int w = 0; w < CW; ++w) {
                    const int c = ch * CW + w;
                    if (c >= p.cells) break;
                    const int cy = c / pw, cx = c - cy * pw;
                    float v4[NPOS];
#pragma unroll
                    for (int s2 = 0; s2 < NPOS; ++s2) {
                        const int oy = POOL ? 2 * cy + (s2 >> 1) : cy, ox = POOL ? 2 * cx + (s2 & 1) : cx;
                        v4[s2] = act_apply(p.act1, zr[oy * p.ow + ox] + acc[a][w * NPOS + s2]);
                    }
                    orow[c] = POOL ? max4_first(v4[0], v4[1], v4[2], v4[3]) : v4[0];
                }
            }
        }
    }
}

namespace {
template <int KH, int KW, int IC, int WP, int HP, int PAD, bool POOL>
int launch_dot(const Stage &S, Src z, Src x, RowMap rm, const PatchArgs &pa, int kmax, float *out, int64_t out_stride,
               cudaStream_t s)
{
    constexpr int KMAX = 8;
    PatchDotParams p{};
    p.z = z.p; p.z_stride = z.stride; p.z_per_input = z.per_input;
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.G = rm.R / rm.T;
    p.ih = S.ih; p.iw = S.iw; p.oh = S.oh; p.ow = S.ow; p.act1 = S.act1;
    p.op = pa.op; p.n_neurons = pa.n_neurons; p.ids = pa.ids; p.neuron_off = pa.neuron_off;
    p.patch_off = pa.patch_off; p.e_all = pa.patch;
    p.dslot = pa.dslot; p.n_dslot = pa.n_dslot; p.dslot_g0 = pa.dslot_g0;
    p.out = out; p.out_stride = out_stride;
    p.cells = POOL ? (S.oh / 2) * (S.ow / 2) : S.oh * S.ow;
    p.rows_per_block = 8;
    p.oc = S.oc;
    if (z.per_input && x.per_input) {
        // memoized: one block per input, a cell and four slots per thread (measured
        // against two cells and / or eight slots per thread: more registers per thread
        // cost more in occupancy than the fewer shared loads save)
        constexpr int CW = 1, SG = 4, NT = 256;
        // the slot filters: staged in shared memory 32 slots at a time, or, where a
        // filter is long (IC > 1: 150 taps), read through L1 for all slots at once so
        // that no block runs a nearly empty last round of slots (measured: conv 6->16
        // 1.83 -> 1.65 ms per 400 mutants x 10,000 inputs; conv 1->6 slower that way)
        constexpr bool EG = IC > 1;
        constexpr int SMAX = EG ? 256 : 32;
        const size_t smem2 =
            ((size_t)HP * WP * IC + (EG ? 0 : (size_t)SMAX * KH * KW * IC) + (size_t)S.oc * S.oh * S.ow) * sizeof(float);
        if (smem2 <= 200 * 1024) {
            auto kern = k_patch_dot_in<KH, KW, IC, WP, HP, PAD, POOL, CW, SG, SMAX, NT, EG>;
            allow_dynamic_smem(kern, (int)smem2);
            kern<<<(unsigned)rm.T, NT, smem2, s>>>(p);
            return 1;
        }
    }
    const size_t smem = ((size_t)KMAX * KH * KW * IC + (size_t)p.rows_per_block * HP * WP * IC) * sizeof(float);
    allow_dynamic_smem(k_patch_dot<KH, KW, IC, WP, HP, PAD, POOL, KMAX>, (int)smem);
    const dim3 grid((unsigned)p.G, (unsigned)((rm.T + p.rows_per_block - 1) / p.rows_per_block));
    k_patch_dot<KH, KW, IC, WP, HP, PAD, POOL, KMAX><<<grid, 256, smem, s>>>(p);
    return 1;
}
}  // namespace

// GF / WS delta values for the small-layer geometries (the neuron count per mutant
// must be <= 8); 0 when the layer has no such kernel.
int patch_dot_supported(const Stage &S, int kmax) { return S.geo > 0 && kmax <= 8 && !S.has_add && !S.gap; }

int launch_patch_dot(const Stage &S, Src z, Src x, RowMap rm, const PatchArgs &pa, int kmax, float *out,
                     int64_t out_stride, cudaStream_t s)
{
    if (rm.R <= 0) return 0;
    switch (S.geo) {
    case 1: return launch_dot<5, 5, 6, 14, 14, 0, true>(S, z, x, rm, pa, kmax, out, out_stride, s);
    case 2: return launch_dot<5, 5, 1, 32, 32, 2, true>(S, z, x, rm, pa, kmax, out, out_stride, s);
    }
    return 0;
}

}  // namespace mure
