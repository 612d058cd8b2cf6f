// Layer kernels of the FP32 arithmetic: implicit-GEMM convolution / dense on the
// CUDA cores, the output layer with the fused argmax / compare / kill epilogue, and
// small row-movement kernels.
//
// Determinism contract (what makes memoized == vanilla bit for bit): every output
// element z[row][pos][n] is the fp32 FMA chain acc = fma(x_k, w_k, acc) over the
// fan-in k = (ky, kx, ci) in ascending order starting from +0 (zero-padding taps
// contribute x = 0), then z = acc + b[n].  Nothing depends on the batch size, the
// tile a row lands in or the number of mutants, so one row gives the same bits in
// the cache build, in a vanilla prefix and in a memoized suffix.
#include <algorithm>

#include "common.cuh"
#include "device_util.cuh"
#include "epilogue.cuh"
#include "simt_tile.cuh"

namespace mure {

struct StageParams {
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T; int R;
    const int32_t *lrow;   // compacted batch: logical rows (per-input reads), else null
    int ih, iw, ic, kh, kw, stride, pad, oh, ow, oc, K;
    const float *Wt;  // [K][oc]
    const float *b;
    int act1, has_add, act2, pool;
    const float *skip; int64_t skip_stride; int skip_per_input; int sk_w, sk_c, sk_stride;
    float *z; int64_t z_stride;
    float *y; int64_t y_stride;
    int P;   // GEMM rows per batch row: oh*ow, ordered (oy, ox), or with pooling
             // 4 * (oh/2) * (ow/2) ordered (py, px, dy, dx)
    int pw;  // pooled width
    int n_tiles;   // column tiles (blockIdx.x: row tile * n_tiles + column tile)
    int vec;       // 16-byte stores of y: channels in fours on 16-byte rows
    Overlay ov;    // mutated channels of the input rows (ov.patch null: none)
};

// Implicit-GEMM convolution / dense on the CUDA cores: BM rows (positions) x BN output
// channels per block, TM x TN sums per thread (simt_tile.cuh), operand tiles
// double-buffered in shared memory, the next pieces in flight while the current are used.  A4: the
// input channels come in fours on 16-byte rows, so a thread fetches four k of its row at once.
// OV (with A4 only): a fetched piece takes the mutated channels from the patch (where: see
// simt_overlay_inline).  Measured on LeNet-5 in fp32 (1,500 x 150, FC 400-120 and 120-84): 0.88 ms
// with 4 x 4 sums per thread and rows materialised first, 0.69 now; what bounds it is the latency
// of a tile's loads (few tiles per SM at these sizes) and 84 or 120 outputs in 128 columns.
template <int BM, int BN, int TM, int TN, bool A4, bool OV>
__global__ void __launch_bounds__(BM / TM * (BN / TN), A4 && !OV && BN != 64 ? 4 : 3) k_stage_simt(const StageParams p)
{
    constexpr int BK = 8, CT = BN / TN, RT = BM / TM, NT = CT * RT;
    constexpr int RS = BM / (TM / 4), CS = BN / (TN / 4);
    constexpr int A4N = BM * BK / 4 / NT, B4N = (BK * BN / 4 + NT - 1) / NT;
    __shared__ __align__(16) float2 As[2][BK][BM];
    __shared__ __align__(16) float Bs[2][BK][BN];
    const int tid = threadIdx.x;
    constexpr int CL = CT < 8 ? CT : 8, RL = 32 / CL;
    const int warp = tid >> 5, lane = tid & 31;
    const int tn = (warp % (CT / CL)) * CL + lane % CL, tm = (warp / (CT / CL)) * RL + lane / CL;
    const unsigned mt = blockIdx.x / (unsigned)p.n_tiles;
    const int n0 = (int)(blockIdx.x - mt * p.n_tiles) * BN;
    // the tile's first batch row and position
    const int64_t m0 = (int64_t)mt * BM, row0 = m0 / p.P;
    const unsigned q0 = (unsigned)(m0 - row0 * p.P);
    auto place = [&](int i, int64_t &row, int &py, int &px, int &oy, int &ox) {
        const unsigned qq = q0 + i, dr = qq / (unsigned)p.P, q = qq - dr * p.P;
        row = row0 + dr;
        if (p.pool) {
            const unsigned w = q >> 2, sub = q & 3;
            py = w / (unsigned)p.pw;
            px = w - py * p.pw;
            oy = 2 * py + (sub >> 1);
            ox = 2 * px + (sub & 1);
        } else {
            py = px = 0;
            oy = q / (unsigned)p.ow;
            ox = q - oy * p.ow;
        }
    };
    // this thread's A row: tid % BM
    const float *xrow = nullptr, *ov_row = nullptr;
    int iy0 = 0, ix0 = 0, ov_n = 0;
    const int32_t *ov_ids = nullptr;
    {
        int64_t row;
        int py, px, oy, ox;
        place(tid % BM, row, py, px, oy, ox);
        if (row < p.R) {
            iy0 = oy * p.stride - p.pad;
            ix0 = ox * p.stride - p.pad;
            const int64_t lr = logical_row(p.lrow, row);
            xrow = p.x + (p.x_per_input ? p.t0 + lr % p.T : row) * p.x_stride;
            if (OV) {
                const int g = (int)(lr / p.T);
                ov_n = p.ov.n_neurons[g];
                ov_ids = p.ov.ids + p.ov.neuron_off[g];
                ov_row = p.ov.patch + lr * p.ov.row_stride;
            }
        }
    }
    float4 ra[A4N], rb[B4N];
    // where this thread's next A pieces stand in the fan-in: channel and tap, advanced by BK a
    // tile (a division per piece and tile took longer than the tile's FMAs)
    int ci[A4N] = {}, kx[A4N] = {}, ky[A4N] = {};
    auto carry = [&](int i) {
        while (ci[i] >= p.ic) {
            ci[i] -= p.ic;
            if (++kx[i] == p.kw) { kx[i] = 0; ++ky[i]; }
        }
    };
#pragma unroll
    for (int i = 0; i < A4N; ++i) {
        kx[i] = ky[i] = 0;
        ci[i] = 4 * (tid / BM + i * (NT / BM));
        carry(i);
    }
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < A4N; ++i) {
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (xrow && ky[i] < p.kh) {
                if (A4) {
                    const int iy = iy0 + ky[i], ix = ix0 + kx[i];
                    if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw) {
                        const int e = (iy * p.iw + ix) * p.ic + ci[i];
                        *reinterpret_cast<float4 *>(v) = __ldg(reinterpret_cast<const float4 *>(xrow + e));
                        if (OV && ov_n > 0) {
                            const int c = e / p.ov.ch, j = e - c * p.ov.ch;   // four channels of one cell
                            for (int q = 0; q < ov_n; ++q) {
                                const int d = __ldg(ov_ids + q) - j;
#pragma unroll
                                for (int u = 0; u < 4; ++u)
                                    if (d == u) v[u] = __ldg(ov_row + q * p.ov.cells + c);
                            }
                        }
                    }
                } else {
                    int c = ci[i], x = kx[i], y = ky[i];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int iy = iy0 + y, ix = ix0 + x;
                        if (y < p.kh && (unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
                            v[u] = __ldg(xrow + ((int64_t)iy * p.iw + ix) * p.ic + c);
                        if (++c == p.ic) { c = 0; if (++x == p.kw) { x = 0; ++y; } }
                    }
                }
            }
            ra[i] = make_float4(v[0], v[1], v[2], v[3]);
            ci[i] += BK;
            carry(i);
        }
#pragma unroll
        for (int i = 0; i < B4N; ++i) {
            const int e = tid + i * NT, k = k0 + e / (BN / 4), n = n0 + 4 * (e % (BN / 4));
            rb[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (e < BK * BN / 4 && k < p.K && n < p.oc) {
                const float *w = p.Wt + (int64_t)k * p.oc + n;
                if ((p.oc & 3) == 0) {
                    rb[i] = __ldg(reinterpret_cast<const float4 *>(w));
                } else {
                    rb[i].x = __ldg(w);
                    if (n + 1 < p.oc) rb[i].y = __ldg(w + 1);
                    if (n + 2 < p.oc) rb[i].z = __ldg(w + 2);
                    if (n + 3 < p.oc) rb[i].w = __ldg(w + 3);
                }
            }
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int i = 0; i < A4N; ++i) {
            const int k = 4 * (tid / BM + i * (NT / BM)), r = tid % BM;
            As[s][k][r] = make_float2(ra[i].x, ra[i].x);
            As[s][k + 1][r] = make_float2(ra[i].y, ra[i].y);
            As[s][k + 2][r] = make_float2(ra[i].z, ra[i].z);
            As[s][k + 3][r] = make_float2(ra[i].w, ra[i].w);
        }
#pragma unroll
        for (int i = 0; i < B4N; ++i) {
            const int e = tid + i * NT;
            if (e < BK * BN / 4) *reinterpret_cast<float4 *>(&Bs[s][e / (BN / 4)][4 * (e % (BN / 4))]) = rb[i];
        }
    };
    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0;
    load(0);
    store(0);
    __syncthreads();
    int s = 0;
    for (int k0 = 0; k0 < p.K; k0 += BK, s ^= 1) {
        const bool more = k0 + BK < p.K;
        if (more) load(k0 + BK);
        simt_tile_fma<BK, BM, BN, TM, TN, RS, CS>(acc, &As[s][0][tm * 4], &Bs[s][0][tn * 4]);
        if (more) store(s ^ 1);
        __syncthreads();
    }
    // epilogue: bias, activation, skip, pooling; rows i .. i + 3 of a group of four are one
    // pooling window
#pragma unroll
    for (int jj = 0; jj < TN; jj += 4) {
        const int n = n0 + (jj / 4) * CS + tn * 4;
        if (n >= p.oc) continue;
        float bias[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) bias[e] = n + e < p.oc ? __ldg(p.b + n + e) : 0.f;
#pragma unroll
        for (int ii = 0; ii < TM; ii += 4) {
            float win[4][4];
            float *yw = nullptr;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int64_t row;
                int py, px, oy, ox;
                place((ii / 4) * RS + tm * 4 + i, row, py, px, oy, ox);
                if (row >= p.R) continue;
                const float2 lo = unpack2(acc[ii + i][jj / 2]), hi = unpack2(acc[ii + i][jj / 2 + 1]);
                float v[4] = {lo.x + bias[0], lo.y + bias[1], hi.x + bias[2], hi.y + bias[3]};
                const float *sr = nullptr;
                if (p.has_add)
                    sr = p.skip + (p.skip_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.skip_stride +
                         ((int64_t)oy * p.sk_stride * p.sk_w + ox * p.sk_stride) * p.sk_c + n;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (n + e >= p.oc) continue;
                    if (p.z) p.z[row * p.z_stride + (int64_t)(n + e) * (p.oh * p.ow) + oy * p.ow + ox] = v[e];   // channel-major
                    v[e] = act_apply(p.act1, v[e]);
                    if (p.has_add) v[e] = act_apply(p.act2, v[e] + (n + e < p.sk_c ? __ldg(sr + e) : 0.f));
                }
                float *yr = p.y + row * p.y_stride + n;
                if (p.pool) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) win[i][e] = v[e];
                    yw = yr + ((int64_t)py * p.pw + px) * p.oc;
                    continue;
                }
                yr += ((int64_t)oy * p.ow + ox) * p.oc;
                if (p.vec) {
                    *reinterpret_cast<float4 *>(yr) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (n + e < p.oc) yr[e] = v[e];
                }
            }
            if (p.pool && yw) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (n + e < p.oc) yw[e] = max4_first(win[0][e], win[1][e], win[2][e], win[3][e]);
            }
        }
    }
}

// Global average pooling: y[r][c] = (sum over positions, ascending, in fp32) / P.
__global__ void k_gap(const float *__restrict__ in, int64_t in_stride, int P, int C, int R, float *__restrict__ y,
                      int64_t y_stride)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)R * C) return;
    const int64_t r = i / C;
    const int c = (int)(i % C);
    y[r * y_stride + c] = gap_sum(in + r * in_stride, P, C, c);
}

// Depthwise convolution stage (MobileNetV2): output channel c at (oy, ox) is the fp32
// FMA chain over its filter taps (ky, kx ascending, from +0) on input channel c, then
// + b; the pre-activation goes to z (channel-major) when requested, act1 to y.  One
// thread per (row, position, channel): consecutive threads read and write
// consecutive channels, and the weights are read as Wt [tap][c].
__global__ void __launch_bounds__(256) k_dwconv(const StageParams p)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per_row = (int64_t)p.oh * p.ow * p.oc;
    if (i >= (int64_t)p.R * per_row) return;
    const int64_t row = i / per_row;
    const int rem = (int)(i - row * per_row);
    const int c = rem % p.oc, pos = rem / p.oc, oy = pos / p.ow, ox = pos - (pos / p.ow) * p.ow;
    const float *xrow = p.x + (p.x_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.x_stride;
    float acc = 0.f;
    for (int ky = 0; ky < p.kh; ++ky) {
        const int iy = oy * p.stride - p.pad + ky;
        for (int kx = 0; kx < p.kw; ++kx) {
            const int ix = ox * p.stride - p.pad + kx;
            if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
                acc = fmaf(__ldg(p.Wt + (int64_t)(ky * p.kw + kx) * p.oc + c),
                           __ldg(xrow + ((int64_t)iy * p.iw + ix) * p.ic + c), acc);
        }
    }
    const float z = acc + __ldg(p.b + c);
    if (p.z) p.z[row * p.z_stride + (int64_t)c * (p.oh * p.ow) + pos] = z;
    p.y[row * p.y_stride + (int64_t)pos * p.oc + c] = act_apply(p.act1, z);
}

// The 3 x 3 depthwise convolution of channels in fours: a thread computes 2 x 4 outputs of four
// channels from one walk over their input field (16-byte loads: 24 of them for 8 outputs at
// stride 1, against 9 per output), the filter in registers.  The same chain per output: taps in
// ascending order, those outside the image left out.  What bounds it is HBM (the layer's rows in
// and out); a block works inside one row, so no thread divides 64-bit indexes.
// Measured on the MobileNetV2-style network (500 inputs x 41 mutants, 33 launches): 9.05 ms with
// a thread per output, 1.80 ms now, about 4.5 TB/s of rows read and written.
template <int STRIDE>
__global__ void __launch_bounds__(256) k_dwconv3(const StageParams p, int c4n, int gx, int units, int blocks_per_row)
{
    constexpr int OY = 2, OX = 4, IX = (OX - 1) * STRIDE + 3, IY = (OY - 1) * STRIDE + 3;
    const int64_t row = blockIdx.x / blocks_per_row;
    const int u = (int)(blockIdx.x - row * blocks_per_row) * 256 + threadIdx.x;
    if (u >= units) return;
    const int c4 = u % c4n, g = u / c4n, ox0 = g % gx * OX, oy0 = g / gx * OY;
    const float *x = p.x + (p.x_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.x_stride + 4 * c4;
    float4 w[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = __ldg(reinterpret_cast<const float4 *>(p.Wt + (int64_t)k * p.oc + 4 * c4));
    const float4 b = __ldg(reinterpret_cast<const float4 *>(p.b) + c4);
    float4 acc[OY][OX];
#pragma unroll
    for (int i = 0; i < OY; ++i)
#pragma unroll
        for (int j = 0; j < OX; ++j) acc[i][j] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int iy0 = oy0 * STRIDE - p.pad, ix0 = ox0 * STRIDE - p.pad;
#pragma unroll
    for (int yy = 0; yy < IY; ++yy) {
        const int iy = iy0 + yy;
        if ((unsigned)iy >= (unsigned)p.ih) continue;
        float4 v[IX];
#pragma unroll
        for (int xx = 0; xx < IX; ++xx)
            v[xx] = (unsigned)(ix0 + xx) < (unsigned)p.iw
                        ? __ldg(reinterpret_cast<const float4 *>(x + ((int64_t)iy * p.iw + ix0 + xx) * p.ic))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < OY; ++i) {
            const int ky = yy - i * STRIDE;
            if (ky < 0 || ky > 2) continue;
#pragma unroll
            for (int j = 0; j < OX; ++j)
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    const int xx = j * STRIDE + kx;
                    if ((unsigned)(ix0 + xx) >= (unsigned)p.iw) continue;
                    acc[i][j].x = fmaf(w[3 * ky + kx].x, v[xx].x, acc[i][j].x);
                    acc[i][j].y = fmaf(w[3 * ky + kx].y, v[xx].y, acc[i][j].y);
                    acc[i][j].z = fmaf(w[3 * ky + kx].z, v[xx].z, acc[i][j].z);
                    acc[i][j].w = fmaf(w[3 * ky + kx].w, v[xx].w, acc[i][j].w);
                }
        }
    }
#pragma unroll
    for (int i = 0; i < OY; ++i)
#pragma unroll
        for (int j = 0; j < OX; ++j) {
            const int oy = oy0 + i, ox = ox0 + j;
            if (oy >= p.oh || ox >= p.ow) continue;
            const int pos = oy * p.ow + ox;
            const float4 z = make_float4(acc[i][j].x + b.x, acc[i][j].y + b.y, acc[i][j].z + b.z, acc[i][j].w + b.w);
            if (p.z) {
                float *zr = p.z + row * p.z_stride + (int64_t)4 * c4 * (p.oh * p.ow) + pos;
                zr[0] = z.x;
                zr[p.oh * p.ow] = z.y;
                zr[2 * p.oh * p.ow] = z.z;
                zr[3 * p.oh * p.ow] = z.w;
            }
            *reinterpret_cast<float4 *>(p.y + row * p.y_stride + (int64_t)pos * p.oc + 4 * c4) =
                make_float4(act_apply(p.act1, z.x), act_apply(p.act1, z.y), act_apply(p.act1, z.z), act_apply(p.act1, z.w));
        }
}

namespace {

bool aligned16(const void *q, int64_t stride) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0 && stride % 4 == 0; }

template <int BM, int BN, int TM, int TN>
void stage_tiles(StageParams p, bool a4, cudaStream_t s)
{
    p.n_tiles = (p.oc + BN - 1) / BN;
    const int64_t tiles = ((int64_t)p.R * p.P + BM - 1) / BM * p.n_tiles;
    if (p.ov.patch) k_stage_simt<BM, BN, TM, TN, true, true><<<(unsigned)tiles, BM / TM * (BN / TN), 0, s>>>(p);
    else if (a4) k_stage_simt<BM, BN, TM, TN, true, false><<<(unsigned)tiles, BM / TM * (BN / TN), 0, s>>>(p);
    else k_stage_simt<BM, BN, TM, TN, false, false><<<(unsigned)tiles, BM / TM * (BN / TN), 0, s>>>(p);
}

}  // namespace

// Whether the stage's kernel applies the patch as it fetches rows of x; else the rows are
// materialised first.  The pieces that a block fetches are fetched again for every tap and column
// tile, and each looks at all mutated channels, so only few channels of rows that are read about
// once are worth it.  Measured, fp32, 32 mutants, the layer with its rows, materialised / inline:
// dense layers on cached rows 1.04 to 1.22 at one channel, 1.00 to 1.17 at two, 0.91 to 1.06 at four,
// 0.7 at sixteen; of 512 outputs 0.98 at one; on rows of their own, where writing the patch over them
// costs one small launch, 0.8 to 1.0 at one; 3 x 3 convolutions 0.8 to 0.98 at one channel, 0.55 to
// 0.75 at eight.  The 1 x 1 kernel of few channels, whose tiles of 128 positions are patched in shared
// memory: on cached rows 1.0 to 1.4 up to an eighth of the channels (64 -> 16: 1.20 at eight, 0.98 at
// 24; 24 -> 96: 1.02 at two, 0.94 at six); on rows of their own 1.02 to 1.13 where there are more
// outputs than inputs, else 0.86 to 1.03; tiles of 64 positions 0.94 at two.
int simt_overlay_inline(const Stage &S, const Overlay &ov, Src x)
{
    if (S.tc || S.variant > 0 || S.ic % 4 != 0 || ov.ch % 4 != 0 || !aligned16(x.p, x.stride)) return 0;
    if (S.c11) return S.oh * S.ow % 128 == 0 && 8 * ov.kmax <= S.ic && (x.per_input || S.oc > S.ic);
    return S.kind == MURE_NODE_DENSE && x.per_input && ov.kmax <= 2 && S.oc <= 128;
}

int launch_stage_simt(const Stage &S, Src x, RowMap rm, float *z_out, int64_t z_stride, Src skip, float *y_out,
                      int64_t y_stride, float *tmp, cudaStream_t s, const Overlay *ov)
{
    if (rm.R <= 0) return 0;
    if (S.tc) return launch_tc(S, x, rm, z_out, z_stride, skip, y_out, y_stride, tmp, s);
    if (S.kind == MURE_NODE_EMBED) return launch_embed(S, x, rm, z_out, z_stride, y_out, y_stride, s);
    if (S.kind == MURE_NODE_LSTM) {
        LstmWs lw;
        lw.proj = tmp;
        return launch_lstm(S, x, rm, z_out, z_stride, y_out, y_stride, nullptr, lw, s);
    }
    if (S.kind == MURE_NODE_DWCONV) {
        StageParams p{};
        p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
        p.t0 = rm.t0; p.T = rm.T; p.R = rm.R; p.lrow = rm.lrow;
        p.ih = S.ih; p.iw = S.iw; p.ic = S.ic; p.kh = S.kh; p.kw = S.kw; p.stride = S.stride; p.pad = S.pad;
        p.oh = S.oh; p.ow = S.ow; p.oc = S.oc; p.K = S.K;
        p.Wt = S.Wt; p.b = S.b; p.act1 = S.act1;
        p.z = z_out; p.z_stride = z_stride;
        p.y = y_out; p.y_stride = y_stride;
        // 3 x 3 filters, channels in fours on 16-byte rows, and at least half a block of 2 x 4
        // output groups per row (a block takes one row's groups; with fewer most of its threads
        // would idle); else a thread per output
        const int gx = (S.ow + 3) / 4, c4n = S.oc / 4;
        const int64_t units = (int64_t)((S.oh + 1) / 2) * gx * c4n, bpr = (units + 255) / 256;
        if (S.kh == 3 && S.kw == 3 && (S.stride == 1 || S.stride == 2) && S.oc % 4 == 0 && units >= 128 &&
            bpr * rm.R < INT32_MAX && aligned16(x.p, x.stride) && aligned16(y_out, y_stride) && aligned16(S.Wt, 0) && aligned16(S.b, 0)) {
            auto go = [&](auto kern) { kern<<<(unsigned)(bpr * rm.R), 256, 0, s>>>(p, c4n, gx, (int)units, (int)bpr); };
            if (S.stride == 1) go(k_dwconv3<1>);
            else go(k_dwconv3<2>);
            return 1;
        }
        const int64_t n = (int64_t)rm.R * S.oh * S.ow * S.oc;
        k_dwconv<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p);
        return 1;
    }
    if (S.variant > 0) return launch_conv_small(S, x, rm, z_out, z_stride, y_out, y_stride, s);
    StageParams p{};
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.R = rm.R; p.lrow = rm.lrow;
    p.ih = S.ih; p.iw = S.iw; p.ic = S.ic; p.kh = S.kh; p.kw = S.kw; p.stride = S.stride; p.pad = S.pad;
    p.oh = S.oh; p.ow = S.ow; p.oc = S.oc; p.K = S.K;
    p.Wt = S.Wt; p.b = S.b;
    p.act1 = S.act1; p.has_add = S.has_add; p.act2 = S.act2; p.pool = S.pool;
    p.skip = skip.p; p.skip_stride = skip.stride; p.skip_per_input = skip.per_input;
    p.sk_w = S.sk_w; p.sk_c = S.sc_c; p.sk_stride = S.sc_stride;
    p.z = z_out; p.z_stride = z_stride;
    // with global average pooling the post-op map goes to the scratch first
    const int mh = S.pool ? S.oh / 2 : S.oh, mw = S.pool ? S.ow / 2 : S.ow;
    const int64_t map_stride = round4((int64_t)mh * mw * S.oc);
    p.y = S.gap ? tmp : y_out;
    p.y_stride = S.gap ? map_stride : y_stride;
    p.pw = S.ow / 2;
    p.P = S.pool ? 4 * (S.oh / 2) * (S.ow / 2) : S.oh * S.ow;
    p.vec = S.oc % 4 == 0 && aligned16(p.y, p.y_stride);
    if (ov) p.ov = *ov;
    const bool a4 = S.ic % 4 == 0 && aligned16(x.p, x.stride);
    int launches = 1;
    if (S.c11 && a4 && p.vec) launch_conv1x1(S, x, rm, z_out, z_stride, skip, p.y, p.y_stride, s, ov);
    else
    // the narrowest tile that holds the outputs: padded columns cost as much as real ones
    if (S.oc <= 16) stage_tiles<128, 16, 4, 4>(p, a4, s);
    else if (S.oc <= 32) stage_tiles<128, 32, 8, 4>(p, a4, s);
    else if (S.oc <= 64) stage_tiles<128, 64, 8, 8>(p, a4, s);
    else stage_tiles<64, 128, 8, 8>(p, a4, s);
    if (S.gap) {
        const int64_t n = (int64_t)rm.R * S.oc;
        k_gap<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(tmp, map_stride, mh * mw, S.oc, rm.R, y_out, y_stride);
        ++launches;
    }
    return launches;
}

// ------------------------------------------------------ output layer + epilogue --

struct FinalParams {
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T; int R;
    const int32_t *lrow;   // compacted batch: logical rows (per-input reads, overlay), else null
    int F, C, act;
    const float *W;  // [C][F]
    const float *Wt; // [F][C] (the same weights, input-major)
    const float *b;
    FinalArgs fa;
    Overlay ov;      // mutated channels of the input rows (ov.patch null: none)
};

// Kill bits of one warp of rows (32 consecutive inputs of one mutant) and the
// near-tie count.  v = the row's logits.
__device__ __forceinline__ void epilogue_row(const FinalArgs &fa, int64_t t0, int T, int64_t row, bool in_range,
                                             const float *v, int C)
{
    const int64_t lr = in_range ? logical_row(fa.lrow, row) : row;
    const int g = (int)(lr / T);
    const int64_t t = t0 + lr % T;
    const bool valid = in_range && t < fa.n_in;
    int arg = 0;
    bool near = false;
    if (valid) {
        arg = argmax_first(v, C);
        near = near_tie(v, C, arg);
    }
    const bool kill = valid && fa.pred0[t] == fa.label[t] && arg != fa.label[t];
    const unsigned kb = __ballot_sync(0xffffffffu, kill);
    const unsigned nb = __ballot_sync(0xffffffffu, near);
    const int lane = threadIdx.x & 31;
    if (fa.compact) {
        // a compacted batch: the warp's rows are any (mutant, input) pairs; the matrix
        // was zeroed, each killed row sets its own bit
        if (kill) atomicOr(fa.kill32 + (int64_t)fa.mutant_id[g] * fa.words32 + (t >> 5), 1u << (t & 31));
        if (lane == 0 && nb && fa.near_ties) atomicAdd(fa.near_ties, (unsigned long long)__popc(nb));
    } else if (lane == 0 && in_range) {
        const int mid = fa.mutant_id[g];
        fa.kill32[(int64_t)mid * fa.words32 + (t >> 5)] = kb;
        if (nb && fa.near_ties) atomicAdd(fa.near_ties, (unsigned long long)__popc(nb));
    }
    if (valid && fa.logits_out) {
        float *o = fa.logits_out + ((int64_t)fa.mutant_id[g] * fa.n_in + t) * C;
        for (int c = 0; c < C; ++c) o[c] = v[c];
    }
}

// CP: the class count rounded up to a multiple of 4 (the accumulators kept per row).
template <int CP>
__global__ void __launch_bounds__(128) k_final_dense(const FinalParams p)
{
    constexpr int RB = 128, FC = 32;
    __shared__ float xs[RB][FC + 1];
    __shared__ __align__(16) float ws[FC][CP];
    const int tid = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * RB;
    const int64_t row = row0 + tid;
    const bool in_range = row < p.R;
    // this row's mutated input channels (overlay), as (slot count, id pointer)
    int ov_k = 0;
    const int32_t *ov_ids = nullptr;
    const int64_t lrow = in_range ? logical_row(p.lrow, row) : row;
    if (p.ov.patch && in_range) {
        const int g = (int)(lrow / p.T);
        ov_k = p.ov.n_neurons[g];
        ov_ids = p.ov.ids + p.ov.neuron_off[g];
    }
    __shared__ const float *xrow_of[RB];
    float acc[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0.f;
    {
        const int64_t r = row0 + tid;
        xrow_of[tid] = r < p.R ? p.x + (p.x_per_input ? (p.t0 + logical_row(p.lrow, r) % p.T) : r) * p.x_stride
                               : nullptr;
    }
    __syncthreads();
    for (int f0 = 0; f0 < p.F; f0 += FC) {
#pragma unroll 8
        for (int i = tid; i < RB * FC; i += RB) {
            const int rl = i / FC, fl = i % FC;
            const float *xr = xrow_of[rl];
            xs[rl][fl] = (xr && f0 + fl < p.F) ? __ldg(xr + f0 + fl) : 0.f;
        }
        for (int i = tid; i < FC * CP; i += RB) {
            const int fl = i / CP, c = i % CP;
            ws[fl][c] = (c < p.C && f0 + fl < p.F) ? __ldg(p.W + (int64_t)c * p.F + f0 + fl) : 0.f;
        }
        __syncthreads();
        const int fe = min(FC, p.F - f0);
        // overlay on this thread's own row (no other thread reads it)
        for (int q = 0; q < ov_k; ++q) {
            const int j = ov_ids[q];
            const int cfirst = f0 - j <= 0 ? 0 : (f0 - j + p.ov.ch - 1) / p.ov.ch;
            for (int c = cfirst; c < p.ov.cells && c * p.ov.ch + j < f0 + fe; ++c)
                xs[tid][c * p.ov.ch + j - f0] = p.ov.patch[lrow * p.ov.row_stride + q * p.ov.cells + c];
        }
        for (int fl = 0; fl < fe; ++fl) {
            const float xv = xs[tid][fl];
#pragma unroll
            for (int c4 = 0; c4 < CP; c4 += 4) {
                const float4 w4 = *reinterpret_cast<const float4 *>(&ws[fl][c4]);
                acc[c4] = fmaf(xv, w4.x, acc[c4]);
                acc[c4 + 1] = fmaf(xv, w4.y, acc[c4 + 1]);
                acc[c4 + 2] = fmaf(xv, w4.z, acc[c4 + 2]);
                acc[c4 + 3] = fmaf(xv, w4.w, acc[c4 + 3]);
            }
        }
        __syncthreads();
    }
    float v[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) {
        const float z = c < p.C ? acc[c] + __ldg(p.b + c) : 0.f;
        if (in_range && c < p.C && p.fa.z_out) p.fa.z_out[row * p.fa.z_stride + c] = z;
        v[c] = act_apply(p.act, z);
    }
    if (p.fa.mode == 1) {  // cache build: logits rows and original predictions
        if (in_range) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                if (c < p.C) p.fa.x_out[row * p.fa.x_stride + c] = v[c];
            p.fa.pred_out[row] = argmax_reg<CP>(v, p.C);
        }
        return;
    }
    if (p.fa.mode == 2) {  // per-row logits for a following delta + epilogue
        if (in_range) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                if (c < p.C) p.fa.logits_rows[row * p.fa.x_stride + c] = v[c];
        }
        return;
    }
    epilogue_reg<CP>(p.fa, p.t0, p.T, row, in_range, v, p.C);
}

// The same output layer with each warp on its own 32 rows (lane = row) and no block-wide
// barrier after the weights are staged: the warp copies its rows' next 32 inputs (16-byte
// loads, eight per lane) while it runs the FMAs of the current 32, through a per-warp
// shared-memory tile.  Each row's sums are the same fp32 chain as k_final_dense's (f
// ascending from +0, fmaf(x, w, acc), then + b), so both kernels give the same bits.
// (One launch of k_final_dense on 6,144 rows of 512 inputs waited 256 us on its loads.)
// Needs F a multiple of 4 and 16-byte aligned rows; the weights [F][CP] in dynamic shared
// memory.
template <int CP>
__global__ void __launch_bounds__(128) k_final_dense_w(const FinalParams p)
{
    extern __shared__ __align__(16) float wsm[];   // [F][CP]
    __shared__ float xs[4][32][33];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < p.F * CP; i += blockDim.x) {
        const int f = i / CP, c = i - f * CP;
        wsm[i] = c < p.C ? __ldg(p.W + (int64_t)c * p.F + f) : 0.f;
    }
    __syncthreads();
    const int64_t row0 = (int64_t)blockIdx.x * 128 + warp * 32;
    const int64_t row = row0 + lane;
    const bool in_range = row < p.R;
    int ov_k = 0;
    const int32_t *ov_ids = nullptr;
    const int64_t lrow = in_range ? logical_row(p.lrow, row) : row;
    if (p.ov.patch && in_range) {
        const int g = (int)(lrow / p.T);
        ov_k = p.ov.n_neurons[g];
        ov_ids = p.ov.ids + p.ov.neuron_off[g];
    }
    // this lane copies 16 bytes (inputs 4 (lane mod 8) .. +3) of rows 4i + lane / 8
    const int fq = 4 * (lane & 7);
    const float *src[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int64_t r = row0 + 4 * i + (lane >> 3);
        src[i] = r < p.R ? p.x + (p.x_per_input ? (p.t0 + logical_row(p.lrow, r) % p.T) : r) * p.x_stride : nullptr;
    }
    auto load = [&](int f0, float4 (&v)[8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = (src[i] && f0 + fq < p.F) ? __ldg(reinterpret_cast<const float4 *>(src[i] + f0 + fq))
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float acc[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0.f;
    float4 cur[8];
    load(0, cur);
    for (int f0 = 0; f0 < p.F; f0 += 32) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float *d = &xs[warp][4 * i + (lane >> 3)][fq];
            d[0] = cur[i].x; d[1] = cur[i].y; d[2] = cur[i].z; d[3] = cur[i].w;
        }
        if (f0 + 32 < p.F) load(f0 + 32, cur);
        __syncwarp();
        const int fe = min(32, p.F - f0);
        // overlay on this lane's own row (no other lane reads it)
        for (int q = 0; q < ov_k; ++q) {
            const int j = ov_ids[q];
            const int cfirst = f0 - j <= 0 ? 0 : (f0 - j + p.ov.ch - 1) / p.ov.ch;
            for (int c = cfirst; c < p.ov.cells && c * p.ov.ch + j < f0 + fe; ++c)
                xs[warp][lane][c * p.ov.ch + j - f0] = p.ov.patch[lrow * p.ov.row_stride + q * p.ov.cells + c];
        }
        for (int fl = 0; fl < fe; ++fl) {
            const float xv = xs[warp][lane][fl];
            const float *wr = wsm + (f0 + fl) * CP;
#pragma unroll
            for (int c4 = 0; c4 < CP; c4 += 4) {
                const float4 w4 = *reinterpret_cast<const float4 *>(wr + c4);
                acc[c4] = fmaf(xv, w4.x, acc[c4]);
                acc[c4 + 1] = fmaf(xv, w4.y, acc[c4 + 1]);
                acc[c4 + 2] = fmaf(xv, w4.z, acc[c4 + 2]);
                acc[c4 + 3] = fmaf(xv, w4.w, acc[c4 + 3]);
            }
        }
    }
    float v[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) {
        const float z = c < p.C ? acc[c] + __ldg(p.b + c) : 0.f;
        if (in_range && c < p.C && p.fa.z_out) p.fa.z_out[row * p.fa.z_stride + c] = z;
        v[c] = act_apply(p.act, z);
    }
    if (p.fa.mode == 1) {  // cache build: logits rows and original predictions
        if (in_range) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                if (c < p.C) p.fa.x_out[row * p.fa.x_stride + c] = v[c];
            p.fa.pred_out[row] = argmax_reg<CP>(v, p.C);
        }
        return;
    }
    if (p.fa.mode == 2) {  // per-row logits for a following delta + epilogue
        if (in_range) {
#pragma unroll
            for (int c = 0; c < CP; ++c)
                if (c < p.C) p.fa.logits_rows[row * p.fa.x_stride + c] = v[c];
        }
        return;
    }
    epilogue_reg<CP>(p.fa, p.t0, p.T, row, in_range, v, p.C);
}

// The output layer of 9 to 12 classes with a block's 32 rows shared by its four warps:
// warp w keeps classes w, w+4 and w+8 of every row (lane = row), so a warp's serial
// instruction stream is a quarter of k_final_dense_w's (which keeps all classes of its
// rows in one warp: ncu showed each of its blocks issue-bound at one warp per scheduler,
// about 32 us per block whatever the grid, a third of it spent on a strided weight
// fill).  A class's sum is the same fp32 chain as k_final_dense's (f ascending from +0,
// fmaf(x, w, acc), then + b), so the bits equal those of the other output-layer kernels.
// The weights come from the input-major copy Wt [F][C] with 16-byte loads all in flight;
// each warp copies the rows' next 32 inputs (16-byte loads) into its own tile of 36-float
// lines (16-byte stores and loads without bank conflicts) while it runs the FMAs of the
// current 32; the warps' sums meet in shared memory, the epilogues go round the warps.  A block
// stays and takes many tiles of 32 rows, its weights placed once (a block per tile: 100 us for
// 279,000 rows of 84 inputs, now 76).  Needs F a multiple of 4 and 16-byte aligned rows;
// dynamic shared memory [F][4][4] (class c at
// [f][c mod 4][c / 4]).
constexpr int kSplitLine = 36;

__global__ void __launch_bounds__(128, 4) k_final_dense_split(const FinalParams p, int tiles)
{
    extern __shared__ __align__(16) float wsm[];   // [F][4][4]
    __shared__ __align__(16) float xs[4][32][kSplitLine];
    __shared__ float sums[2][32][13];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < p.F * 16; i += 128) wsm[i] = 0.f;
    __syncthreads();   // padding zeroed before the weights are placed
    {
        const int n4 = p.F * p.C / 4;
        const float4 *w4p = reinterpret_cast<const float4 *>(p.Wt);
        for (int i0 = threadIdx.x; i0 < n4; i0 += 8 * 128) {
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * 128;
                v[u] = i < n4 ? __ldg(w4p + i) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int i = i0 + u * 128;
                if (i >= n4) continue;
                int f = 4 * i / p.C, c = 4 * i - f * p.C;
                const float e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    wsm[f * 16 + (c & 3) * 4 + (c >> 2)] = e[k];
                    if (++c == p.C) { c = 0; ++f; }
                }
            }
        }
    }
    __syncthreads();   // the weights
    const float *wq = wsm + 4 * warp;
    const float *xr = &xs[warp][lane][0];
    const int fq = 4 * (lane & 7);
    int it = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++it) {
        const int buf = it & 1;
        const int64_t row0 = (int64_t)tile * 32;
        const int64_t row = row0 + lane;
        const bool in_range = row < p.R;
        int ov_k = 0;
        const int32_t *ov_ids = nullptr;
        const int64_t lrow = in_range ? logical_row(p.lrow, row) : row;
        if (p.ov.patch && in_range) {
            const int g = (int)(lrow / p.T);
            ov_k = p.ov.n_neurons[g];
            ov_ids = p.ov.ids + p.ov.neuron_off[g];
        }
        // this lane copies 16 bytes (inputs 4 (lane mod 8) .. +3) of rows 4i + lane / 8
        const float *src[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int64_t r = row0 + 4 * i + (lane >> 3);
            src[i] = r < p.R ? p.x + (p.x_per_input ? (p.t0 + logical_row(p.lrow, r) % p.T) : r) * p.x_stride : nullptr;
        }
        auto load = [&](int f0, float4 (&v)[8]) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = (src[i] && f0 + fq < p.F) ? __ldg(reinterpret_cast<const float4 *>(src[i] + f0 + fq))
                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 cur[8];
        load(0, cur);
        float a0 = 0.f, a1 = 0.f, a2 = 0.f;
        for (int f0 = 0; f0 < p.F; f0 += 32) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; ++i) *reinterpret_cast<float4 *>(&xs[warp][4 * i + (lane >> 3)][fq]) = cur[i];
            if (f0 + 32 < p.F) load(f0 + 32, cur);
            __syncwarp();
            const int fe = min(32, p.F - f0);
            // overlay on this lane's own row (no other lane reads it)
            for (int q = 0; q < ov_k; ++q) {
                const int j = ov_ids[q];
                const int cfirst = f0 - j <= 0 ? 0 : (f0 - j + p.ov.ch - 1) / p.ov.ch;
                for (int c = cfirst; c < p.ov.cells && c * p.ov.ch + j < f0 + fe; ++c)
                    xs[warp][lane][c * p.ov.ch + j - f0] = p.ov.patch[lrow * p.ov.row_stride + q * p.ov.cells + c];
            }
            if (fe == 32) {
#pragma unroll
                for (int f4 = 0; f4 < 32; f4 += 4) {
                    const float4 x4 = *reinterpret_cast<const float4 *>(xr + f4);
                    const float xq[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float4 w4 = *reinterpret_cast<const float4 *>(wq + (f0 + f4 + e) * 16);
                        a0 = fmaf(xq[e], w4.x, a0);
                        a1 = fmaf(xq[e], w4.y, a1);
                        a2 = fmaf(xq[e], w4.z, a2);
                    }
                }
            } else {
                for (int fl = 0; fl < fe; ++fl) {
                    const float xv = xr[fl];
                    const float4 w4 = *reinterpret_cast<const float4 *>(wq + (f0 + fl) * 16);
                    a0 = fmaf(xv, w4.x, a0);
                    a1 = fmaf(xv, w4.y, a1);
                    a2 = fmaf(xv, w4.z, a2);
                }
            }
        }
        sums[buf][lane][warp] = a0;
        sums[buf][lane][warp + 4] = a1;
        sums[buf][lane][warp + 8] = a2;
        // one barrier per tile: the other warps go on to the next tile, whose sums go to the other
        // buffer; they write this one again only after every warp has come to the next barrier.
        // The warps take the epilogue in turn
        __syncthreads();
        if (warp != (it & 3)) continue;
        float v[12];
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const float z = c < p.C ? sums[buf][lane][c] + __ldg(p.b + c) : 0.f;
            if (in_range && c < p.C && p.fa.z_out) p.fa.z_out[row * p.fa.z_stride + c] = z;
            v[c] = act_apply(p.act, z);
        }
        if (p.fa.mode == 1) {  // cache build: logits rows and original predictions
            if (in_range) {
#pragma unroll
                for (int c = 0; c < 12; ++c)
                    if (c < p.C) p.fa.x_out[row * p.fa.x_stride + c] = v[c];
                p.fa.pred_out[row] = argmax_reg<12>(v, p.C);
            }
        } else if (p.fa.mode == 2) {  // per-row logits for a following delta + epilogue
            if (in_range) {
#pragma unroll
                for (int c = 0; c < 12; ++c)
                    if (c < p.C) p.fa.logits_rows[row * p.fa.x_stride + c] = v[c];
            }
        } else {
            epilogue_reg<12>(p.fa, p.t0, p.T, row, in_range, v, p.C);
        }
    }
}

__global__ void __launch_bounds__(128) k_epilogue(const float *__restrict__ lg, int64_t stride, int per_input, int C,
                                                  int64_t t0, int T, int R, const FinalArgs fa, const Overlay ov)
{
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool in_range = row < R;
    float v[kMaxClasses];
    const float *src = lg + (per_input ? t0 + row % T : row) * stride;
#pragma unroll
    for (int c = 0; c < kMaxClasses; ++c) v[c] = (in_range && c < C) ? src[c] : 0.f;
    if (ov.patch && in_range) {
        const int g = (int)(row / T);
        const int32_t *ids = ov.ids + ov.neuron_off[g];
        for (int q = 0; q < ov.n_neurons[g]; ++q) {
            const float val = ov.patch[row * ov.row_stride + q * ov.cells];
#pragma unroll
            for (int c = 0; c < kMaxClasses; ++c)
                if (c == ids[q]) v[c] = val;
        }
    }
    epilogue_row(fa, t0, T, row, in_range, v, C);
}

// The output layer for rows (per input or per row) with a dense overlay: each
// thread copies its own input row (16-byte loads, all in flight at once) into its own
// shared-memory row, writes the mutated channels there and runs the same fp32 chain as
// k_final_dense (f ascending, fmaf(x, w, acc)), so both kernels give the same bits.
// No block-wide barrier sits between the loads and the FMAs.
constexpr int kRowsF = 100;   // floats per staged row (F <= 96), a multiple of 4

template <int CP, int UF>
__global__ void __launch_bounds__(128) k_final_dense_rows(const FinalParams p)
{
    extern __shared__ __align__(16) float fsm[];
    float *ws = fsm;                              // [F][CP]
    float *xr = fsm + p.F * CP + threadIdx.x * kRowsF;
    const int tid = threadIdx.x;
    const int64_t row = (int64_t)blockIdx.x * 128 + tid;
    const bool in_range = row < p.R;
    for (int i = tid; i < p.F * CP; i += 128) {
        const int fl = i / CP, c = i % CP;
        ws[i] = c < p.C ? __ldg(p.W + (int64_t)c * p.F + fl) : 0.f;
    }
    if (in_range) {
        const int64_t lrow = logical_row(p.lrow, row);
        const float4 *src = reinterpret_cast<const float4 *>(p.x + (p.x_per_input ? p.t0 + lrow % p.T : row) * p.x_stride);
        float4 v[kRowsF / 4];
#pragma unroll
        for (int i = 0; i < kRowsF / 4; ++i)
            if (4 * i < p.F) v[i] = __ldg(src + i);
#pragma unroll
        for (int i = 0; i < kRowsF / 4; ++i)
            if (4 * i < p.F) *reinterpret_cast<float4 *>(xr + 4 * i) = v[i];
        if (p.ov.patch) {
            const int g = (int)(lrow / p.T);
            const int k = p.ov.n_neurons[g];
            const int32_t *ids = p.ov.ids + p.ov.neuron_off[g];
            for (int q = 0; q < k; ++q) xr[ids[q]] = p.ov.patch[lrow * p.ov.row_stride + q];
        }
    }
    __syncthreads();   // the weights
    float acc[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) acc[c] = 0.f;
    if (in_range) {
        // four inputs per 16-byte load (rows 400 bytes apart: no bank conflicts)
#pragma unroll UF
        for (int f4 = 0; f4 < p.F; f4 += 4) {
            const float4 x4 = *reinterpret_cast<const float4 *>(xr + f4);
            const float xq[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float xv = xq[e];
#pragma unroll
                for (int c4 = 0; c4 < CP; c4 += 4) {
                    const float4 w4 = *reinterpret_cast<const float4 *>(ws + (f4 + e) * CP + c4);
                    acc[c4] = fmaf(xv, w4.x, acc[c4]);
                    acc[c4 + 1] = fmaf(xv, w4.y, acc[c4 + 1]);
                    acc[c4 + 2] = fmaf(xv, w4.z, acc[c4 + 2]);
                    acc[c4 + 3] = fmaf(xv, w4.w, acc[c4 + 3]);
                }
            }
        }
    }
    float v[CP];
#pragma unroll
    for (int c = 0; c < CP; ++c) {
        const float z = c < p.C ? acc[c] + __ldg(p.b + c) : 0.f;
        v[c] = act_apply(p.act, z);
    }
    epilogue_reg<CP>(p.fa, p.t0, p.T, row, in_range, v, p.C);
}

int launch_gap(const float *in, int64_t in_stride, int P, int C, int R, float *y, int64_t y_stride, cudaStream_t s)
{
    const int64_t n = (int64_t)R * C;
    if (n <= 0) return 0;
    k_gap<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(in, in_stride, P, C, R, y, y_stride);
    return 1;
}

int launch_final_dense(const Stage &S, Src x, RowMap rm, const FinalArgs &fa, cudaStream_t s, const Overlay *ov)
{
    if (rm.R <= 0) return 0;
    FinalParams p{};
    if (ov) p.ov = *ov;
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.R = rm.R; p.lrow = rm.lrow;
    p.F = S.K; p.C = S.oc; p.act = S.act1;
    p.W = S.W; p.Wt = S.Wt; p.b = S.b;
    p.fa = fa;
    const unsigned blocks = (unsigned)((rm.R + 127) / 128);
    const int cp = (p.C + 3) & ~3;
    // per-input rows with a small dense overlay, mutants' kill epilogue only: each
    // thread stages its own row (measured on the LeNet-5 workload, FC 84-10 of the FC
    // 120-84 mutants: 0.68 -> 0.56 ms per step; on row-per-row inputs it was slower)
    if (x.per_input && fa.mode == 0 && !fa.z_out && p.F <= kRowsF - 4 && p.F % 4 == 0 && cp == 12 &&
        (x.stride & 3) == 0 && (reinterpret_cast<uintptr_t>(x.p) & 15) == 0 && (!ov || (ov->cells == 1 && ov->kmax <= 4))) {
        const size_t smem = ((size_t)p.F * 12 + 128 * kRowsF) * sizeof(float);
        allow_dynamic_smem(k_final_dense_rows<12, 3>, ((kRowsF - 4) * 12 + 128 * kRowsF) * (int)sizeof(float));
        k_final_dense_rows<12, 3><<<blocks, 128, smem, s>>>(p);
        return 1;
    }
    // aligned rows of whole 16-byte pieces, weights that fit in shared memory: per-warp rows
    // with the next inputs in flight
    const size_t wbytes = (size_t)p.F * cp * sizeof(float);
    constexpr int kWeightBytes = 96 * 1024;
    if (p.F % 4 == 0 && (x.stride & 3) == 0 && (reinterpret_cast<uintptr_t>(x.p) & 15) == 0 && cp <= 12 &&
        wbytes <= kWeightBytes) {
        auto go = [&](auto kern) {
            allow_dynamic_smem(kern, kWeightBytes);
            kern<<<blocks, 128, wbytes, s>>>(p);
        };
        if (cp <= 4) go(k_final_dense_w<4>);
        else if (cp <= 8) go(k_final_dense_w<8>);
        else {
            // 9 to 12 classes: a block's 32 rows shared by four warps
            const size_t sbytes = (size_t)p.F * 16 * sizeof(float);
            allow_dynamic_smem(k_final_dense_split, kWeightBytes / 12 * 16);
            // blocks that stay (four per SM) and take several tiles: the weights are placed once
            // per block, not once per 32 rows
            const int tiles = (rm.R + 31) / 32;
            k_final_dense_split<<<(unsigned)std::min(tiles, 4 * sm_count()), 128, sbytes, s>>>(p, tiles);
        }
        return 1;
    }
    if (cp <= 4) k_final_dense<4><<<blocks, 128, 0, s>>>(p);
    else if (cp <= 8) k_final_dense<8><<<blocks, 128, 0, s>>>(p);
    else if (cp <= 12) k_final_dense<12><<<blocks, 128, 0, s>>>(p);
    else if (cp <= 16) k_final_dense<16><<<blocks, 128, 0, s>>>(p);
    else if (cp <= 32) k_final_dense<32><<<blocks, 128, 0, s>>>(p);
    else k_final_dense<96><<<blocks, 128, 0, s>>>(p);
    return 1;
}

int launch_epilogue(Src logits, int C, RowMap rm, const FinalArgs &fa, cudaStream_t s, const Overlay *ov)
{
    if (rm.R <= 0) return 0;
    Overlay o;
    if (ov) o = *ov;
    k_epilogue<<<(unsigned)((rm.R + 127) / 128), 128, 0, s>>>(logits.p, logits.stride, logits.per_input, C, rm.t0,
                                                              rm.T, rm.R, fa, o);
    return 1;
}

}  // namespace mure
