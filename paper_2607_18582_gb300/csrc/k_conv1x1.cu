// 1 x 1 convolutions of few channels (the expansions and projections of MobileNetV2's blocks) in
// fp32 on the CUDA cores, in the tensor-core precision modes too where that is faster.  Such a layer moves (ic + oc) 4 bytes per position for ic x oc FMAs: at 16
// to 96 channels it is bound by HBM, not by either arithmetic unit, and the tensor-core kernel's
// per-tile hand-overs (about 1,000 cycles per K-step) cost more than the products themselves.
//
// Persistent blocks walk tiles of TP positions of one row, which are one contiguous piece of
// memory: 16-byte asynchronous copies bring the next tile while the current one is computed, the
// weights stay in shared memory.  A thread takes PP positions x four outputs; oc / 4 neighbouring
// lanes share a position, so its inputs are read by broadcast and a warp's outputs leave as one
// contiguous piece; the staged positions are four floats apart more than their channels, so that
// the lanes' groups read different banks.  Per four input channels: PP + 4 16-byte loads for
// 16 PP FMAs.
//
// Arithmetic: the chain of the other fp32 kernels (acc = fma(x_k, w_k, acc), k ascending from +0,
// then + bias, the same post-ops), so that they agree bit for bit.
#include <algorithm>

#include "common.cuh"
#include "device_util.cuh"

namespace mure {

namespace {

struct Conv11Params {
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T; int R;
    const int32_t *lrow;
    int ic, oc, P, tp, tiles_per_row;
    int64_t tiles;
    const float *Wt;   // [ic][oc]
    const float *b;
    int act1, has_add, act2;
    const float *skip; int64_t skip_stride; int skip_per_input; int sk_c;
    float *z; int64_t z_stride;
    float *y; int64_t y_stride;
    Overlay ov;
};

constexpr int kThreads11 = 128;
// the largest layer's weights and staged tiles: 4,096 products (conv1x1_geometry), 128 channels
constexpr int kSmemMax11 = (4096 + 2 * 128 * (128 + 4)) * (int)sizeof(float);

__device__ __forceinline__ void copy16(float *dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

template <int PP>
__global__ void __launch_bounds__(kThreads11, 4) k_conv1x1(const Conv11Params p)
{
    extern __shared__ __align__(16) float sm[];
    float *ws = sm;                     // [ic][oc]
    float *xs = sm + p.ic * p.oc;       // [2][tp][ic + 4]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ol = p.oc / 4, ns = 32 / ol;            // lanes per position, positions groups per warp
    const int sub = lane / ol, n = 4 * (lane - sub * ol);
    const bool live = sub < ns;
    const int pitch = p.ic + 4, tile_floats = p.tp * pitch;
    // the pieces this thread copies: number tid, tid + 128, ..., as (position, four channels)
    const int icq = p.ic / 4, step_pos = kThreads11 / icq, step_c = kThreads11 - step_pos * icq;
    const int pos0 = tid / icq, c0 = tid - pos0 * icq;
    auto row_of = [&](int64_t tile, int &q0) {
        const int64_t row = tile / p.tiles_per_row;
        q0 = (int)(tile - row * p.tiles_per_row) * p.tp;
        return row;
    };
    auto fetch = [&](int64_t tile, int buf) {
        if (tile < p.tiles) {
            int q0;
            const int64_t row = row_of(tile, q0);
            const float *src = p.x + (p.x_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.x_stride +
                               (int64_t)q0 * p.ic;
            float *dst = xs + buf * tile_floats;
            int pos = pos0, c = c0;
            for (int i = 4 * tid; i < p.tp * p.ic; i += 4 * kThreads11) {
                copy16(dst + pos * pitch + 4 * c, src + i);
                pos += step_pos;
                c += step_c;
                if (c >= icq) { c -= icq; ++pos; }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(blockIdx.x, 0);
    for (int i = tid; i < p.ic * p.oc / 4; i += kThreads11)
        reinterpret_cast<float4 *>(ws)[i] = __ldg(reinterpret_cast<const float4 *>(p.Wt) + i);
    const float4 bias = live ? __ldg(reinterpret_cast<const float4 *>(p.b + n)) : make_float4(0.f, 0.f, 0.f, 0.f);
    int buf = 0;
    for (int64_t tile = blockIdx.x; tile < p.tiles; tile += gridDim.x, buf ^= 1) {
        fetch(tile + gridDim.x, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        int q0;
        const int64_t row = row_of(tile, q0);
        const int64_t lr = logical_row(p.lrow, row);
        float *xt = xs + buf * tile_floats;
        if (p.ov.patch) {
            // the mutant's channels of these positions
            const int g = (int)(lr / p.T), k = p.ov.n_neurons[g];
            const int32_t *ids = p.ov.ids + p.ov.neuron_off[g];
            for (int q = 0; q < k; ++q) {
                const int j = ids[q];
                for (int c = tid; c < p.tp; c += kThreads11)
                    xt[c * pitch + j] = __ldg(p.ov.patch + lr * p.ov.row_stride + q * p.ov.cells + q0 + c);
            }
            __syncthreads();
        }
        const float *sr = p.has_add ? p.skip + (p.skip_per_input ? p.t0 + lr % p.T : row) * p.skip_stride + (int64_t)q0 * p.sk_c
                                    : nullptr;
        float *yr = p.y + row * p.y_stride + (int64_t)q0 * p.oc;
        // positions p0, p0 + ns, ...: the warp's groups side by side
        for (int p0 = warp * ns * PP + sub; live && p0 < p.tp; p0 += 4 * ns * PP) {
            float acc[PP][4];
#pragma unroll
            for (int i = 0; i < PP; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
            const float *xp[PP], *wp = ws + n;
#pragma unroll
            for (int i = 0; i < PP; ++i) xp[i] = xt + min(p0 + i * ns, p.tp - 1) * pitch;
            for (int k = 0; k < p.ic; k += 4, wp += 4 * p.oc) {
                float4 w[4], xv[PP];
#pragma unroll
                for (int u = 0; u < 4; ++u) w[u] = *reinterpret_cast<const float4 *>(wp + u * p.oc);
#pragma unroll
                for (int i = 0; i < PP; ++i) xv[i] = *reinterpret_cast<const float4 *>(xp[i] + k);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float we[4] = {w[u].x, w[u].y, w[u].z, w[u].w};
#pragma unroll
                    for (int i = 0; i < PP; ++i) {
                        const float a = u == 0 ? xv[i].x : u == 1 ? xv[i].y : u == 2 ? xv[i].z : xv[i].w;
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[i][e] = fmaf(a, we[e], acc[i][e]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < PP; ++i) {
                const int pos = p0 + i * ns;
                if (pos >= p.tp) break;
                float v[4] = {acc[i][0] + bias.x, acc[i][1] + bias.y, acc[i][2] + bias.z, acc[i][3] + bias.w};
                if (p.z) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) p.z[row * p.z_stride + (int64_t)(n + e) * p.P + q0 + pos] = v[e];   // channel-major
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = act_apply(p.act1, v[e]);
                if (p.has_add) {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        v[e] = act_apply(p.act2, v[e] + (n + e < p.sk_c ? __ldg(sr + (int64_t)pos * p.sk_c + n + e) : 0.f));
                }
                *reinterpret_cast<float4 *>(yr + (int64_t)pos * p.oc + n) = make_float4(v[0], v[1], v[2], v[3]);
            }
        }
        __syncthreads();   // the buffer is free for the tile after next
    }
}

}  // namespace

// Which layers the kernel takes: 1 x 1, stride 1, no pooling, channels in fours, maps of whole
// tiles, an add only of a map of the same geometry, and at most 4,096 products per position.
// Measured on 4,096 rows of 8 x 8, 16 x 16 and 32 x 32 maps against the implicit-GEMM kernel of the
// fp32 mode, 53 shapes of 1,024 to 4,096 products: 0.29 to 0.99 of its time.
int conv1x1_geometry(const Stage &S)
{
    return S.kind == MURE_NODE_CONV2D && S.kh == 1 && S.kw == 1 && S.stride == 1 && S.pad == 0 && !S.pool && S.ic % 4 == 0 &&
           S.oc % 4 == 0 && S.ic <= 128 && S.oc <= 128 && S.ic * S.oc <= 4096 && S.oh * S.ow % 64 == 0 &&
           (!S.has_add || (S.sc_stride == 1 && S.sk_w == S.ow));
}

// Whether it takes them from the tensor-core kernel too.  More input channels mean fewer blocks on
// an SM (the staged tiles) and no more output channels at once, so the line falls with both.  The
// same measurement as a share of the tensor-core kernel's time, 3xTF32 (one TF32 product, whose time
// is only some 5 % shorter: the hand-overs bound it, not the MMAs): 16 -> 64 0.41 to 0.46 (0.41 to
// 0.49), 36 -> 112 0.75 (0.80), 36 -> 80 0.91 (0.98), 48 -> 64 0.78 to 0.92 (0.83 to 0.98), 48 -> 48 0.78 to
// 1.01 (0.89 to 1.09), 64 -> 32 0.73 to 0.91 (0.78 to 0.95), 80 -> 32 0.86 to 0.90 (1.00 to 1.05), 96 -> 16
// 0.74 to 0.99 (0.76 to 1.08), 96 -> 24 1.08 to 1.21 (1.12 to 1.27; kept, its fp32 sums are the more
// exact ones); past the line 40 -> 80 0.95 to 1.27 (1.04 to 1.38), 64 -> 40 1.13 (1.19), 96 -> 32 1.11 to
// 1.25, 128 -> 32 1.28 to 1.70.  64 -> 64 is 0.88 (0.91) on 8 x 8 maps, whose tiles of 64 positions leave
// room for more blocks, and 1.13 to 1.16 (1.17 to 1.21) on larger ones.  The whole MobileNetV2-style
// job (500 x 41): 13.4 -> 10.3 ms, and the logits' error against 64 bits falls from 8.4e-7 to 2.3e-7
// (one TF32 product: 1.8e-4 to 4.2e-5).
int conv1x1_over_tc(const Stage &S)
{
    if (S.ic <= 36 || (S.ic <= 48 && S.oc <= 64)) return 1;
    if (S.oh * S.ow % 128 != 0 && S.ic <= 64 && S.oc <= 64) return 1;
    return S.ic <= 96 && S.oc <= 32 && S.ic * S.oc <= 2560;
}

int launch_conv1x1(const Stage &S, Src x, RowMap rm, float *z_out, int64_t z_stride, Src skip, float *y_out, int64_t y_stride,
                   cudaStream_t s, const Overlay *ov)
{
    Conv11Params p{};
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.R = rm.R; p.lrow = rm.lrow;
    p.ic = S.ic; p.oc = S.oc; p.P = S.oh * S.ow;
    p.tp = p.P % 128 == 0 ? 128 : 64;
    p.tiles_per_row = p.P / p.tp;
    p.tiles = (int64_t)rm.R * p.tiles_per_row;
    p.Wt = S.Wt; p.b = S.b;
    p.act1 = S.act1; p.has_add = S.has_add; p.act2 = S.act2;
    p.skip = skip.p; p.skip_stride = skip.stride; p.skip_per_input = skip.per_input; p.sk_c = S.sc_c;
    p.z = z_out; p.z_stride = z_stride;
    p.y = y_out; p.y_stride = y_stride;
    if (ov) p.ov = *ov;
    const int smem = (S.ic * S.oc + 2 * p.tp * (S.ic + 4)) * (int)sizeof(float);
    const unsigned blocks = (unsigned)std::min<int64_t>(p.tiles, 4 * sm_count());
    auto go = [&](auto kern) {
        allow_dynamic_smem(kern, kSmemMax11);
        kern<<<blocks, kThreads11, smem, s>>>(p);
    };
    // the positions per thread with the fewer rounds over a tile (of 16 outputs eight per thread
    // would leave half the lanes without work)
    const int ns = 32 / (S.oc / 4);
    auto rounds = [&](int pp) { return (p.tp + 4 * ns * pp - 1) / (4 * ns * pp) * pp; };
    if (rounds(4) < rounds(8)) go(k_conv1x1<4>);
    else go(k_conv1x1<8>);
    return 1;
}

}  // namespace mure
