// Mutant-side kernels: descriptor expansion (GF noise, WS shuffles), the delta
// kernel that rewrites only the mutated neurons' channels of a layer on top of its
// original output, and the score reduction.
#include <algorithm>

#include "common.cuh"
#include "device_util.cuh"

namespace mure {

// ------------------------------------------------------------------ expansion --

// GF: standard normals by Box-Muller in fp64 on SplitMix64 draws; normals 2p and 2p + 1 of a
// stream share draws 2p and 2p + 1, so a thread makes both.  fp64 is what bounds it (two
// operations per cycle and SM): a slot's fan-in is spread over blocks of 512 values (one block
// per slot took 464 us for one embedding channel of 20,000 entries, now 14).
constexpr int kExpandValues = 512;

__global__ void __launch_bounds__(kExpandValues / 2) k_expand_gf(const ExpandArgs a)
{
    const SlotJob jb = a.jobs[blockIdx.x];
    if (jb.op != MURE_OP_GF) return;
    const uint64_t stream = splitmix64(jb.seed, (uint64_t)jb.q);
    const double sigma = (double)jb.param * a.sigma[jb.layer];
    for (int64_t f = (int64_t)blockIdx.y * kExpandValues + 2 * threadIdx.x; f < jb.F; f += (int64_t)gridDim.y * kExpandValues) {
        const double u1 = (double)((splitmix64(stream, (uint64_t)f) >> 11) + 1) * (1.0 / 9007199254740992.0);
        const double u2 = (double)((splitmix64(stream, (uint64_t)f + 1) >> 11) + 1) * (1.0 / 9007199254740992.0);
        const double r = sqrt(-2.0 * log(u1));
        const double th = 6.283185307179586476925286766559 * u2;
        float *out = a.patch + jb.out_off + f;
        out[0] = (float)(sigma * (r * cos(th)));
        if (f + 1 < jb.F) out[1] = (float)(sigma * (r * sin(th)));
    }
}

// WS: Fisher-Yates from the last index down; step i swaps places i and j_i, draw F-1-i giving
// j_i = floor(u (i+1)).
__device__ __forceinline__ int shuffle_partner(uint64_t stream, int F, int i)
{
    const double u = (double)(splitmix64(stream, (uint64_t)(F - 1 - i)) >> 11) * (1.0 / 9007199254740992.0);
    const int j = (int)(u * (double)(i + 1));
    return j > i ? i : j;
}

// The same permutation without the serial chain of swaps.  Before step i, place p holds what
// the last earlier step that swapped into p (the smallest e > i with j_e = p) found at its own
// place e, or p itself if none did.  So with A(i) = the value at place i before step i:
// A(i) = A(e), e the smallest e > i with j_e = i, or i; and the result at i is A(e), e the
// smallest e > i with j_e = j_i, or j_i.  The steps into each place form short lists (their
// expected length grows with log F), and A follows a short chain.  Lists and chains in
// shared memory, 8 F bytes; above kShuffleMax places one thread swaps in global memory as
// before.  The MLP's 784 inputs: 155 us with
// one thread swapping, now 8.
constexpr int kShuffleMax = 25000;

__global__ void __launch_bounds__(1024) k_expand_ws(const ExpandArgs a)
{
    extern __shared__ int sh[];
    const SlotJob jb = a.jobs[blockIdx.x];
    if (jb.op != MURE_OP_WS) return;
    const uint64_t stream = splitmix64(jb.seed, (uint64_t)jb.q);
    float *out = a.patch + jb.out_off;
    const float *w = a.W[jb.layer] + (int64_t)jb.j * jb.F;
    int32_t *perm = a.perm + jb.perm_off;
    const int F = jb.F, tid = threadIdx.x, nt = blockDim.x;
    auto write = [&](int f, int v) {
        const float wp = __ldg(w + v);
        out[f] = a.ws_as_weights ? wp : wp - __ldg(w + f);
    };
    if (F > kShuffleMax) {
        for (int f = tid; f < F; f += nt) perm[f] = f;
        __syncthreads();
        if (tid == 0) {
            for (int i = F - 1; i >= 1; --i) {
                const int j = shuffle_partner(stream, F, i);
                const int32_t t = perm[i];
                perm[i] = perm[j];
                perm[j] = t;
            }
        }
        __syncthreads();
        for (int f = tid; f < F; f += nt) write(f, perm[f]);
        return;
    }
    int *head = sh, *link = sh + F;
    for (int f = tid; f < F; f += nt) head[f] = -1;
    __syncthreads();
    for (int i = 1 + tid; i < F; i += nt) link[i] = atomicExch(head + shuffle_partner(stream, F, i), i);
    __syncthreads();
    // the smallest step above i into place p (-1: none)
    auto next = [&](int p, int i) {
        int best = -1;
        for (int e = head[p]; e >= 0; e = link[e])
            if (e > i && (best < 0 || e < best)) best = e;
        return best;
    };
    // perm: A's chain; out (this thread's own places, as bits): the result's start, an index of
    // A or ~value
    for (int i = tid; i < F; i += nt) {
        perm[i] = next(i, i);
        int start = 0;
        if (i > 0) {
            const int j = shuffle_partner(stream, F, i), e = next(j, i);
            start = e >= 0 ? e : ~j;
        }
        out[i] = __int_as_float(start);
    }
    __syncthreads();
    for (int f = tid; f < F; f += nt) head[f] = perm[f];
    __syncthreads();
    for (int f = tid; f < F; f += nt) {
        const int start = __float_as_int(out[f]);
        int v = ~start;
        if (start >= 0)
            for (v = start; head[v] >= 0;) v = head[v];
        write(f, v);
    }
}

int launch_expand(const ExpandArgs &ea, cudaStream_t s)
{
    int launches = 0;
    const int f_ws = ea.max_ws <= kShuffleMax ? ea.max_ws : kShuffleMax;
    for (int64_t j0 = 0; j0 < ea.n_jobs; j0 += 65535) {
        ExpandArgs a = ea;
        a.jobs = ea.jobs + j0;
        const unsigned n = (unsigned)(ea.n_jobs - j0 < 65535 ? ea.n_jobs - j0 : 65535);
        if (ea.max_gf > 0) {
            const int chunks = (ea.max_gf - 1) / kExpandValues + 1;
            k_expand_gf<<<dim3(n, (unsigned)std::min(chunks, 1024)), kExpandValues / 2, 0, s>>>(a);
            ++launches;
        }
        if (ea.max_ws > 0) {
            const int smem = 2 * f_ws * (int)sizeof(int);
            allow_dynamic_smem(k_expand_ws, 2 * kShuffleMax * (int)sizeof(int));
            k_expand_ws<<<n, f_ws > 1024 ? 1024 : 256, smem, s>>>(a);
            ++launches;
        }
    }
    return launches;
}

// Population standard deviation of each layer's weights: two passes in fp64, fixed
// block-reduction tree.
__global__ void k_layer_std(const float *const *W, const int64_t *n, double *out)
{
    __shared__ double red[256];
    const float *w = W[blockIdx.x];
    const int64_t cnt = n[blockIdx.x];
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < cnt; i += 256) s += (double)w[i];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const double mean = red[0] / (double)cnt;
    __syncthreads();
    double ss = 0.0;
    for (int64_t i = threadIdx.x; i < cnt; i += 256) {
        const double d = (double)w[i] - mean;
        ss += d * d;
    }
    red[threadIdx.x] = ss;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sqrt(red[0] / (double)cnt);
}

int launch_layer_std(const float *const *W, const int64_t *n, int L, double *out, cudaStream_t s)
{
    if (L <= 0) return 0;
    k_layer_std<<<L, 256, 0, s>>>(W, n, out);
    return 1;
}

// ---------------------------------------------------------------------- delta --
//
// The delta of a group at layer l: the values of the mutated neurons' channels of
// x_{l+1} (after layer l's activation, skip add, pooling and GAP), computed from the
// original pre-activation z_l and, for GF / WS, the layer's input x_l.  They go to a
// compact per-row patch buffer patch[r][q][c] (slot q < kmax, output cell c of layer
// l); the first kernel of the suffix applies it on top of the unmutated row.

struct PatchValsParams {
    int ih, iw, ic, kh, kw, stride, pad, oh, ow, oc, K;
    int act1, has_add, act2, pool, gap;
    int sk_w, sk_c, sk_stride;
    int cells;           // output cells of layer l (pooled positions; 1 with GAP)
    int mcells, mcw;     // cells of the post-op map (pooled or not) and its width
    const float *z; int64_t z_stride; int z_per_input;   // channel-major [oc][oh*ow]
    const float *x; int64_t x_stride; int x_per_input;
    const float *skip; int64_t skip_stride; int skip_per_input;
    int64_t t0; int T; int G;
    PatchArgs pa;
    int kmax;
    float *out; int64_t out_stride;
    int warp_dot;        // 1: fan-in sums split across a warp (layers with < 32 positions)
    int skip_dot_ops;    // 1: GF / WS values come from k_patch_dot
    int only_dot_ops;    // 1: the other operators come from k_patch_vals_staged
    int skip_copy_ops;   // 1: NEB / NS slots are applied by the consumer (window GEMM)
    int dw;              // depthwise layer: neuron j's fan-in is its kh x kw filter on input channel j
    int embed;           // embedding: channel j at step t is table entry W[j][id_t]; GF / WS add e[id_t]
    int vocab;
    const float *W, *b;  // the layer's weights [oc][K] and biases (depthwise NS)
};

struct SlotCtx {
    const float *z, *x, *s, *e;
    int op, j, sj;
};

// NS on a depthwise layer: the two neurons exchange filters and biases, but each filter
// stays on its own output channel's input channel, so the mutated channel j is
// recomputed, b[m] + sum_k W[m][k] x_j[k] (m its partner), not taken from channel m.
__device__ __forceinline__ bool dw_switch(const PatchValsParams &p, int op) { return p.dw && op == MURE_OP_NS; }

// Mutated output of neuron j at conv position (oy, ox) after act1, skip and act2;
// `dot` is the GF / WS correction sum_k e_k x_k at that position (depthwise NS: the
// partner's filter on channel j).
__device__ __forceinline__ float slot_post(const PatchValsParams &p, const SlotCtx &d, int oy, int ox, float dot)
{
    float zz = d.z[(int64_t)d.sj * (p.oh * p.ow) + oy * p.ow + ox];
    if (dw_switch(p, d.op)) zz = dot + __ldg(p.b + d.sj);   // the forward kernel's chain: taps from +0, then + b
    else if (d.op == MURE_OP_NAI) zz = -zz;
    else if (d.op == MURE_OP_GF || d.op == MURE_OP_WS) zz = zz + dot;
    float v = d.op == MURE_OP_NEB ? 0.f : act_apply(p.act1, zz);
    if (p.has_add) {
        const float sv = d.j < p.sk_c ? d.s[((int64_t)oy * p.sk_stride * p.sk_w + ox * p.sk_stride) * p.sk_c + d.j] : 0.f;
        v = act_apply(p.act2, v + sv);
    }
    return v;
}

// sum_k e_k x_k over the receptive field of (oy, ox): one thread, ascending k.
__device__ __forceinline__ float dot_serial(const PatchValsParams &p, const SlotCtx &d, int oy, int ox)
{
    float acc = 0.f;
    if (p.embed) {
        // the one-hot input of an embedding: the term of the step's id
        const int id = (int)__ldg(d.x + ox);
        return (unsigned)id < (unsigned)p.vocab ? acc + __ldg(d.e + id) : acc;
    }
    const int iy0 = oy * p.stride - p.pad, ix0 = ox * p.stride - p.pad;
    if (p.dw) {
        // a depthwise neuron: its filter taps (ky, kx) on input channel j
        for (int ky = 0; ky < p.kh; ++ky) {
            const int iy = iy0 + ky;
            for (int kx = 0; kx < p.kw; ++kx) {
                const int ix = ix0 + kx;
                if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
                    acc = fmaf(__ldg(d.e + ky * p.kw + kx), __ldg(d.x + ((int64_t)iy * p.iw + ix) * p.ic + d.j), acc);
            }
        }
        return acc;
    }
    int k = 0;
    for (int ky = 0; ky < p.kh; ++ky) {
        const int iy = iy0 + ky;
        for (int kx = 0; kx < p.kw; ++kx, k += p.ic) {
            const int ix = ix0 + kx;
            if ((unsigned)iy >= (unsigned)p.ih || (unsigned)ix >= (unsigned)p.iw) continue;
            const float *xp = d.x + ((int64_t)iy * p.iw + ix) * p.ic;
            const float *ep = d.e + k;
            for (int ci = 0; ci < p.ic; ++ci) acc = fmaf(__ldg(ep + ci), __ldg(xp + ci), acc);
        }
    }
    return acc;
}

// The same sum with a warp: lane i takes k = i, i+32, ... in ascending order, then a
// butterfly over the lanes; every lane ends with the same value.
__device__ __forceinline__ float dot_warp(const PatchValsParams &p, const SlotCtx &d, int oy, int ox, int lane)
{
    float acc = 0.f;
    if (p.embed) {
        // one term: every lane returns it (no butterfly)
        const int id = (int)__ldg(d.x + ox);
        return (unsigned)id < (unsigned)p.vocab ? acc + __ldg(d.e + id) : acc;
    }
    const int iy0 = oy * p.stride - p.pad, ix0 = ox * p.stride - p.pad;
    if (p.dw) {
        for (int k = lane; k < p.K; k += 32) {
            const int ky = k / p.kw, kx = k - ky * p.kw, iy = iy0 + ky, ix = ix0 + kx;
            if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
                acc = fmaf(__ldg(d.e + k), __ldg(d.x + ((int64_t)iy * p.iw + ix) * p.ic + d.j), acc);
        }
    } else if (p.kh == 1 && p.kw == 1 && p.ih == 1 && p.iw == 1) {
        for (int k = lane; k < p.K; k += 32) acc = fmaf(__ldg(d.e + k), __ldg(d.x + k), acc);
    } else {
        for (int k = lane; k < p.K; k += 32) {
            const int ci = k % p.ic, t = k / p.ic, kx = t % p.kw, ky = t / p.kw;
            const int iy = iy0 + ky, ix = ix0 + kx;
            if ((unsigned)iy < (unsigned)p.ih && (unsigned)ix < (unsigned)p.iw)
                acc = fmaf(__ldg(d.e + k), __ldg(d.x + ((int64_t)iy * p.iw + ix) * p.ic + ci), acc);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    return acc;
}

// Value of map cell c (a pooled window or one position) of slot d.  In warp-dot
// mode every lane of the warp must call it with the same c.
__device__ __forceinline__ float cell_value(const PatchValsParams &p, const SlotCtx &d, int c, int lane)
{
    const bool dot = d.op == MURE_OP_GF || d.op == MURE_OP_WS || dw_switch(p, d.op);
    const int cy = c / p.mcw, cx = c % p.mcw;
    if (!p.pool) {
        const float dv = dot ? (p.warp_dot ? dot_warp(p, d, cy, cx, lane) : dot_serial(p, d, cy, cx)) : 0.f;
        return slot_post(p, d, cy, cx, dv);
    }
    float w4[4];
#pragma unroll
    for (int sub = 0; sub < 4; ++sub) {
        const int oy = 2 * cy + (sub >> 1), ox = 2 * cx + (sub & 1);
        const float dv = dot ? (p.warp_dot ? dot_warp(p, d, oy, ox, lane) : dot_serial(p, d, oy, ox)) : 0.f;
        w4[sub] = slot_post(p, d, oy, ox, dv);
    }
    return max4_first(w4[0], w4[1], w4[2], w4[3]);
}

// One warp per (mutant g, slot q) of one input (blockIdx.y), so the mutants of an
// input read its z and x while they are in L2; the warp's lanes take the cells (one
// lane per cell), or, for layers with fewer than 32 positions, share each cell's dot
// product.
__global__ void __launch_bounds__(256) k_patch_vals(const PatchValsParams p)
{
    extern __shared__ float gap_buf[];  // [8][mcells] with GAP in lane mode
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int item = (int)blockIdx.x * 8 + warp;     // warp-uniform
    if (item >= p.G * p.kmax) return;
    const int g = item / p.kmax, q = item - g * p.kmax;
    if (q >= p.pa.n_neurons[g]) return;
    const int op = p.pa.op[g];
    const bool gfws = op == MURE_OP_GF || op == MURE_OP_WS;
    const bool dot = gfws || dw_switch(p, op);
    if (gfws && p.skip_dot_ops) return;
    if (!dot && p.only_dot_ops) return;
    const int32_t *ids = p.pa.ids + p.pa.neuron_off[g];
    SlotCtx d;
    d.op = op;
    d.j = ids[q];
    d.sj = op == MURE_OP_NS ? ids[q ^ 1] : d.j;
    // the fan-in terms of the sum: GF / WS patch, or (depthwise NS) the partner's filter
    const float *e = gfws ? p.pa.patch + p.pa.patch_off[g] + (int64_t)q * p.K
                          : dot ? p.W + (int64_t)d.sj * p.K : nullptr;
    if (!dot && (p.warp_dot || p.cells < 32)) {
        // no fan-in sum and few cells: one input per lane, its cells in order (a GAP
        // value is the same ascending sum over the map cells as below)
        for (int tl = blockIdx.y * 32 + lane; tl < p.T; tl += gridDim.y * 32) {
            const int64_t r = (int64_t)g * p.T + tl, t = p.t0 + tl;
            d.z = p.z + (p.z_per_input ? t : r) * p.z_stride;
            d.x = nullptr;
            d.s = p.has_add ? p.skip + (p.skip_per_input ? t : r) * p.skip_stride : nullptr;
            d.e = nullptr;
            float *o = p.out + r * p.out_stride + q * p.cells;
            if (p.gap) {
                float s = 0.f;
                for (int cc = 0; cc < p.mcells; ++cc) s += cell_value(p, d, cc, lane);
                o[0] = s / (float)p.mcells;
            } else {
                for (int c = 0; c < p.cells; ++c) o[c] = cell_value(p, d, c, lane);
            }
        }
        return;
    }
    for (int tl = blockIdx.y; tl < p.T; tl += gridDim.y) {
        const int64_t r = (int64_t)g * p.T + tl, t = p.t0 + tl;
        d.z = p.z + (p.z_per_input ? t : r) * p.z_stride;
        d.x = dot ? p.x + (p.x_per_input ? t : r) * p.x_stride : nullptr;
        d.s = p.has_add ? p.skip + (p.skip_per_input ? t : r) * p.skip_stride : nullptr;
        d.e = e;
        float *o = p.out + r * p.out_stride + q * p.cells;
        if (p.gap) {
            // the map cells, then their ascending fp32 sum / count
            float s = 0.f;
            if (p.warp_dot) {
                for (int cc = 0; cc < p.mcells; ++cc) s += cell_value(p, d, cc, lane);
            } else {
                float *gb = gap_buf + warp * p.mcells;
                for (int cc = lane; cc < p.mcells; cc += 32) gb[cc] = cell_value(p, d, cc, lane);
                __syncwarp();
                for (int cc = 0; cc < p.mcells; ++cc) s += gb[cc];
                __syncwarp();
            }
            if (lane == 0) o[0] = s / (float)p.mcells;
        } else if (p.warp_dot) {
            for (int c = 0; c < p.cells; ++c) {
                const float v = cell_value(p, d, c, lane);
                if (lane == 0) o[c] = v;
            }
        } else {
            for (int c = lane + 32 * blockIdx.z; c < p.cells; c += 32 * gridDim.z) o[c] = cell_value(p, d, c, lane);
        }
    }
}

// The operators without a fan-in sum (NAI, NEB, NS) of a convolution layer in
// memoized mode, one input per block: the input's cached pre-activation maps are
// staged in shared memory once and every mutant slot of the batch reads its channel
// there (the mutants of a batch share the inputs).  The arithmetic is slot_post's,
// so the values equal those of k_patch_vals bit for bit.
template <bool PAIR>
__global__ void __launch_bounds__(256) k_patch_vals_staged(const PatchValsParams p)
{
    extern __shared__ __align__(16) float zs[];   // [oc][oh * ow] of the block's input, then the cell table
    const int P = p.oh * p.ow, nz = p.oc * P;
    int *coff = reinterpret_cast<int *>(zs + nz);   // cell -> top-left position of its window
    const int tl = blockIdx.x;
    const float *z = p.z + (p.t0 + tl) * p.z_stride;
    for (int i = threadIdx.x; i < nz; i += blockDim.x) zs[i] = z[i];
    for (int c = threadIdx.x; c < p.mcells; c += blockDim.x)
        coff[c] = p.pool ? 2 * (c / p.mcw) * p.ow + 2 * (c % p.mcw) : c;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the batch's NEB / NAI / NS slots (listed by the host), one warp per slot
    for (int64_t sl = warp; sl < p.pa.n_vslot; sl += blockDim.x >> 5) {
        const int4 e = p.pa.vslot[sl];
        const int g = e.x - p.pa.dslot_g0, q = e.y, sj = e.z, op = e.w;
        if (p.skip_copy_ops && (op == MURE_OP_NEB || op == MURE_OP_NS)) continue;
        const float *zc = zs + sj * P;
        float *o = p.out + ((int64_t)g * p.T + tl) * p.out_stride + q * p.cells;
        auto post = [&](float zz) {
            if (op == MURE_OP_NAI) zz = -zz;
            return op == MURE_OP_NEB ? 0.f : act_apply(p.act1, zz);
        };
        auto cell = [&](int c) {
            const int b = coff[c];
            return p.pool ? max4_first(post(zc[b]), post(zc[b + 1]), post(zc[b + p.ow]), post(zc[b + p.ow + 1]))
                          : post(zc[b]);
        };
        if constexpr (PAIR) {
            // two neighbouring pooling windows per lane: their 2x4 inputs are two
            // 16-byte loads (the host checks the alignment), one 8-byte store
            for (int c = 2 * lane; c < p.cells; c += 64) {
                float2 r;
                if (op == MURE_OP_NEB) {
                    r = make_float2(0.f, 0.f);
                } else {
                    const int b = coff[c];
                    const float4 u = *reinterpret_cast<const float4 *>(zc + b);
                    const float4 v = *reinterpret_cast<const float4 *>(zc + b + p.ow);
                    r.x = max4_first(post(u.x), post(u.y), post(v.x), post(v.y));
                    r.y = max4_first(post(u.z), post(u.w), post(v.z), post(v.w));
                }
                *reinterpret_cast<float2 *>(o + c) = r;
            }
        } else {
            for (int c = lane; c < p.cells; c += 32) o[c] = cell(c);
        }
    }
}

// Dense layers in memoized mode, kDenseIn inputs per block: the inputs' cached rows
// x and pre-activations z are staged in shared memory; a thread per (slot, input)
// copies the operators without a fan-in sum, a warp per GF / WS slot (the host's list)
// keeps its delta row in registers and forms the dot products of the block's inputs
// exactly as dot_warp does (lane i sums k = i, i+32, ... ascending, then a butterfly).
constexpr int kDenseIn = 8;
constexpr int kDenseKMax = 1024;

template <int KPER>
__global__ void __launch_bounds__(256) k_patch_vals_dense_in(const PatchValsParams p)
{
    extern __shared__ float sm2[];
    const int K = p.K, OC = p.oc;
    float *xs = sm2;                     // [kDenseIn][K]
    float *zs = xs + kDenseIn * K;       // [kDenseIn][OC]
    const int tl0 = blockIdx.x * kDenseIn;
    const int ni = min(kDenseIn, p.T - tl0);
    for (int i = threadIdx.x; i < ni * K; i += blockDim.x) {
        const int a = i / K, k = i - a * K;
        xs[i] = __ldg(p.x + (p.t0 + tl0 + a) * p.x_stride + k);
    }
    for (int i = threadIdx.x; i < ni * OC; i += blockDim.x) {
        const int a = i / OC, c = i - a * OC;
        zs[i] = __ldg(p.z + (p.t0 + tl0 + a) * p.z_stride + c);
    }
    __syncthreads();
    // operators without a fan-in sum
    for (int it = threadIdx.x; it < p.G * p.kmax * kDenseIn; it += blockDim.x) {
        const int sl = it / kDenseIn, a = it - sl * kDenseIn;
        const int g = sl / p.kmax, q = sl - g * p.kmax;
        if (a >= ni || q >= p.pa.n_neurons[g]) continue;
        const int op = p.pa.op[g];
        if (op == MURE_OP_GF || op == MURE_OP_WS) continue;
        const int32_t *ids = p.pa.ids + p.pa.neuron_off[g];
        const int sj = op == MURE_OP_NS ? ids[q ^ 1] : ids[q];
        float zz = zs[a * OC + sj];
        if (op == MURE_OP_NAI) zz = -zz;
        p.out[((int64_t)g * p.T + tl0 + a) * p.out_stride + q] = op == MURE_OP_NEB ? 0.f : act_apply(p.act1, zz);
    }
    // GF / WS: a warp per slot
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kPer = KPER;   // >= ceil(K / 32): the unrolled loop has no dead steps
    for (int64_t s2 = warp; s2 < p.pa.n_dslot; s2 += blockDim.x >> 5) {
        const int g = p.pa.dslot[2 * s2] - p.pa.dslot_g0, q = p.pa.dslot[2 * s2 + 1];
        const int j = p.pa.ids[p.pa.neuron_off[g] + q];
        const float *e = p.pa.patch + p.pa.patch_off[g] + (int64_t)q * K;
        float ev[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) ev[i] = lane + 32 * i < K ? __ldg(e + lane + 32 * i) : 0.f;
        for (int a = 0; a < ni; ++a) {
            const float *xa = xs + a * K;
            float acc = 0.f;
#pragma unroll
            for (int i = 0; i < kPer; ++i)
                if (lane + 32 * i < K) acc = fmaf(ev[i], xa[lane + 32 * i], acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0)
                p.out[((int64_t)g * p.T + tl0 + a) * p.out_stride + q] = act_apply(p.act1, zs[a * OC + j] + acc);
        }
    }
}

// Dense layers whose rows have their own z (vanilla rows, later layers of multi-layer mutants):
// a warp per (mutant, RPW of its rows), every slot of a row at once.  Operators without a
// fan-in sum: a row's slots on neighbouring lanes, 32 / slots rows per load.  GF / WS: the
// weight deltas of SG slots stay in registers for all the warp's rows, a row is loaded once for
// them, and each sum is dot_warp's (lane i takes k = i, i + 32, ... ascending, then the
// butterfly; with SG values the halves of the warp each keep half of them at the first exchanges,
// which adds the same pairs).  It was a warp per (mutant, slot), which read every row again for
// each of its slots: FC 400-120 of LeNet-5's 3 % model-wide mutants, 279,000 rows, 280 us and 16 more
// to move the patch into the rows, now 164.  Writes the patch, or (y non-null) the neurons' places in the rows themselves.
template <int KPER>
__global__ void __launch_bounds__(256, KPER <= 16 ? 2 : 1) k_patch_dense_rows(const PatchValsParams p, float *y, int64_t y_stride, int rpw)
{
    constexpr int SG = KPER <= 16 ? 4 : 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = blockIdx.x;
    const int n = p.pa.n_neurons[g];
    if (n == 0) return;
    const int op = p.pa.op[g];
    const int32_t *ids = p.pa.ids + p.pa.neuron_off[g];
    const int tl0 = (blockIdx.y * 8 + warp) * rpw, tl1 = min(tl0 + rpw, p.T);
    auto put = [&](int64_t r, int q, int j, float v) {
        if (y) y[r * y_stride + j] = v;
        else p.out[r * p.out_stride + q] = v;
    };
    if (op != MURE_OP_GF && op != MURE_OP_WS) {
        int w = 1;   // lanes per row
        while (w < n && w < 32) w <<= 1;
        for (int q = lane % w; q < n; q += w) {
            const int j = ids[q], sj = op == MURE_OP_NS ? ids[q ^ 1] : j;
#pragma unroll 4
            for (int tl = tl0 + lane / w; tl < tl1; tl += 32 / w) {
                const int64_t r = (int64_t)g * p.T + tl;
                float zz = op == MURE_OP_NEB ? 0.f : __ldg(p.z + (p.z_per_input ? p.t0 + tl : r) * p.z_stride + sj);
                if (op == MURE_OP_NAI) zz = -zz;
                put(r, q, j, op == MURE_OP_NEB ? 0.f : act_apply(p.act1, zz));
            }
        }
        return;
    }
    const float *e = p.pa.patch + p.pa.patch_off[g];
    for (int q0 = 0; q0 < n; q0 += SG) {
        float ev[SG][KPER];
#pragma unroll
        for (int a = 0; a < SG; ++a)
#pragma unroll
            for (int i = 0; i < KPER; ++i)
                ev[a][i] = q0 + a < n && lane + 32 * i < p.K ? __ldg(e + (int64_t)(q0 + a) * p.K + lane + 32 * i) : 0.f;
        // the slot whose sum this lane ends with
        const int hi = lane >> 4 & 1, b = lane >> 3 & 1, mine = q0 + (SG == 4 ? 2 * hi + b : hi);
        const int j = mine < n ? ids[mine] : 0;
        for (int tl = tl0; tl < tl1; ++tl) {
            const int64_t r = (int64_t)g * p.T + tl, t = p.t0 + tl;
            const float *xr = p.x + (p.x_per_input ? t : r) * p.x_stride;
            const float zv = __ldg(p.z + (p.z_per_input ? t : r) * p.z_stride + j);
            float acc[SG];
#pragma unroll
            for (int a = 0; a < SG; ++a) acc[a] = 0.f;
            float xv[KPER];
#pragma unroll
            for (int i = 0; i < KPER; ++i) xv[i] = lane + 32 * i < p.K ? __ldg(xr + lane + 32 * i) : 0.f;
#pragma unroll
            for (int i = 0; i < KPER; ++i)
                if (lane + 32 * i < p.K) {
#pragma unroll
                    for (int a = 0; a < SG; ++a) acc[a] = fmaf(ev[a][i], xv[i], acc[a]);
                }
            float sum;
            if constexpr (SG == 4) {
                const float s0 = (hi ? acc[2] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[2], 16);
                const float s1 = (hi ? acc[3] : acc[1]) + __shfl_xor_sync(0xffffffffu, hi ? acc[1] : acc[3], 16);
                sum = (b ? s1 : s0) + __shfl_xor_sync(0xffffffffu, b ? s0 : s1, 8);
            } else {
                sum = (hi ? acc[1] : acc[0]) + __shfl_xor_sync(0xffffffffu, hi ? acc[0] : acc[1], 16);
                sum += __shfl_xor_sync(0xffffffffu, sum, 8);
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if ((lane & (SG == 4 ? 7 : 15)) == 0 && mine < n) put(r, mine, j, act_apply(p.act1, zv + sum));
        }
    }
}

int patch_rows_supported(const Stage &S, Src z)
{
    return S.kind == MURE_NODE_DENSE && !z.per_input && !S.has_add && !S.gap && !S.pool && S.oh * S.ow == 1 &&
           S.K <= kDenseKMax;
}

static int launch_dense_rows(const PatchValsParams &p, float *y, int64_t y_stride, cudaStream_t s)
{
    // rows per warp: enough to pay for the deltas in registers, few enough to fill the GPU
    int rpw = 8;
    while (rpw < 32 && (int64_t)p.G * p.T > (int64_t)sm_count() * 64 * rpw) rpw *= 2;
    while ((p.T + 8 * rpw - 1) / (8 * rpw) > 65535) rpw *= 2;
    const dim3 grid((unsigned)p.G, (unsigned)((p.T + 8 * rpw - 1) / (8 * rpw)));
    if (p.K <= 128) k_patch_dense_rows<4><<<grid, 256, 0, s>>>(p, y, y_stride, rpw);
    else if (p.K <= 256) k_patch_dense_rows<8><<<grid, 256, 0, s>>>(p, y, y_stride, rpw);
    else if (p.K <= 512) k_patch_dense_rows<16><<<grid, 256, 0, s>>>(p, y, y_stride, rpw);
    else k_patch_dense_rows<kDenseKMax / 32><<<grid, 256, 0, s>>>(p, y, y_stride, rpw);
    return 1;
}

static PatchValsParams patch_vals_params(const Stage &S, Src z, Src x, Src skip, RowMap rm, const PatchArgs &pa, int kmax)
{
    PatchValsParams p{};
    p.ih = S.ih; p.iw = S.iw; p.ic = S.ic; p.kh = S.kh; p.kw = S.kw; p.stride = S.stride; p.pad = S.pad;
    p.oh = S.oh; p.ow = S.ow; p.oc = S.oc; p.K = S.K;
    p.act1 = S.act1; p.has_add = S.has_add; p.act2 = S.act2; p.pool = S.pool; p.gap = S.gap;
    p.sk_w = S.sk_w; p.sk_c = S.sc_c; p.sk_stride = S.sc_stride;
    p.mcw = S.pool ? S.ow / 2 : S.ow;
    p.mcells = (S.pool ? S.oh / 2 : S.oh) * p.mcw;
    p.cells = S.gap ? 1 : p.mcells;
    p.z = z.p; p.z_stride = z.stride; p.z_per_input = z.per_input;
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.skip = skip.p; p.skip_stride = skip.stride; p.skip_per_input = skip.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.G = rm.R / rm.T;
    p.pa = pa;
    p.kmax = kmax;
    p.warp_dot = (S.oh * S.ow) < 32;
    p.dw = S.kind == MURE_NODE_DWCONV;
    p.embed = S.kind == MURE_NODE_EMBED;
    p.vocab = S.vocab;
    p.W = S.W;
    p.b = S.b;
    return p;
}

int launch_patch_rows(const Stage &S, Src z, Src x, RowMap rm, const PatchArgs &pa, int kmax, float *y, int64_t y_stride,
                      cudaStream_t s)
{
    if (rm.R <= 0 || kmax <= 0) return 0;
    return launch_dense_rows(patch_vals_params(S, z, x, Src{nullptr, 0, 0}, rm, pa, kmax), y, y_stride, s);
}

int launch_patch_vals(const Stage &S, Src z, Src x, Src skip, RowMap rm, const PatchArgs &pa, int kmax, float *out,
                      int64_t out_stride, cudaStream_t s, bool skip_dot_ops, bool skip_copy_ops)
{
    if (rm.R <= 0 || kmax <= 0) return 0;
    PatchValsParams p = patch_vals_params(S, z, x, skip, rm, pa, kmax);
    p.out = out; p.out_stride = out_stride;
    p.skip_dot_ops = skip_dot_ops;
    p.skip_copy_ops = skip_copy_ops;
    if (patch_rows_supported(S, z) && !skip_dot_ops) return launch_dense_rows(p, nullptr, 0, s);
    const int64_t n_items = (int64_t)p.G * kmax;
    // each warp walks several inputs (blockIdx.y, +gridDim.y, ...): enough blocks to
    // fill the GPU, few enough that block scheduling stays negligible.  Without fan-in
    // sums in the launch, a layer of fewer than 32 cells takes a lane per input (32 inputs
    // per block row), so more than ceil(T / 32) block rows would only idle (ncu: 4 x 608
    // blocks for 2,048 inputs of VGG's conv 256->256, most of them empty)
    const int64_t gx = (n_items + 7) / 8;
    const bool lane_per_input = skip_dot_ops && S.kind != MURE_NODE_DWCONV && (p.warp_dot || p.cells < 32);
    const int64_t gy = std::max<int64_t>(1, std::min<int64_t>(lane_per_input ? (rm.T + 31) / 32 : rm.T,
                                                              (sm_count() * 16 + gx - 1) / gx));
    // few slots and inputs: a slot's cells are split over blocks too (MobileNetV2's depthwise
    // layers, 4 mutants x 320 inputs on 320 blocks: 20 launches of a job 1.00 ms, now 0.59)
    const int64_t gz = !S.gap && !p.warp_dot
                           ? std::max<int64_t>(1, std::min<int64_t>(p.cells / 64, sm_count() * 16 / std::max<int64_t>(gx * gy, 1)))
                           : 1;
    const dim3 grid((unsigned)gx, (unsigned)gy, (unsigned)gz);
    const size_t smem = (S.gap && !p.warp_dot) ? 8 * (size_t)p.mcells * sizeof(float) : 0;
    // memoized dense layers: all operators per block of inputs
    if (z.per_input && x.per_input && S.kind == MURE_NODE_DENSE && !S.has_add && !S.gap && !S.pool &&
        S.K <= kDenseKMax && S.oh * S.ow == 1) {
        const size_t sm = (size_t)kDenseIn * (S.K + S.oc) * 4;
        if (sm <= 48 * 1024) {
            const unsigned blocks = (unsigned)((rm.T + kDenseIn - 1) / kDenseIn);
            // the unrolled dot loop sized to the fan-in (measured on the LeNet-5
            // workload: FC 400-120 0.222 -> 0.148 ms, FC 120-84 0.207 -> 0.106 ms)
            if (S.K <= 128) k_patch_vals_dense_in<4><<<blocks, 256, sm, s>>>(p);
            else if (S.K <= 256) k_patch_vals_dense_in<8><<<blocks, 256, sm, s>>>(p);
            else if (S.K <= 512) k_patch_vals_dense_in<16><<<blocks, 256, sm, s>>>(p);
            else k_patch_vals_dense_in<kDenseKMax / 32><<<blocks, 256, sm, s>>>(p);
            return 1;
        }
    }
    // memoized convolution layers whose maps fit in shared memory: the non-dot
    // operators per input, staged
    const size_t staged_smem = ((size_t)S.oc * S.oh * S.ow + p.mcells) * 4;
    const bool staged = z.per_input && S.kind == MURE_NODE_CONV2D && !S.has_add && !S.gap &&
                        staged_smem <= 48 * 1024;
    int launches = 0;
    if (staged) {
        if (pa.n_vslot > 0) {
            // pairs of windows: even window columns, 16-byte aligned rows and slots
            // (measured on conv 1->6: the delta of 400 mutants x 10,000 inputs
            // 3.20 -> 3.02 ms)
            const bool pair = S.pool && p.mcw % 2 == 0 && S.ow % 4 == 0 && p.cells % 2 == 0 && out_stride % 2 == 0 &&
                              (reinterpret_cast<uintptr_t>(out) & 7) == 0 && (S.oh * S.ow) % 4 == 0;
            if (pair) k_patch_vals_staged<true><<<(unsigned)rm.T, 256, staged_smem, s>>>(p);
            else k_patch_vals_staged<false><<<(unsigned)rm.T, 256, staged_smem, s>>>(p);
            ++launches;
        }
        if (skip_dot_ops) return launches;
        p.only_dot_ops = 1;
    }
    k_patch_vals<<<grid, 256, smem, s>>>(p);
    return launches + 1;
}

// Materialise rows: out = base with the overlay's channels written in (for suffix kernels
// that read plain rows), TPR threads per row: a warp, or the whole block where eight rows don't
// fit 48 KiB.  16-byte copies through shared memory, the patch written there in between.  A row
// waits on a chain of loads (its mutant's neurons, then the patch), so what counts is rows in
// flight and that the chain starts with the copy and all lanes follow it at once.  140,800 rows
// of LeNet's 14 x 14 x 6 maps: one element per thread and index division 507 us, a block per row
// 311, now 164 (97 the writes); 279,000 rows of 120 values, a channel at a time per row 123 us,
// now 63.
template <int TPR>
__global__ void __launch_bounds__(256) k_rows_overlay(const float *__restrict__ base, int64_t base_stride,
                                                      int base_per_input, int64_t t0, int T, int R, int n4,
                                                      const Overlay ov, float *out, int64_t out_stride,
                                                      const int32_t *lrow)
{
    extern __shared__ __align__(16) float sm[];  // [256 / TPR][4 n4]
    const int tid = threadIdx.x % TPR;
    const int64_t r = (int64_t)blockIdx.x * (256 / TPR) + threadIdx.x / TPR;
    float *row = sm + (threadIdx.x / TPR) * 4 * n4;
    const bool ok = r < R;
    const int64_t lr = ok ? logical_row(lrow, r) : 0;
    const uint32_t g = (uint32_t)lr / (uint32_t)T;   // (a batch's rows are below 2^31)
    const int n = ok ? __ldg(ov.n_neurons + g) : 0;
    const int32_t *ids = ov.ids + (ok ? __ldg(ov.neuron_off + g) : 0);
    auto sync = [] {
        if (TPR == 32) __syncwarp();
        else __syncthreads();
    };
    if (ok) {
        const float4 *src =
            reinterpret_cast<const float4 *>(base + (base_per_input ? t0 + (lr - (int64_t)g * T) : r) * base_stride);
#pragma unroll 4
        for (int i = tid; i < n4; i += TPR) reinterpret_cast<float4 *>(row)[i] = __ldg(src + i);
    }
    sync();
    if (ok) {
        // every lane takes values of every mutated channel: value i is cell i mod cells of channel
        // i / cells
        const float *patch = ov.patch + lr * ov.row_stride;
        const uint32_t cells = (uint32_t)ov.cells;
#pragma unroll 2
        for (uint32_t i = tid; i < n * cells; i += TPR) {
            const uint32_t q = i / cells;
            row[(i - q * cells) * ov.ch + __ldg(ids + q)] = __ldg(patch + i);
        }
    }
    sync();
    if (ok) {
        float4 *dst = reinterpret_cast<float4 *>(out + r * out_stride);
#pragma unroll 4
        for (int i = tid; i < n4; i += TPR) dst[i] = reinterpret_cast<const float4 *>(row)[i];
    }
}

// Large rows: copy the base rows, then scatter the overlay (two ordered launches).  A block copies
// 1,024 16-byte pieces of a row, four per thread in flight (an index division and a load at a time
// per thread: 127 us for ResNet-20's four copies of a job, now 102; MobileNet's eight 300, now 256).
__global__ void __launch_bounds__(256) k_copy_rows(const float4 *__restrict__ src, int64_t src_stride4, int per_input, int n4,
                                                   int chunks, int64_t t0, int T, float4 *__restrict__ dst,
                                                   int64_t dst_stride4, const int32_t *lrow)
{
    const uint32_t r = blockIdx.x / chunks;
    const int e0 = (int)(blockIdx.x - r * chunks) * 1024 + threadIdx.x;
    const float4 *s = src + (per_input ? t0 + (uint32_t)logical_row(lrow, r) % (uint32_t)T : r) * src_stride4;
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (e0 + 256 * i < n4) v[i] = __ldg(s + e0 + 256 * i);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (e0 + 256 * i < n4) dst[r * dst_stride4 + e0 + 256 * i] = v[i];
}

__global__ void k_overlay_scatter(int64_t T, int64_t R, const Overlay ov, float *out, int64_t out_stride,
                                  const int32_t *lrow)
{
    const int64_t per_row = (int64_t)ov.kmax * ov.cells;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < R * per_row;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / per_row, lr = logical_row(lrow, r);
        const int rem = (int)(i - r * per_row), q = rem / ov.cells, c = rem - q * ov.cells;
        const uint32_t g = (uint32_t)lr / (uint32_t)T;
        if (q >= ov.n_neurons[g]) continue;
        const int j = ov.ids[ov.neuron_off[g] + q];
        out[r * out_stride + (int64_t)c * ov.ch + j] = ov.patch[lr * ov.row_stride + q * ov.cells + c];
    }
}

int launch_rows_overlay(Src base, int64_t n_floats, RowMap rm, const Overlay &ov, float *out, int64_t out_stride,
                        cudaStream_t s)
{
    if (rm.R <= 0) return 0;
    // large rows, or rows patched in place (only the mutated channels are written)
    if (n_floats > 8192 || (base.p == out && !base.per_input)) {
        int launches = 0;
        if (!(base.p == out && !base.per_input)) {
            const int64_t n4 = (n_floats + 3) / 4, chunks = (n4 + 1023) / 1024;
            k_copy_rows<<<(unsigned)(rm.R * chunks), 256, 0, s>>>(reinterpret_cast<const float4 *>(base.p), base.stride / 4,
                                                                 base.per_input, (int)n4, (int)chunks, rm.t0, rm.T,
                                                                 reinterpret_cast<float4 *>(out), out_stride / 4, rm.lrow);
            ++launches;
        }
        const int64_t total = (int64_t)rm.R * ov.kmax * ov.cells;
        if (total > 0) {
            const int64_t blocks = std::min<int64_t>((total + 255) / 256, (int64_t)sm_count() * 64);
            k_overlay_scatter<<<(unsigned)blocks, 256, 0, s>>>(rm.T, rm.R, ov, out, out_stride, rm.lrow);
            ++launches;
        }
        return launches;
    }
    const int n4 = (int)((n_floats + 3) / 4);   // rows are whole 16-byte pieces
    const int per_block = n4 <= 384 ? 8 : 1;    // (8 rows in 48 KiB)
    const size_t smem = (size_t)per_block * n4 * 16;
    const unsigned blocks = (unsigned)((rm.R + per_block - 1) / per_block);
    if (per_block == 8)
        k_rows_overlay<32><<<blocks, 256, smem, s>>>(base.p, base.stride, base.per_input, rm.t0, rm.T, rm.R, n4, ov, out,
                                                     out_stride, rm.lrow);
    else
        k_rows_overlay<256><<<blocks, 256, smem, s>>>(base.p, base.stride, base.per_input, rm.t0, rm.T, rm.R, n4, ov, out,
                                                      out_stride, rm.lrow);
    return 1;
}

// --------------------------------------------------------------------- scores --

__global__ void __launch_bounds__(128) k_scores(const uint32_t *__restrict__ kill32, int64_t n_mut, int64_t words32,
                                                const int32_t *__restrict__ label, unsigned long long *totals)
{
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (i >= n_mut) return;
    // the set of killing labels as kLabelWords 32-bit words (up to kMaxClasses labels)
    uint32_t any = 0, labels[kLabelWords] = {};
    for (int64_t w = lane; w < words32; w += 32) {
        uint32_t bits = kill32[i * words32 + w];
        any |= bits;
        while (bits) {
            const int b = __ffs(bits) - 1;
            const int lb = label[w * 32 + b];
#pragma unroll
            for (int k = 0; k < kLabelWords; ++k)
                if ((lb >> 5) == k) labels[k] |= 1u << (lb & 31);
            bits &= bits - 1;
        }
    }
    int count = 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
#pragma unroll
    for (int k = 0; k < kLabelWords; ++k) {
        uint32_t m = labels[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m |= __shfl_xor_sync(0xffffffffu, m, o);
        count += __popc(m);
    }
    if (lane == 0) {
        if (any) atomicAdd(&totals[0], 1ull);
        atomicAdd(&totals[1], (unsigned long long)count);
    }
}

int launch_scores(const uint32_t *kill32, int64_t n_mut, int64_t words32, const int32_t *label, int n_classes,
                  unsigned long long *totals, cudaStream_t s)
{
    (void)n_classes;
    if (n_mut <= 0) return 0;
    k_scores<<<(unsigned)((n_mut + 3) / 4), 128, 0, s>>>(kill32, n_mut, words32, label, totals);
    return 1;
}

__global__ void k_label_set(const int32_t *__restrict__ label, int64_t n, uint32_t *mask)
{
    uint32_t m[kLabelWords] = {};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int lb = label[i];
#pragma unroll
        for (int k = 0; k < kLabelWords; ++k)
            if ((lb >> 5) == k) m[k] |= 1u << (lb & 31);
    }
#pragma unroll
    for (int k = 0; k < kLabelWords; ++k) {
        uint32_t v = m[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicOr(mask + k, v);
    }
}

int launch_label_set(const int32_t *label, int64_t n, uint32_t *mask, cudaStream_t s)
{
    if (n <= 0) return 0;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 1024) blocks = 1024;
    k_label_set<<<(unsigned)blocks, 256, 0, s>>>(label, n, mask);
    return 1;
}

__global__ void __launch_bounds__(256) k_pack_rows(const float *__restrict__ in, int64_t in_stride, int n, int64_t total,
                                                   float *__restrict__ out)
{
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < total; i += (int64_t)gridDim.x * 256)
        out[i] = in[i / n * in_stride + i % n];
}

int launch_pack_rows(const float *in, int64_t in_stride, int n, int64_t R, float *out, cudaStream_t s)
{
    const int64_t total = R * n;
    if (total <= 0) return 0;
    k_pack_rows<<<(unsigned)std::min<int64_t>((total + 255) / 256, 4096), 256, 0, s>>>(in, in_stride, n, total, out);
    return 1;
}

}  // namespace mure
