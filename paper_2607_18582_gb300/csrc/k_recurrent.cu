// The recurrent family (the paper's RNN models, Sec. 5.3 / Table 1): an embedding of
// token ids and LSTM layers.  Sequences are rows of 1 x T x C values (NHWC with
// H = 1); the ids are integers held in floats.
//
// An LSTM neuron is a unit: its fan-in is the four gate rows of input and recurrent
// weights, W[j][gate][0 .. cin + H), and its biases b[j][gate].  A mutant of an LSTM
// layer changes that layer's whole output from the first step on (the recurrence feeds
// every unit's h to every unit), so there is no channel patch: the layer is recomputed
// for every row of the mutant from its cached input, with the mutated units' rows
// rewritten on the fly (GF / WS: W + e, NAI: -W and -b, NS: the partner's rows and
// biases, NEB: h_j held at 0), and the suffix runs from its output.
#include <climits>
#include "common.cuh"
#include "device_util.cuh"
#include "simt_tile.cuh"

namespace mure {

namespace {

// --------------------------------------------------------------- embedding --

struct EmbedParams {
    const float *x; int64_t x_stride; int x_per_input;   // ids [row][T]
    int64_t t0; int T; int R;
    const int32_t *lrow;
    int steps, dim, vocab;
    const float *Wt;      // [vocab][dim]
    float *z; int64_t z_stride;   // channel-major [dim][steps] (nullable)
    float *y; int64_t y_stride;   // [steps][dim]
    int *err;
};

// Position t, channel j of a row: W[j][id_t].  An id outside [0, vocab) records
// INVALID_ARG in the context's error word and reads entry 0 (no access outside the
// table).
__global__ void __launch_bounds__(256) k_embed(const EmbedParams p)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t per_row = (int64_t)p.steps * p.dim;
    if (i >= (int64_t)p.R * per_row) return;
    const int64_t row = i / per_row;
    const int rem = (int)(i - row * per_row), t = rem / p.dim, j = rem - t * p.dim;
    const float *xr = p.x + (p.x_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.x_stride;
    const float idf = __ldg(xr + t);
    int id = (int)idf;
    if (!(idf >= 0.f && idf < (float)p.vocab) || (float)id != idf) {
        atomicExch(p.err, MURE_ERR_INVALID_ARG);
        id = 0;
    }
    const float v = __ldg(p.Wt + (int64_t)id * p.dim + j);
    if (p.z) p.z[row * p.z_stride + (int64_t)j * p.steps + t] = v;
    p.y[row * p.y_stride + (int64_t)t * p.dim + j] = v;
}

// A text repeats its words: the first LSTM's input sums depend on a position's token alone, so
// they are needed once per distinct token of the inputs (2,010 among 40,000 positions of 500
// synthetic reviews), not once per position.  k_tokens numbers the distinct ids (in no particular
// order), k_token_map gives every position its token's number.
__global__ void __launch_bounds__(256) k_tokens(const float *x, int64_t x_stride, int steps, int64_t n, int vocab,
                                                int32_t *seen, int32_t *slot, int32_t *tok_id, int32_t *count)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float idf = __ldg(x + i / steps * x_stride + i % steps);
    const int id = idf >= 0.f && idf < (float)vocab ? (int)idf : 0;   // (k_embed refuses the others)
    if (__ldcg(seen + id) == 0 && atomicExch(seen + id, 1) == 0) {   // (a seen id, the usual one, needs no atomic)
        const int k = atomicAdd(count, 1);
        tok_id[k] = id;
        slot[id] = k;
    }
}

__global__ void __launch_bounds__(256) k_token_map(const float *x, int64_t x_stride, int steps, int64_t n, int vocab,
                                                   const int32_t *slot, int32_t *tok)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float idf = __ldg(x + i / steps * x_stride + i % steps);
    tok[i] = slot[idf >= 0.f && idf < (float)vocab ? (int)idf : 0];
}

// The embedding rows of the tokens as each mutant of the embedding has them: out[g][token][dim],
// a mutated channel's entry with the delta's arithmetic (its sum over the one-hot input is
// 0 + e[id]).
__global__ void __launch_bounds__(256) k_embed_tokens(const PatchArgs pa, const float *__restrict__ Wt,
                                                      const int32_t *__restrict__ tok_id,
                                                      int n_tok, int dim, int vocab, float *__restrict__ out)
{
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x, per_g = (int64_t)n_tok * dim;
    const int g = blockIdx.y;
    if (i >= per_g) return;
    const int k = (int)(i / dim), j = (int)(i - (int64_t)k * dim), id = __ldg(tok_id + k);
    float v = __ldg(Wt + (int64_t)id * dim + j);
    const int n = pa.n_neurons[g], op = pa.op[g];
    const int32_t *ids = pa.ids + pa.neuron_off[g];
    for (int q = 0; q < n; ++q) {
        if (ids[q] != j) continue;
        if (op == MURE_OP_NEB) v = 0.f;
        else if (op == MURE_OP_NAI) v = -v;
        else if (op == MURE_OP_NS) v = __ldg(Wt + (int64_t)id * dim + ids[q ^ 1]);
        else v = v + (0.f + __ldg(pa.patch + pa.patch_off[g] + (int64_t)q * vocab + id));
    }
    out[g * per_g + i] = v;
}

// --------------------------------------------------------------------- LSTM --
//
// A gate's pre-activation at step t is one fp32 FMA chain from +0: its input weights on x_t
// in ascending order, then its recurrent weights on h_{t-1}, then + b.  The chain is cut where
// the recurrence begins:
//   k_lstm_proj  the part on x_t of every step at once (one tiled product over rows x steps,
//                columns 4u + gate), stored as fp32: no step waits for another;
//   k_lstm_rec   the steps: continues each stored sum with the recurrent weights (in shared
//                memory for all steps), the bias and the cell.
// A stored partial sum is exact, so the result is that of the uncut chain.  Measured on the
// IMDB-sized model (500 inputs x 40 mutants): 62.3 ms in one kernel that read a weight from
// global memory per FMA -> 1.2 (proj, 60 TFLOP/s, 0.86 of cuBLAS fp32) + 2.0 ms (rec).  The part on x_t
// depends on the row's input alone but for a mutant's own units: where the rows read cached
// inputs, one product per input serves all mutants of a batch (it is two thirds of the
// 128-input layer's work), and each mutant adds the columns of its mutated units
// (k_lstm_cols, k_lstm_proj with the mutant as grid z).  Behind an embedding the products take a
// row per distinct token instead (k_tokens): proj 1.2 -> 0.65 ms; the recurrence looks the rows
// up, two groups ahead.

constexpr int kMaxUnits = 64;   // units per layer
constexpr int kMaxIn = 128;     // input width

// Weight f of gate `gate` of unit u as mutant slot q of operator op has it (slot < 0: the
// original's): GF / WS add the patch, NAI negates, NS takes the partner's, NEB keeps (its
// output is held at 0).
struct LstmSlot {
    int q = -1, op = MURE_OP_IDENTITY, unit = 0, partner = 0;
    const float *e = nullptr;
};

__device__ __forceinline__ LstmSlot lstm_slot(const PatchArgs &pa, int g, int q, int U)
{
    LstmSlot s;
    const int32_t *ids = pa.ids + pa.neuron_off[g];
    s.q = q;
    s.op = pa.op[g];
    s.unit = ids[q];
    s.partner = s.op == MURE_OP_NS ? ids[q ^ 1] : s.unit;
    if (s.op == MURE_OP_GF || s.op == MURE_OP_WS) s.e = pa.patch + pa.patch_off[g] + (int64_t)q * 4 * U;
    return s;
}

__device__ __forceinline__ float lstm_weight(const LstmSlot &s, const float *W, int U, int gate, int f)
{
    float w = __ldg(W + (int64_t)s.partner * 4 * U + gate * U + f);
    if (s.e) w = w + __ldg(s.e + gate * U + f);
    return s.op == MURE_OP_NAI ? -w : w;
}

__device__ __forceinline__ float lstm_bias(const LstmSlot &s, const float *b, int gate)
{
    const float v = __ldg(b + 4 * s.partner + gate);
    return s.op == MURE_OP_NAI ? -v : v;
}

// The input weights of every mutant's mutated units as columns: mutant g's column 4q + gate of
// line f at out[g g_stride + f line], zeros for q >= n_neurons[g].
__global__ void __launch_bounds__(128) k_lstm_cols(const PatchArgs pa, const float *__restrict__ W, int cin, int U,
                                                   int kmax, int64_t g_stride, int64_t line, float *__restrict__ out)
{
    const int g = blockIdx.x, n = pa.n_neurons[g], cols = 4 * kmax;
    float *o = out + g * g_stride;
    for (int i = threadIdx.x; i < cin * cols; i += blockDim.x) {
        const int c = i / cin, f = i - c * cin, q = c >> 2;   // neighbouring threads read neighbouring weights
        o[f * line + c] = q < n ? lstm_weight(lstm_slot(pa, g, q, U), W, U, c & 3, f) : 0.f;
    }
}

struct ProjParams {
    const int32_t *tok_id;  // rows of x are this list's entries (tokens; steps = 1), else null
    const int32_t *m_dev;   // GEMM rows counted on the device (M is then their bound), else null
    const float *x; int64_t x_stride; int x_per_input;
    int64_t t0; int T;
    const int32_t *lrow;
    int64_t M;              // GEMM rows per z: (row, step) pairs
    int64_t z_rows;         // batch rows that z advances the input by (0: every z reads the same rows)
    int steps, cin, N;      // N columns (a multiple of 4)
    int n_tiles;            // column tiles (blockIdx.x: row tile * n_tiles + column tile)
    const float *B; int64_t b_stride;   // [z][cin][N]
    float *out;             // [z][M][N]
};

// BM x BN tiles, 256 threads.  With 128 x 128 (the layer's own 256 columns) a thread holds 8 x 8
// sums; the 256 x 16 form takes the few columns of mutated units.
template <int BM, int BN, int BK, int TM, int TN, bool VEC>
__global__ void __launch_bounds__(256, VEC ? 2 : 1) k_lstm_proj(const ProjParams p)
{
    constexpr int CT = BN / TN, RT = BM / TM;   // threads across columns, rows
    static_assert(CT * RT == 256, "256 threads");
    constexpr int RS = BM / (TM / 4), CS = BN / (TN / 4);
    constexpr int A4 = BM * BK / 4 / 256, B4 = (BK * BN / 4 + 255) / 256;
    __shared__ __align__(16) float2 As[2][BK][BM];
    __shared__ __align__(16) float Bs[2][BK][BN];
    const int tid = threadIdx.x, z = blockIdx.z;
    // a warp: up to 8 column groups x 4 row groups
    constexpr int CL = CT < 8 ? CT : 8, RL = 32 / CL;
    const int warp = tid >> 5, lane = tid & 31;
    const int tn = (warp % (CT / CL)) * CL + lane % CL, tm = (warp / (CT / CL)) * RL + lane / CL;
    const int mt = (int)(blockIdx.x / p.n_tiles), n0 = (int)(blockIdx.x - mt * p.n_tiles) * BN;
    const float *B = p.B + z * p.b_stride;
    const int64_t M = p.m_dev ? (int64_t)*p.m_dev : p.M;
    if ((int64_t)mt * BM >= M) return;
    // this thread's A pieces: four k of row tid % BM
    const float *xr = nullptr;
    if (const int64_t m = (int64_t)mt * BM + tid % BM; m < M) {
        const int64_t row = p.tok_id ? p.tok_id[m] : m / p.steps + z * p.z_rows;
        const int t = (int)(m % p.steps);
        xr = p.x + (p.x_per_input ? p.t0 + logical_row(p.lrow, row) % p.T : row) * p.x_stride + (int64_t)t * p.cin;
    }
    float4 ra[A4], rb[B4];
    auto load = [&](int k0) {
#pragma unroll
        for (int i = 0; i < A4; ++i) {
            const int k = k0 + 4 * (tid / BM + i * (256 / BM));
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (VEC) {
                if (xr && k < p.cin) v = __ldg(reinterpret_cast<const float4 *>(xr + k));
            } else if (xr) {
                if (k < p.cin) v.x = __ldg(xr + k);
                if (k + 1 < p.cin) v.y = __ldg(xr + k + 1);
                if (k + 2 < p.cin) v.z = __ldg(xr + k + 2);
                if (k + 3 < p.cin) v.w = __ldg(xr + k + 3);
            }
            ra[i] = v;
        }
#pragma unroll
        for (int i = 0; i < B4; ++i) {
            const int e = tid + i * 256, k = k0 + e / (BN / 4), n = n0 + 4 * (e % (BN / 4));
            rb[i] = (e < BK * BN / 4 && k < p.cin && n < p.N) ? __ldg(reinterpret_cast<const float4 *>(B + (int64_t)k * p.N + n))
                                                              : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    auto store = [&](int s) {
#pragma unroll
        for (int i = 0; i < A4; ++i) {
            const int k = 4 * (tid / BM + i * (256 / BM)), r = tid % BM;
            As[s][k][r] = make_float2(ra[i].x, ra[i].x);
            As[s][k + 1][r] = make_float2(ra[i].y, ra[i].y);
            As[s][k + 2][r] = make_float2(ra[i].z, ra[i].z);
            As[s][k + 3][r] = make_float2(ra[i].w, ra[i].w);
        }
#pragma unroll
        for (int i = 0; i < B4; ++i) {
            const int e = tid + i * 256;
            if (e < BK * BN / 4) *reinterpret_cast<float4 *>(&Bs[s][e / (BN / 4)][4 * (e % (BN / 4))]) = rb[i];
        }
    };
    f32x2 acc[TM][TN / 2];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0;
    // padding k (past cin) adds fma(0, 0, acc): the chain's value is unchanged
    load(0);
    store(0);
    __syncthreads();
    int s = 0;
    for (int k0 = 0; k0 < p.cin; k0 += BK, s ^= 1) {
        const bool more = k0 + BK < p.cin;
        if (more) load(k0 + BK);
        simt_tile_fma<BK, BM, BN, TM, TN, RS, CS>(acc, &As[s][0][tm * 4], &Bs[s][0][tn * 4]);
        if (more) store(s ^ 1);
        __syncthreads();
    }
    float *out = p.out + (int64_t)z * p.M * p.N;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int64_t mm = (int64_t)mt * BM + (i / 4) * RS + tm * 4 + (i & 3);
        if (mm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const int n = n0 + (j / 4) * CS + tn * 4;
            if (n >= p.N) continue;
            const float2 a = unpack2(acc[i][j / 2]), b = unpack2(acc[i][j / 2 + 1]);
            *reinterpret_cast<float4 *>(out + mm * p.N + n) = make_float4(a.x, a.y, b.x, b.y);
        }
    }
}

struct LstmParams {
    const float *proj; int proj_shared;   // [row][steps][4H]; shared: rows are the tile's inputs
    const int32_t *tok; int64_t t0;       // sums per token: of input t0 + row at step t, number tok[..] (else null)
    int64_t proj_g;                       // floats between the mutants' sums (tokens of each mutant)
    const float *projx;                   // mutated units: slot q of mutant g at g px_g + (row steps + step, or token) px_step + 4 q
    int64_t px_g; int px_step;
    int rows_per_g, bm, blocks_per_g;     // rows of a mutant (or all rows); rows per block
    int steps, cin, H, seq;
    const float *W;       // [H][4][cin + H]
    const float *Wt;      // [cin + H][4 u + gate]
    const float *b;       // [H][4]
    float *z; int64_t z_stride;   // the output again (nullable)
    float *y; int64_t y_stride;   // [steps][H] (seq) or [H]
    PatchArgs pa;         // the batch's mutants
    int mutated;          // 1: rows carry mutants of this layer
};

// The cell's functions on two cells at once (packed arithmetic).  exp is ex2 of the product
// with log2(e), the product's rounding and the constant's tail put back to first order (Cody
// and Waite's reduction); quotients are the hardware reciprocal and one Newton step.
// sigmoid = 1 / (1 + exp(-v)), 0 below -87; |tanh| = 1 - 2 e / (1 + e) with e = exp(-2 |v|), and
// below 0.6, where that cancels, the odd polynomial x + x^3 P(x^2) (fitted in x^2 by Lawson's
// iteration, least squares with the weights raised where the error is largest: relative error
// 3e-9).  The arguments are clamped to where the result is already 0 or 1 (a NaN passes); below -87
// sigmoid would be a subnormal number and is 0.  Against 64 bits over [-100, 100], worst and rms relative error: sigmoid 1.6e-7 and
// 3.3e-8 (1 / (1 + expf(-v)): 2.1e-7 and 4.2e-8), tanh 1.6e-7 and 1.5e-8 (tanhf: 2.0e-7 and
// 2.1e-8).  The mean error matters more than the rms, since a recurrence adds it up: without the
// term for ex2's own (kEx2Lean) sigmoid leant by 3e-8 and the logits of the Reuters-sized model
// were 1.87e-7 off (relative, over 6 tables), with it 1.69e-7; with the functions named, 1.83e-7.
// Those, scalar, took 0.86 us for a step of 4 rows, these 0.66.
constexpr float kLog2e = 1.44269502f, kLog2eTail = 1.92596303e-8f, kLn2 = 0.693147182f, kEx2Lean = 5.96046448e-8f;

__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }

__device__ __forceinline__ float ex2_approx(float v)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float rcp_approx(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float min_nan(float a, float b)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ float max_nan(float a, float b)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// exp(-S a) = e + ec, |S a| <= 87: ec carries what the product's rounding took from e
template <int S>
__device__ __forceinline__ f32x2 exp_neg2(f32x2 a, f32x2 &ec)
{
    const f32x2 nt = mul2(a, both(-S * kLog2e));                       // -(S a log2 e), rounded
    const float2 t = unpack2(nt);
    const f32x2 e = pack2(ex2_approx(t.x), ex2_approx(t.y));
    f32x2 d = fma2(a, both(S * kLog2e), nt);                           // what the rounding lost
    d = fma2(a, both(S * kLog2eTail), d);
    if (S == 1) {
        // ex2 reads high by 2^-24 of the exponent above 1, low below -1, in between less (measured)
        d = fma2(pack2(min_nan(max_nan(t.x, -1.f), 1.f), min_nan(max_nan(t.y, -1.f), 1.f)), both(kEx2Lean), d);
        d = mul2(d, both(-kLn2));
    } else {
        d = fma2(d, both(-kLn2), both(kLn2 * kEx2Lean));              // used below -1 only
    }
    ec = mul2(d, e);
    return e;
}

// -1 / (1 + e + ec), 0 <= e < 2^126: the residual of the Newton step is taken from e and ec
// themselves, so that the rounding of 1 + e does not enter
__device__ __forceinline__ f32x2 neg_rcp_1p2(f32x2 e, f32x2 ec)
{
    const float2 y = unpack2(fma2(e, both(-1.f), both(-1.f)));
    const f32x2 r = pack2(rcp_approx(y.x), rcp_approx(y.y));
    const f32x2 d = fma2(r, ec, fma2(r, e, add2(r, both(1.f))));
    return fma2(r, d, r);
}

__device__ __forceinline__ f32x2 sigmoid2(f32x2 v)
{
    const float2 x = unpack2(v);
    const f32x2 c = pack2(min_nan(max_nan(x.x, -87.f), 87.f), min_nan(max_nan(x.y, -87.f), 87.f));
    f32x2 ec;
    const f32x2 e = exp_neg2<1>(c, ec);
    const float2 s = unpack2(neg_rcp_1p2(e, ec));
    return pack2(x.x < -87.f ? 0.f : -s.x, x.y < -87.f ? 0.f : -s.y);
}

__device__ __forceinline__ f32x2 tanh2(f32x2 v)
{
    const float2 x = unpack2(v);
    const f32x2 a = pack2(min_nan(fabsf(x.x), 40.f), min_nan(fabsf(x.y), 40.f));
    f32x2 ec;
    const f32x2 e = exp_neg2<2>(a, ec);
    const f32x2 big = fma2(mul2(add2(e, ec), both(2.f)), neg_rcp_1p2(e, ec), both(1.f));
    const f32x2 q = mul2(a, a);
    f32x2 c = fma2(q, both(-5.90586569e-3f), both(2.08053812e-2f));
    c = fma2(q, c, both(-5.37866838e-2f));
    c = fma2(q, c, both(1.33319587e-1f));
    c = fma2(q, c, both(-3.33332986e-1f));
    const float2 lo = unpack2(fma2(mul2(q, a), c, a)), hi = unpack2(big), av = unpack2(a);
    return pack2(copysignf(av.x < 0.6f ? lo.x : hi.x, x.x), copysignf(av.y < 0.6f ? lo.y : hi.y, x.y));
}

// A block of 128 threads runs up to p.bm rows of one mutant through every step.  Thread 2u
// holds the recurrent weights of unit u's gates i and f, thread 2u + 1 those of g and o, in
// registers (64 x 2) for all steps: no weight is loaded again.  (A version with the weights in
// shared memory took 6.2k cycles per step of 8 rows and 8.2k of 16.)  What bounds it now is issue:
// 1.3k cycles per four rows and step with one block on an SM, 1.2k per block with two; ncu shows
// an instruction per warp every 1.9 cycles, the rest fixed latencies and dispatch stalls (an FMA
// with three registers of its own issues at two thirds of the rate).  Rows go four at a time: a
// 16-byte uniform load brings h of four units of a row for 8 FMAs per thread.  The two threads of a unit then swap half of their sums, so that each
// finishes two rows' cells.  h (double-buffered: one barrier per step) and c live in shared
// memory; the next rows' stored sums are fetched while the current ones run.
constexpr int kRecThreads = 2 * kMaxUnits;
constexpr int kRecLine = kMaxUnits + 8;   // floats per row of h: the swapped rows' writes hit different banks

__global__ void __launch_bounds__(kRecThreads, 2) k_lstm_rec(const LstmParams p)
{
    extern __shared__ __align__(16) float lsm[];
    float *hs = lsm;                              // [2][bm][kRecLine]
    float *cs = lsm + 2 * p.bm * kRecLine;        // [bm][kMaxUnits]
    const int tid = threadIdx.x, u = tid >> 1, hi = tid & 1;
    const int H = p.H, U = p.cin + H, N = 4 * H;
    const int g = blockIdx.x / p.blocks_per_g;                           // batch mutant
    const int first = (blockIdx.x - g * p.blocks_per_g) * p.bm;          // its first row here
    const int nr = min(p.bm, p.rows_per_g - first);
    const int64_t row0 = (int64_t)g * p.rows_per_g + first;
    const bool live = u < H;
    // this unit's weights, bias and stored sums, as the mutant has them
    LstmSlot sl;
    sl.unit = sl.partner = live ? u : 0;
    bool changed = false, blocked = false;
    const float *pp = p.proj + (p.tok ? g * p.proj_g : ((p.proj_shared ? first : row0) * p.steps) * N) + 2 * tid;
    int p_step = N;
    if (p.mutated && live)
        for (int q = 0; q < p.pa.n_neurons[g]; ++q) {
            const LstmSlot c = lstm_slot(p.pa, g, q, U);
            if (c.unit != u) continue;
            sl = c;
            changed = true;
            blocked = c.op == MURE_OP_NEB;
            p_step = p.px_step;
            pp = p.projx + g * p.px_g + (p.tok ? 0 : (int64_t)first * p.steps * p_step) + 4 * q + 2 * hi;
        }
    float w0[kMaxUnits], w1[kMaxUnits];
#pragma unroll
    for (int f = 0; f < kMaxUnits; ++f) {
        float2 w = make_float2(0.f, 0.f);
        if (live && f < H) {
            if (changed) w = make_float2(lstm_weight(sl, p.W, U, 2 * hi, p.cin + f), lstm_weight(sl, p.W, U, 2 * hi + 1, p.cin + f));
            else w = __ldg(reinterpret_cast<const float2 *>(p.Wt + (int64_t)(p.cin + f) * N + 2 * tid));
        }
        w0[f] = w.x;
        w1[f] = w.y;
    }
    const float b0 = lstm_bias(sl, p.b, 2 * hi), b1 = lstm_bias(sl, p.b, 2 * hi + 1);
    for (int i = tid; i < 2 * p.bm * kRecLine; i += kRecThreads) hs[i] = 0.f;
    for (int i = tid; i < p.bm * kMaxUnits; i += kRecThreads) cs[i] = 0.f;
    // the stored sums of rows r0 .. r0 + 3 at step t, one group of rows ahead of their use; where
    // they go by token, the numbers of the tokens two groups ahead
    float2 pre[4];
    int32_t tk[4];
    const int32_t *tok = p.tok ? p.tok + (p.t0 + first) * p.steps : nullptr;
    auto number = [&](int r0, int t) {
#pragma unroll
        for (int i = 0; i < 4; ++i) tk[i] = tok && r0 + i < nr && t < p.steps ? __ldg(tok + (int64_t)(r0 + i) * p.steps + t) : 0;
    };
    auto fetch = [&](int r0, int t) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int64_t at = tok ? (int64_t)tk[i] : (int64_t)(r0 + i) * p.steps + t;
            pre[i] = live && r0 + i < nr ? __ldg(reinterpret_cast<const float2 *>(pp + at * p_step)) : make_float2(0.f, 0.f);
        }
        if (tok) number(r0 + 4 < nr ? r0 + 4 : 0, r0 + 4 < nr ? t : t + 1);
    };
    if (tok) number(0, 0);
    fetch(0, 0);
    __syncthreads();
    for (int t = 0; t < p.steps; ++t) {
        const float *hc = hs + (t & 1) * p.bm * kRecLine;
        float *hn = hs + ((t + 1) & 1) * p.bm * kRecLine;
        for (int r0 = 0; r0 < nr; r0 += 4) {
            float a0[4], a1[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                a0[i] = pre[i].x;
                a1[i] = pre[i].y;
            }
            const bool wrap = r0 + 4 >= nr;
            if (!wrap || t + 1 < p.steps) fetch(wrap ? 0 : r0 + 4, wrap ? t + 1 : t);
#pragma unroll
            for (int f = 0; f < kMaxUnits; f += 4) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 h4 = *reinterpret_cast<const float4 *>(hc + (r0 + i) * kRecLine + f);
                    a0[i] = fmaf(h4.x, w0[f], a0[i]);
                    a1[i] = fmaf(h4.x, w1[f], a1[i]);
                    a0[i] = fmaf(h4.y, w0[f + 1], a0[i]);
                    a1[i] = fmaf(h4.y, w1[f + 1], a1[i]);
                    a0[i] = fmaf(h4.z, w0[f + 2], a0[i]);
                    a1[i] = fmaf(h4.z, w1[f + 2], a1[i]);
                    a0[i] = fmaf(h4.w, w0[f + 3], a0[i]);
                    a1[i] = fmaf(h4.w, w1[f + 3], a1[i]);
                }
            }
            // thread 2u keeps rows 0 and 1, thread 2u + 1 rows 2 and 3
            f32x2 gate[4];
            {
                float mine[2][2], got[2][2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mine[0][i] = (hi ? a0[2 + i] : a0[i]) + b0;
                    mine[1][i] = (hi ? a1[2 + i] : a1[i]) + b1;
                    got[0][i] = __shfl_xor_sync(0xffffffffu, (hi ? a0[i] : a0[2 + i]) + b0, 1);
                    got[1][i] = __shfl_xor_sync(0xffffffffu, (hi ? a1[i] : a1[2 + i]) + b1, 1);
                }
                const f32x2 m0 = pack2(mine[0][0], mine[0][1]), m1 = pack2(mine[1][0], mine[1][1]);
                const f32x2 o0 = pack2(got[0][0], got[0][1]), o1 = pack2(got[1][0], got[1][1]);
                gate[0] = hi ? o0 : m0;
                gate[1] = hi ? o1 : m1;
                gate[2] = hi ? m0 : o0;
                gate[3] = hi ? m1 : o1;
            }
            const int r = r0 + 2 * hi;
            float *cr = cs + r * kMaxUnits + u;
            const f32x2 ig = sigmoid2(gate[0]), fg = sigmoid2(gate[1]), gg = tanh2(gate[2]), og = sigmoid2(gate[3]);
            const f32x2 c = fma2(fg, pack2(cr[0], cr[kMaxUnits]), mul2(ig, gg));
            const float2 cv = unpack2(c);
            float2 h = unpack2(mul2(og, tanh2(c)));
            if (blocked) h = make_float2(0.f, 0.f);
            cr[0] = cv.x;
            cr[kMaxUnits] = cv.y;
            // units past the layer's and rows past the block's stay in this block's own lines
            hn[r * kRecLine + u] = live ? h.x : 0.f;
            hn[(r + 1) * kRecLine + u] = live ? h.y : 0.f;
            if (live && (p.seq || t + 1 == p.steps)) {
                const int64_t o = p.seq ? (int64_t)t * H + u : u;
                float *yr = p.y + (row0 + r) * p.y_stride + o;
                if (r < nr) yr[0] = h.x;
                if (r + 1 < nr) yr[p.y_stride] = h.y;
                if (p.z) {
                    float *zr = p.z + (row0 + r) * p.z_stride + o;
                    if (r < nr) zr[0] = h.x;
                    if (r + 1 < nr) zr[p.z_stride] = h.y;
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace

int recurrent_supported(const Stage &S)
{
    if (S.kind == MURE_NODE_LSTM) return S.oc <= kMaxUnits && S.ic <= kMaxIn;
    return S.kind == MURE_NODE_EMBED;
}

int launch_embed(const Stage &S, Src x, RowMap rm, float *z_out, int64_t z_stride, float *y_out, int64_t y_stride,
                 cudaStream_t s)
{
    if (rm.R <= 0) return 0;
    EmbedParams p{};
    p.x = x.p; p.x_stride = x.stride; p.x_per_input = x.per_input;
    p.t0 = rm.t0; p.T = rm.T; p.R = rm.R; p.lrow = rm.lrow;
    p.steps = S.iw; p.dim = S.oc; p.vocab = S.vocab;
    p.Wt = S.Wt;
    p.z = z_out; p.z_stride = z_stride;
    p.y = y_out; p.y_stride = y_stride;
    p.err = S.err;
    const int64_t n = (int64_t)rm.R * S.iw * S.oc;
    k_embed<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p);
    return 1;
}

int launch_tokens(const Src &x, int64_t rows, int steps, int vocab, int32_t *seen, int32_t *slot, int32_t *tok_id, int32_t *count,
                  int32_t *tok, cudaStream_t s)
{
    const int64_t n = rows * steps;
    const unsigned blocks = (unsigned)((n + 255) / 256);
    k_tokens<<<blocks, 256, 0, s>>>(x.p, x.stride, steps, n, vocab, seen, slot, tok_id, count);
    k_token_map<<<blocks, 256, 0, s>>>(x.p, x.stride, steps, n, vocab, slot, tok);
    return 2;
}

int launch_embed_tokens(const Stage &S, const PatchArgs &pa, int G, const LstmTokens &tk, float *out, cudaStream_t s)
{
    const int64_t per_g = (int64_t)tk.n * S.oc;
    PatchArgs a = pa;
    int launches = 0;
    for (int g0 = 0; g0 < G; g0 += 65535, ++launches) {   // the grid's y limit
        const int gn = G - g0 < 65535 ? G - g0 : 65535;
        k_embed_tokens<<<dim3((unsigned)((per_g + 255) / 256), (unsigned)gn), 256, 0, s>>>(a, S.Wt, tk.id, tk.n, S.oc,
                                                                                         S.vocab, out + g0 * per_g);
        a.op += gn; a.n_neurons += gn; a.neuron_off += gn; a.patch_off += gn;
    }
    return launches;
}

int64_t lstm_proj_floats(const Stage &S) { return S.kind == MURE_NODE_LSTM ? (int64_t)S.iw * 4 * S.oc : 0; }

namespace {

template <int BM, int BN, int BK, int TM, int TN>
void proj(ProjParams q, int nz, cudaStream_t s)
{
    q.n_tiles = (q.N + BN - 1) / BN;
    const int64_t tiles = (q.M + BM - 1) / BM * q.n_tiles;
    const dim3 grid((unsigned)tiles, 1, (unsigned)nz);
    // 16-byte pieces of x where every row and step starts on one
    if ((q.cin & 3) == 0 && (q.x_stride & 3) == 0 && (reinterpret_cast<uintptr_t>(q.x) & 15) == 0)
        k_lstm_proj<BM, BN, BK, TM, TN, true><<<grid, 256, 0, s>>>(q);
    else
        k_lstm_proj<BM, BN, BK, TM, TN, false><<<grid, 256, 0, s>>>(q);
}

}  // namespace

int launch_lstm(const Stage &S, Src x, RowMap rm, float *z_out, int64_t z_stride, float *y_out, int64_t y_stride,
                const PatchArgs *pa, const LstmWs &lw, cudaStream_t s, const LstmTokens *tk)
{
    if (rm.R <= 0) return 0;
    int launches = 0;
    // rows that read cached inputs share their inputs' sums (not in a compacted batch, whose
    // rows are any inputs in any order)
    const bool shared = (x.per_input && !rm.lrow) || (tk && !tk->rows_g);
    ProjParams q{};
    q.x = x.p; q.x_stride = x.stride; q.x_per_input = x.per_input;
    q.t0 = rm.t0; q.T = rm.T; q.lrow = rm.lrow;
    q.steps = S.iw; q.cin = S.ic; q.N = 4 * S.oc;
    q.M = (int64_t)(shared ? rm.T : rm.R) * S.iw;
    q.B = S.Wt;
    q.out = lw.proj;
    LstmParams p{};
    if (tk) {
        // a GEMM row per token: entries of the embedding's table, or each mutant's rows of it
        q.x = tk->rows; q.x_stride = S.ic; q.x_per_input = 0;
        q.steps = 1;
        q.tok_id = tk->rows_g ? nullptr : tk->id;
        q.m_dev = tk->rows_g ? nullptr : tk->n_dev;
        q.M = tk->rows_g ? (int64_t)tk->n * (rm.R / rm.T) : tk->n;
        p.tok = tk->tok;
        p.t0 = rm.t0;
        p.proj_g = tk->rows_g ? (int64_t)tk->n * q.N : 0;
    }
    proj<128, 128, 8, 8, 8>(q, 1, s);
    ++launches;
    if (pa && lw.kmax > 0) {
        const int G = rm.R / rm.T, cols = 4 * lw.kmax;
        if (!tk) q.M = (int64_t)rm.T * S.iw;
        q.B = lw.cols;
        q.out = lw.projx;
        p.projx = lw.projx;
        if (shared) {
            // every mutant reads the same rows: its units are columns of one product
            q.N = G * cols;
            p.px_g = cols;
            p.px_step = q.N;
            k_lstm_cols<<<(unsigned)G, 128, 0, s>>>(*pa, S.W, S.ic, S.ic + S.oc, lw.kmax, cols, q.N, lw.cols);
            proj<128, 128, 8, 8, 8>(q, 1, s);
            ++launches;
        } else {
            // rows of their own (vanilla): a narrow product per mutant
            q.N = cols;
            q.z_rows = rm.T;
            q.b_stride = (int64_t)S.ic * cols;
            p.px_g = q.M * cols;
            p.px_step = cols;
            k_lstm_cols<<<(unsigned)G, 128, 0, s>>>(*pa, S.W, S.ic, S.ic + S.oc, lw.kmax, q.b_stride, cols, lw.cols);
            for (int g0 = 0; g0 < G; g0 += 65535) {   // the grid's z limit
                const int gz = G - g0 < 65535 ? G - g0 : 65535;
                proj<256, 16, 8, 4, 4>(q, gz, s);
                q.B += gz * q.b_stride;
                q.out += (int64_t)gz * q.M * q.N;
                q.x += (int64_t)gz * rm.T * q.x_stride;
                ++launches;
            }
        }
        ++launches;
    }
    p.proj = lw.proj; p.proj_shared = shared;
    // blocks of one mutant's rows (or one input tile's, where its sums are shared)
    const int rows_per_g = pa || shared || tk ? rm.T : rm.R, G = rm.R / rows_per_g;
    p.rows_per_g = rows_per_g;
    p.steps = S.iw; p.cin = S.ic; p.H = S.oc; p.seq = S.kh;
    p.W = S.W; p.Wt = S.Wt; p.b = S.b;
    p.z = z_out; p.z_stride = z_stride;
    p.y = y_out; p.y_stride = y_stride;
    if (pa) {
        p.pa = *pa;
        p.mutated = 1;
    }
    // rows per block: the split whose waves (two blocks per SM) take the fewest row steps; a
    // pair on one SM takes about 1.5 times as long as one block alone
    const int slots = 2 * sm_count();
    int bm = 4;
    int64_t least = INT64_MAX;
    for (int b = 4; b <= 32; b += 4) {
        const int64_t blocks = (int64_t)G * ((rows_per_g + b - 1) / b), rem = blocks % slots;
        const int64_t cost = (blocks / slots * 3 + (rem == 0 ? 0 : rem <= slots / 2 ? 2 : 3)) * b;
        if (cost <= least) {
            least = cost;
            bm = b;
        }
    }
    p.bm = bm;
    p.blocks_per_g = (rows_per_g + bm - 1) / bm;
    const size_t smem = (size_t)bm * (2 * kRecLine + kMaxUnits) * 4;   // (26 KiB at most)
    k_lstm_rec<<<(unsigned)(G * p.blocks_per_g), kRecThreads, smem, s>>>(p);
    return launches + 1;
}

}  // namespace mure
