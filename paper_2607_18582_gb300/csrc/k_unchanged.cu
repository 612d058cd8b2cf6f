// Exact unchanged-row elimination (memoized mode; beyond the paper, sound by the
// argument of its soundness theorem).  A single-layer mutant changes only the
// channels of layer l it lists, so row r's suffix (layers l+1 .. L-1) is a function of
// its x_{l+1} alone, the tensor the first suffix stage reads: where every mutated
// channel of the row's patch equals the cached original x_{l+1} of its input bit for
// bit, the suffix reproduces the original forward pass (the kernels are deterministic
// and batch-invariant), so the row's prediction is the original's, its kill bit is 0
// and its logits are the cached original logits.  Such rows are dropped before the
// suffix; the others are listed in ascending order for a compacted batch.
#include "common.cuh"
#include "device_util.cuh"

namespace mure {

namespace {

constexpr int kGroup = 32;   // rows per block of the flags kernel and per entry of the counts

// One warp per row (4 rows per warp in turn): flags[r] = 1 for a row to run, 0 for an
// unchanged row or a padding input; group_cnt[b] = the rows to run of block b.  Most rows
// differ within the first cells, so the comparison stops at the first chunk that does; a chunk
// keeps four loads of each side in flight per lane.  Few rows per block, since a batch has
// only thousands of them (256 per block and whole channels compared: 183 us for 2,000 rows of
// a 32 x 32 map, now 10).
__global__ void __launch_bounds__(256) k_unchanged_flags(const UnchangedArgs ua, int64_t t0, int T, int R,
                                                         int32_t *flags, int32_t *group_cnt)
{
    __shared__ int cnt;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) cnt = 0;
    __syncthreads();
    int mine = 0;
    for (int i = 0; i < kGroup / 8; ++i) {
        const int64_t r = (int64_t)blockIdx.x * kGroup + warp * (kGroup / 8) + i;
        if (r >= R) break;
        const int g = (int)(r / T);
        const int64_t t = t0 + r % T;
        int run = 0;
        if (t < ua.fa.n_in) {
            const int k = ua.n_neurons[g];
            const int32_t *ids = ua.ids + ua.neuron_off[g];
            const float *prow = ua.patch + r * ua.row_stride;
            const float *orig = ua.base + t * ua.base_stride;
            bool same = true;
            for (int q = 0; q < k && same; ++q) {
                const int j = ids[q];
                for (int c0 = 0; c0 < ua.cells && same; c0 += 128) {
                    bool eq = true;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int c = c0 + 32 * u + lane;
                        if (c < ua.cells)
                            eq &= __float_as_uint(__ldg(prow + (int64_t)q * ua.cells + c)) ==
                                  __float_as_uint(__ldg(orig + (int64_t)c * ua.ch + j));
                    }
                    same = __all_sync(0xffffffffu, eq);
                }
            }
            run = same ? 0 : 1;
            if (same) {
                // the original logits stand for the row's
                const float *lg = ua.logits + t * ua.logits_stride;
                const int mid = ua.fa.mutant_id[g];
                if (ua.fa.logits_out)
                    for (int c = lane; c < ua.C; c += 32) ua.fa.logits_out[((int64_t)mid * ua.fa.n_in + t) * ua.C + c] = lg[c];
                if (lane == 0 && ua.fa.near_ties) {
                    float v[kMaxClasses];
                    for (int c = 0; c < ua.C; ++c) v[c] = lg[c];
                    const int arg = argmax_first(v, ua.C);
                    if (near_tie(v, ua.C, arg)) atomicAdd(ua.fa.near_ties, 1ull);
                }
            }
        }
        if (lane == 0) flags[r] = run;
        mine += run;
    }
    if (lane == 0 && mine) atomicAdd(&cnt, mine);
    __syncthreads();
    if (threadIdx.x == 0) group_cnt[blockIdx.x] = cnt;
}

// Exclusive scan of the group counts (one block); count = their sum.
__global__ void __launch_bounds__(1024) k_unchanged_scan(int32_t *group_cnt, int ng, int32_t *count)
{
    __shared__ int32_t part[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto warp_scan = [&](int32_t v) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t n = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += n;
        }
        return v;
    };
    int32_t carry = 0;
    for (int base = 0; base < ng; base += 1024) {
        const int i = base + threadIdx.x;
        const int32_t v = i < ng ? group_cnt[i] : 0;
        const int32_t incl = warp_scan(v);
        if (lane == 31) part[warp] = incl;
        __syncthreads();
        if (warp == 0) part[lane] = warp_scan(part[lane]);
        __syncthreads();
        if (i < ng) group_cnt[i] = carry + (warp > 0 ? part[warp - 1] : 0) + incl - v;
        carry += part[31];
        __syncthreads();
    }
    if (threadIdx.x == 0) *count = carry;
}

// lrow[offset of r's group + rank of r among the group's rows to run] = r; a warp per group.
__global__ void __launch_bounds__(256) k_unchanged_compact(const int32_t *flags, const int32_t *group_off, int R,
                                                           int32_t *lrow)
{
    const int lane = threadIdx.x & 31;
    const int64_t grp = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5), r = grp * kGroup + lane;
    const int f = r < R ? flags[r] : 0;
    const unsigned b = __ballot_sync(0xffffffffu, f);
    if (f) lrow[group_off[grp] + __popc(b & ((1u << lane) - 1u))] = (int32_t)r;
}

}  // namespace

int launch_unchanged(const UnchangedArgs &ua, RowMap rm, int32_t *flags, int32_t *group_cnt, int32_t *lrow,
                     int32_t *count, cudaStream_t s)
{
    const int ng = (rm.R + kGroup - 1) / kGroup;
    k_unchanged_flags<<<ng, 256, 0, s>>>(ua, rm.t0, rm.T, rm.R, flags, group_cnt);
    k_unchanged_scan<<<1, 1024, 0, s>>>(group_cnt, ng, count);
    k_unchanged_compact<<<(ng + 7) / 8, 256, 0, s>>>(flags, group_cnt, rm.R, lrow);
    return 3;
}

}  // namespace mure
