// wup.cu -- kernels of the paper's iterative w_up scheme (section
// "Sub-sampling algorithm"), its removal sweep restated as parallel rounds.
//
// An iteration recomputes every live point's S nearest neighbours and cost
// (a full search), takes w_up as the m-th smallest key (cost, index) and
// then removes points above w_up in rounds: a candidate (live, clean, key
// above w_up) goes when no adjacent candidate has a larger key, adjacency
// meaning that one of the two lies among the first k stored neighbours of
// the other.  Removed points leave their reverse neighbours' stored lists;
// a point with at least k stored points left takes its new cost from the
// first k of them, one with fewer is dirty until the next iteration (the
// paper's extended k+b neighbourhood and dirty flag).
//
//   wup_list_kernel    the iteration's candidates, listed; w_up itself
//   wup_beat_kernel    of two adjacent candidates the one of smaller key is
//                      marked as beaten
//   wup_pick_kernel    candidates that nothing beat are removed
//   wup_update_kernel  removed points leave the candidates' stored lists; new cost
//                      from the first k, or dirty; what is still a candidate is
//                      listed for the next round
//
// Keys only fall within an iteration and the next one searches every live point
// again, so a point below w_up at its start can neither become a candidate nor
// be read by one: a round touches the listed candidates alone, whose number
// falls from round to round, and all that the others need of a point is whether
// it still is a candidate (a byte).  With full passes over the cloud and two
// atomic maxima per neighbour a round was six launches over every point and a host
// read; now three launches over the list, four rounds a host read (wasted ones
// find an empty list).  What bounds a round is its three launches.
// 700k room points, k = 6, to 20 % (15 iterations, 224 rounds): 18.3 -> 9.5 ms, of which
// the rounds 14.1 -> 6.2 (7.8 ms with chained launches).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define FULLM 0xffffffffu

// The candidates: live points at or above the selection's boundary, which counts
// the keys that must go but is not a key itself.  w_up stays fixed while keys
// fall during an iteration, so it must be the key: the smallest one listed,
// found per block and, by the block that finishes last, over the blocks.
struct WupKey {
    u64 p;
    int i;
    __device__ __forceinline__ void least(u64 q, int j) {
        if (key_gt(p, i, q, j)) {
            p = q;
            i = j;
        }
    }
};
// The least key of a block of 256, in thread 0.
__device__ __forceinline__ WupKey wup_block_least(WupKey k) {
    __shared__ WupKey s_k[8];
    for (int o = 16; o; o >>= 1) {
        const u64 p = __shfl_xor_sync(FULLM, k.p, o);
        const int i = __shfl_xor_sync(FULLM, k.i, o);
        k.least(p, i);
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_k[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < 8; w++) k.least(s_k[w].p, s_k[w].i);
    return k;
}

__global__ void __launch_bounds__(256)
    wup_list_kernel(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n,
                    RoundDev* rd, uint8_t* cand, uint8_t* beaten, int* list, WupDev* wd,
                    WupKey* block_least) {
    chain();
    const u64 tp = rd->tau_prim;
    const int ti = rd->tau_idx;
    WupKey least = {~0ull, 0x7fffffff};
    for (int64_t b = blockIdx.x * (int64_t)256; b < n; b += (int64_t)gridDim.x * 256) {
        const int64_t s = b + threadIdx.x;
        bool in = false;
        if (s < n) {
            const u64 p = prim[s];
            in = alive[s] && p >= tp;
            if (in && (p == tp || p <= least.p)) {
                const int i = pos[s].w;
                in = !key_gt(tp, ti, p, i);
                if (in) least.least(p, i);
            }
            cand[s] = in;
            if (in) beaten[s] = 0;
        }
        const int slot = block_append(in, &wd->count[0]);
        if (in) list[slot] = (int)s;
    }
    least = wup_block_least(least);
    __shared__ bool s_last;
    if (threadIdx.x == 0) {
        block_least[blockIdx.x] = least;
        __threadfence();
        s_last = atomicAdd(&wd->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    least.p = ~0ull;
    least.i = 0x7fffffff;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += 256)
        least.least(__ldcg(&block_least[b].p), __ldcg(&block_least[b].i));
    least = wup_block_least(least);
    if (threadIdx.x == 0) {
        rd->tau_prim = least.p;
        rd->tau_idx = least.i;
    }
}

__global__ void __launch_bounds__(256)
    wup_beat_kernel(const BufView b, const uint8_t* cand, const int* list, int in, int slot,
                    int k, WupDev* wd, uint8_t* beaten) {
    chain();
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // for the launches of this round
        wd->count[in ^ 1] = 0;
        wd->removed[slot] = 0;
    }
    const int n = wd->count[in];
    for (int t = blockIdx.x * 256 + threadIdx.x; t < n; t += gridDim.x * 256) {
        const int s = list[t];
        int x[8];
        load_nbr8(b.nbr, s, x);
        const u64 ps = b.prim[s];
        bool c[8];
#pragma unroll
        for (int i = 0; i < 8; i++) c[i] = i < k && x[i] >= 0 && cand[x[i]];
        bool lost = false;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (!c[i]) continue;
            const u64 px = b.prim[x[i]];
            const bool loses =
                px != ps ? px > ps : key_gt(px, b.pos[x[i]].w, ps, b.pos[s].w);
            if (loses) lost = true;
            else beaten[x[i]] = 1;
        }
        if (lost) beaten[s] = 1;
    }
}

__global__ void __launch_bounds__(256)
    wup_pick_kernel(const int* list, int in, int slot, WupDev* wd, uint8_t* cand, uint8_t* beaten,
                    uint8_t* alive) {
    chain();
    const int n = wd->count[in];
    unsigned long long c = 0;
    for (int t = blockIdx.x * 256 + threadIdx.x; t < n; t += gridDim.x * 256) {
        const int s = list[t];
        if (beaten[s]) {
            beaten[s] = 0;
        } else {
            alive[s] = 0;
            cand[s] = 0;
            c++;
        }
    }
    block_add(&wd->removed[slot], c);
}

// Removed points leave the stored lists (order kept); the cost is the sum of
// 1 / d^2 over the first k stored points left, nearest first, in binary64.
__global__ void __launch_bounds__(256)
    wup_update_kernel(BufView b, const uint8_t* alive, const int* list, int* next, int in, int k,
                      const RoundDev* rd, uint8_t* cand, WupDev* wd) {
    chain();
    const int n = wd->count[in];
    const u64 tp = rd->tau_prim;
    const int ti = rd->tau_idx;
    for (int t0 = blockIdx.x * 256; t0 < n; t0 += gridDim.x * 256) {  // uniform over the block
        const int t = t0 + threadIdx.x;
        bool stays = false;
        int s = 0;
        if (t < n) {
            s = list[t];
            stays = alive[s];
        }
        if (stays) {
            int ids[8];
            load_nbr8(b.nbr, s, ids);
            bool dead = false;
#pragma unroll
            for (int i = 0; i < 8; i++) dead |= !alive[ids[i] >= 0 ? ids[i] : s];
            if (dead) {
                const int r = keep_live8(alive, ids);
                stays = r >= k;
                if (stays) {
                    store_nbr8(b.nbr, s, ids);
                    const int4 ps = b.pos[s];
                    u64 d[8];
#pragma unroll
                    for (int i = 0; i < 8; i++) d[i] = i < k ? sqd(ps, b.pos[ids[i]]) : 0;
                    double c = 0.0;
#pragma unroll
                    for (int i = 0; i < 8; i++)
                        if (i < k) c = __dadd_rn(c, __ddiv_rn(1.0, (double)d[i]));
                    const u64 p = key_prim_cost(c);
                    b.prim[s] = p;
                    stays = !key_gt(tp, ti, p, ps.w);
                }
                if (!stays) cand[s] = 0;
            }
        }
        const int slot = block_append(stays, &wd->count[in ^ 1]);
        if (stays) next[slot] = s;
    }
}

// The candidates of an iteration and w_up: tau takes the smallest live key at or
// above the selection's boundary.
cudaError_t wup_launch_list(const BufView& b, const uint8_t* alive, int64_t n, RoundDev* rd,
                            const WupBuffers& w, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(w.wd, 0, sizeof(WupDev), st);
    if (e) return e;
    int64_t blocks = (n + 255) / 256;
    if (blocks > wup_blocks()) blocks = wup_blocks();
    launch_chained(wup_list_kernel, (unsigned)blocks, 256, 0, st, b.prim, b.pos, alive, n, rd,
                   w.cand, w.beaten, w.list[0], w.wd, (WupKey*)w.block_least);
    note_launch();
    return cudaGetLastError();
}

int64_t wup_blocks() { return (int64_t)device_sms() * 8; }
size_t wup_least_bytes() { return (size_t)wup_blocks() * sizeof(WupKey); }

// WUP_BATCH removal rounds on the candidates in list[in], at most `most` of
// them; wd->removed[j]: the points round j removed.  An even number of rounds:
// the candidates left are in list[in] again.
cudaError_t wup_launch_rounds(const BufView& b, uint8_t* alive, int64_t most, int S, int k,
                              const RoundDev* rd, const WupBuffers& w, cudaStream_t st) {
    static_assert(WUP_BATCH % 2 == 0, "the lists change places every round");
    if (S != 8 || k > S || most <= 0) return cudaErrorInvalidValue;
    const unsigned g = list_blocks(most, 256, 8);
    for (int j = 0; j < WUP_BATCH; j++) {
        const int in = j & 1;
        launch_chained(wup_beat_kernel, g, 256, 0, st, b, w.cand, w.list[in], in, j, k, w.wd,
                       w.beaten);
        launch_chained(wup_pick_kernel, g, 256, 0, st, w.list[in], in, j, w.wd, w.cand, w.beaten,
                       alive);
        launch_chained(wup_update_kernel, g, 256, 0, st, b, alive, w.list[in], w.list[in ^ 1], in,
                       k, rd, w.cand, w.wd);
        for (int i = 0; i < 3; i++) note_launch();
    }
    return cudaGetLastError();
}

}  // namespace pd
