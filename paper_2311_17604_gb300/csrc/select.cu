// select.cu -- the removal threshold of a round (rule R2): the rank-th largest
// live key, on the device, for one cloud or for every scan of a packed batch.
//
// Keys are 96 bits, (prim << 32 | input index).  Two full passes take the two
// leading 12-bit digits (sign and exponent, then 12 mantissa bits): each counts
// its digit in a shared histogram per block, and the block that finishes last
// finds the digit's bin.  A third pass lists the keys that agree with both
// digits, a thousandth of the points or so, and one cluster of 8 blocks (of eight
// scans where a batch holds many) settles the remaining digits over that list.  The
// leading digit alone would keep a whole power of two of keys, so listing after it
// moved most of the points once more per round: a radix select with a histogram, a
// find and a compaction launch per digit took 23 launches.  Measured, selection of all rounds of one decimation: 9.8M outdoor
// points, k = 4 (287 rounds) 35.4 -> 17 ms; 3.8M points in a packed batch of 12 (612
// rounds) 135 -> 28.5 ms; 200k room points, k = 1 (19 rounds) 1.30 -> 0.38 ms.
//
// Any threshold between the rank-th largest key and the next smaller one has
// the same effect: the lower boundary of a bin serves when the bin ends on the
// rank.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

namespace cg = cooperative_groups;

#define SEL_T 512          // threads per block
#define SEL_CLUSTER 8      // blocks of the cluster that settles a list
// Scans of a batch up to which each has a cluster of its own.  Above, eight share one:
// a launch of mostly idle blocks costs more than long lists one after the other (400
// small scans 7.66 ms with a cluster each, 7.50; 1000 13.7, 13.3; 100 9.14, 9.18; 70
// voxelised scans, long lists all, 57.7 and 61.0).
#define SEL_CLUSTER_MAX 256

struct SelBin {
    int bin;                      // -1: the rank is beyond the count
    unsigned long long cum, cnt;  // keys above the bin, keys in it
    unsigned long long total;
};

// The bin of a 4096-bin histogram that holds rank r counted from the top
// (row(bin): its count); every thread of a block of SEL_T calls it.
template <class Row>
__device__ SelBin sel_bin(Row row, long long r) {
    __shared__ unsigned long long s_w[SEL_T / 32];
    __shared__ SelBin s_b;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int per = 4096 / SEL_T;  // thread t owns bins [4095 - per t - per + 1, 4095 - per t]
    uint32_t c[per];
    unsigned long long s = 0;
#pragma unroll
    for (int j = 0; j < per; j++) {
        c[j] = row(4095 - per * t - j);
        s += c[j];
    }
    unsigned long long inc = s;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
    }
    __syncthreads();  // a previous call's readers are done
    if (lane == 31) s_w[w] = inc;
    if (t == 0) s_b.bin = -1;
    __syncthreads();
    unsigned long long before = inc - s, total = 0;
    for (int i = 0; i < SEL_T / 32; i++) {
        if (i < w) before += s_w[i];
        total += s_w[i];
    }
    if ((long long)before < r && (long long)(before + s) >= r) {
        unsigned long long cum = before;
#pragma unroll
        for (int j = 0; j < per; j++) {
            if ((long long)(cum + c[j]) >= r) {
                s_b.bin = 4095 - per * t - j;
                s_b.cum = cum;
                s_b.cnt = c[j];
                break;
            }
            cum += c[j];
        }
    }
    if (t == 0) s_b.total = total;
    __syncthreads();
    return s_b;
}

// The selection state of a cloud (RoundDev) or a scan (SegDev) takes the bin
// found in digit `pass`; one thread calls it.
template <class State>
__device__ void sel_take(State& S, const SelBin& f, long long r, int pass, RoundDev* rd) {
    S.pre[pass] = (unsigned)f.bin;
    S.rank = r - (long long)f.cum;
    if ((long long)(f.cum + f.cnt) == r || pass == 7) {
        unsigned __int128 v = 0;
        for (int p = 0; p < 8; p++) {
            v <<= 12;
            if (p <= pass) v |= S.pre[p];
        }
        S.tau_prim = (unsigned long long)(v >> 32);
        S.tau_idx = (int)(uint32_t)v;
        S.done = 1;
        // packed batch: the least threshold over the scans (a prefilter)
        if (rd->seg) atomicMin(&rd->tau_prim, S.tau_prim);
    }
}

// What a round examines: everything above the target (k = 1), or a band of
// the largest keys.
__device__ inline long long sel_rank(const RoundDev* rd, long long live, long long need) {
    if (rd->density_k1) return need;
    const long long band = (long long)(rd->band * (double)live);
    // with weights a quarter of what must go at most: their rounds are not
    // provably the sequential order, and narrower ones stay closer to it
    const long long most = rd->density ? need : (need + 3) / 4;
    const long long rank = band < most ? band : most;
    return rank < 1 ? 1 : rank;
}

// True in every thread of the block that is the last of n to arrive.
__device__ inline bool last_block(unsigned* ticket, unsigned n) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(ticket, 1u) == n - 1;
        if (s_last) *ticket = 0;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// The positions of work item w: a block of one cloud's grid-stride, or a chunk
// of one scan.
struct SelItem {
    int seg;
    long long lo, hi;
    unsigned items;  // of this scan
};
__device__ inline SelItem sel_item(const RoundDev* rd, const SegDev* seg, const int* items, int w) {
    SelItem it;
    it.seg = items[w];
    const SegDev& s = seg[it.seg];
    const int c0 = rd->seg_chunk0[it.seg];
    it.lo = s.b + (long long)(w - c0) * PD_SEG_CHUNK;
    it.hi = it.lo + PD_SEG_CHUNK < s.e ? it.lo + PD_SEG_CHUNK : s.e;
    it.items = (unsigned)(rd->seg_chunk0[it.seg + 1] - c0);
    return it;
}

// Counts digit PASS (0, 1) of the live keys in [lo, hi) step `stride` blocks,
// four loads in flight per thread.
template <int PASS>
__device__ __forceinline__ void sel_count(const u64* __restrict__ prim,
                                          const uint8_t* __restrict__ alive, long long lo,
                                          long long hi, long long stride, uint32_t pre0,
                                          uint32_t* h) {
    for (long long i0 = lo + threadIdx.x; i0 < hi; i0 += stride) {
        u64 p[4];
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const long long i = i0 + j * SEL_T;
            in[j] = i < hi && alive[i];
            p[j] = i < hi ? prim[i] : 0;
        }
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const uint32_t d0 = (uint32_t)(p[j] >> 52);
            if (PASS == 0) {
                if (in[j]) atomicAdd(&h[d0], 1u);
            } else if (in[j] && d0 == pre0) {
                atomicAdd(&h[(uint32_t)(p[j] >> 40) & 0xfffu], 1u);
            }
        }
    }
}

// One full pass.  hist: 4096 words per cloud or scan, zero on entry and exit.
template <int PASS, bool SEG>
__global__ void __launch_bounds__(SEL_T)
    sel_pass_kernel(const u64* prim, const uint8_t* alive, int64_t n, uint32_t* hist,
                    RoundDev* rd, SegDev* seg, const int* items) {
    chain();
    __shared__ uint32_t h[4096];
    if (PASS == 0 && blockIdx.x == 0 && threadIdx.x == 0) {  // the round's counters
        rd->ncand = rd->nslow = rd->nsrc = rd->npairs = rd->ndep = 0;
        rd->nreq = rd->nfq = rd->nlq = 0;
        rd->take_src = rd->take_filt = rd->take_req = 0;
        rd->overflow = 0;
        rd->removed = 0;
        rd->cap_over = 0;
        rd->fix_unconverged = 0;
        rd->finished = 0;
        for (int i = 0; i < PD_FIX_ITERS; i++) rd->changed[i] = 0;
    }
    const int nitems = SEG ? rd->seg_chunk0[rd->nseg] : (int)gridDim.x;
    for (int w = blockIdx.x; w < nitems; w += gridDim.x) {  // one cloud: once
        SelItem it;
        it.seg = 0;
        uint32_t pre0 = 0;
        if (SEG) {
            it = sel_item(rd, seg, items, w);
            if (PASS > 0 && seg[it.seg].done) continue;
            if (PASS > 0) pre0 = seg[it.seg].pre[0];
        } else {
            if (PASS > 0 && rd->done) return;
            if (PASS > 0) pre0 = rd->pre[0];
        }
        for (int x = threadIdx.x; x < 4096; x += SEL_T) h[x] = 0;
        __syncthreads();
        if (SEG) sel_count<PASS>(prim, alive, it.lo, it.hi, 4 * SEL_T, pre0, h);
        else
            sel_count<PASS>(prim, alive, (long long)w * 4 * SEL_T, n,
                            (long long)gridDim.x * 4 * SEL_T, pre0, h);
        __syncthreads();
        uint32_t* row = hist + (size_t)it.seg * 4096;
        for (int x = threadIdx.x; x < 4096; x += SEL_T)
            if (h[x]) atomicAdd(&row[x], h[x]);
        SegDev* S = SEG ? &seg[it.seg] : nullptr;
        if (!last_block(SEG ? &S->ticket : &rd->ticket, SEG ? it.items : gridDim.x)) continue;
        // the last block of the cloud or scan: find the bin, clear the row
        auto get = [&](int b) { return __ldcg(row + b); };
        long long r, need = 0;
        SelBin f;
        if (PASS == 0 && SEG) {
            f = sel_bin(get, 1);  // for the live count
            need = (long long)f.total - S->m;
            r = rd->seg_rank_one ? 1 : sel_rank(rd, (long long)f.total, need);
            if (need > 0) f = sel_bin(get, r);
            if (threadIdx.x == 0) {
                S->live = (long long)f.total;
                S->need = need;
                S->done = 0;
                S->len = 0;
            }
        } else if (PASS == 0) {
            need = rd->live - rd->m;
            r = sel_rank(rd, rd->live, need);
            f = sel_bin(get, r);
            if (threadIdx.x == 0) {
                rd->need = need;
                rd->done = 0;
                rd->len = 0;
            }
        } else {
            r = SEG ? S->rank : rd->rank;
            f = sel_bin(get, r);
        }
        if (threadIdx.x == 0) {
            if (SEG) {
                if (PASS == 0 && need <= 0) {  // target reached: nothing of this scan goes
                    S->rank = 0;
                    S->done = 1;
                    S->tau_prim = ~0ull;
                    S->tau_idx = 0x7fffffff;
                } else if (f.bin < 0) {  // rank beyond the live count: cannot happen
                    S->done = 1;
                    S->tau_prim = ~0ull;
                    S->tau_idx = 0x7fffffff;
                    rd->overflow = 1;
                } else {
                    sel_take(*S, f, r, PASS, rd);
                }
            } else if (f.bin < 0) {
                rd->done = 1;
                rd->overflow = 1;
            } else {
                sel_take(*rd, f, r, PASS, rd);
            }
        }
        __syncthreads();
        for (int x = threadIdx.x; x < 4096; x += SEL_T) row[x] = 0;
        __syncthreads();
    }
}

// Lists the live keys that agree with both leading digits.
template <bool SEG>
__global__ void __launch_bounds__(SEL_T)
    sel_list_kernel(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n, u64* lp,
                    int* li, RoundDev* rd, SegDev* seg, const int* items) {
    chain();
    __shared__ int s_w[SEL_T / 32], s_at;
    const int nitems = SEG ? rd->seg_chunk0[rd->nseg] : (int)gridDim.x;
    for (int w = blockIdx.x; w < nitems; w += gridDim.x) {
        long long lo, hi, stride, base = 0;
        uint32_t want;
        int* count;
        if (SEG) {
            const SelItem it = sel_item(rd, seg, items, w);
            SegDev& S = seg[it.seg];
            if (S.done) continue;
            lo = it.lo;
            hi = it.hi;
            stride = 4 * SEL_T;
            base = S.b;
            want = (S.pre[0] << 12) | S.pre[1];
            count = &S.len;
        } else {
            if (rd->done) break;
            lo = (long long)w * 4 * SEL_T;
            hi = n;
            stride = (long long)gridDim.x * 4 * SEL_T;
            want = (rd->pre[0] << 12) | rd->pre[1];
            count = &rd->len;
        }
        for (long long i0 = lo + threadIdx.x; i0 - threadIdx.x < hi; i0 += stride) {
            u64 p[4];
            bool take[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const long long i = i0 + j * SEL_T;
                p[j] = i < hi ? prim[i] : 0;
                take[j] = i < hi && (uint32_t)(p[j] >> 40) == want && alive[i];
            }
            // one atomic per block and step: same-address atomics serialise in L2
            unsigned m[4];
            int mine = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                m[j] = __ballot_sync(0xffffffffu, take[j]);
                mine += __popc(m[j]);
            }
            if (!__syncthreads_or(mine)) continue;
            const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
            if (lane == 0) s_w[wp] = mine;
            __syncthreads();
            if (threadIdx.x == 0) {
                int acc = 0;
                for (int k = 0; k < SEL_T / 32; k++) {
                    const int c = s_w[k];
                    s_w[k] = acc;
                    acc += c;
                }
                s_at = atomicAdd(count, acc);
            }
            __syncthreads();
            int at = s_at + s_w[wp];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (take[j]) {
                    const long long o = base + at + __popc(m[j] & ((1u << lane) - 1u));
                    lp[o] = p[j];
                    li[o] = pos[i0 + j * SEL_T].w;
                }
                at += __popc(m[j]);
            }
        }
    }
}

// A remaining digit over a long list (many equal keys, as a voxelised cloud
// has): the whole grid counts, the last block finds.
__global__ void __launch_bounds__(SEL_T)
    sel_digit_kernel(const u64* lp, const int* li, int pass, uint32_t* hist, RoundDev* rd) {
    chain();
    __shared__ uint32_t h[4096];
    if (rd->done) return;
    for (int x = threadIdx.x; x < 4096; x += SEL_T) h[x] = 0;
    __syncthreads();
    const long long len = rd->len;
    uint32_t pre[8];
    for (int q = 2; q < pass; q++) pre[q] = rd->pre[q];
    for (long long j = blockIdx.x * (long long)SEL_T + threadIdx.x; j < len;
         j += (long long)gridDim.x * SEL_T) {
        const u64 p = lp[j];
        const int id = li[j];
        bool ok = true;
        for (int q = 2; q < pass; q++) ok = ok && key_digit(p, id, q) == pre[q];
        if (ok) atomicAdd(&h[key_digit(p, id, pass)], 1u);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < 4096; x += SEL_T)
        if (h[x]) atomicAdd(&hist[x], h[x]);
    if (!last_block(&rd->ticket, gridDim.x)) return;
    const long long r = rd->rank;
    const SelBin f = sel_bin([&](int b) { return __ldcg(hist + b); }, r);
    if (threadIdx.x == 0) {
        if (f.bin < 0) {
            rd->done = 1;
            rd->overflow = 1;
        } else {
            sel_take(*rd, f, r, pass, rd);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < 4096; x += SEL_T) hist[x] = 0;
}

// The remaining digits over the lists of `per` scans (a cloud's own list: 1) per
// cluster.  Up to SEL_SMEM keys (the usual case) one block takes them into shared
// memory and steps over the digits that all of them share (equal keys: the whole of
// prim); a cluster's blocks take a scan each.  A longer list is shared by the blocks
// of the cluster, which add their counts into block 0's histogram, one such list of
// the cluster after the other: with one block per scan a gridded scan's list was one
// multiprocessor's work (a lattice of 8.0M points packed with 64 scans of 5k, k = 1:
// 71.7 -> 22.9 ms; of 1.0M 10.2 -> 5.8).
#define SEL_SMEM 2048

struct SelList {
    int i;  // the scan
    long long base, len, r;
    bool done;
};
template <bool SEG>
__device__ __forceinline__ SelList sel_list(const RoundDev* rd, const SegDev* seg, int i) {
    SelList l;
    l.i = i;
    l.done = SEG ? seg[i].done : rd->done;
    l.base = SEG ? seg[i].b : 0;
    l.len = SEG ? seg[i].len : rd->len;
    l.r = SEG ? seg[i].rank : rd->rank;
    return l;
}
// One thread: the bin found in digit `pass` of list l, rank r of what is left.
template <bool SEG>
__device__ __forceinline__ void sel_settle(RoundDev* rd, SegDev* seg, int i, const SelBin& f,
                                           long long r, int pass) {
    if (f.bin < 0) {
        rd->overflow = 1;  // cannot happen; settled on the host
        if (SEG) seg[i].done = 1;
        else rd->done = 1;
    } else if (SEG) {
        sel_take(seg[i], f, r, pass, rd);
    } else {
        sel_take(*rd, f, r, pass, rd);
    }
}

template <bool SEG>
__global__ void __launch_bounds__(SEL_T)
    sel_rest_kernel(const u64* lp, const int* li, RoundDev* rd, SegDev* seg, int nseg, int per) {
    chain();
    __shared__ uint32_t h[4096];
    __shared__ u64 sp[SEL_SMEM];
    __shared__ int si[SEL_SMEM];
    __shared__ u64 s_dp;
    __shared__ uint32_t s_di;
    __shared__ SelBin s_f;
    cg::cluster_group cl = cg::this_cluster();
    const int nb = (int)cl.num_blocks(), br = (int)cl.block_rank();
    const int i0 = (int)(blockIdx.x / nb) * per;  // the cluster's first scan
    uint32_t pre[8];
    // a short list: this block's own
    if (br < per && i0 + br < nseg) {
        const SelList l = sel_list<SEG>(rd, seg, i0 + br);
        if (!l.done && l.len <= SEL_SMEM) {
            if (threadIdx.x == 0) {
                s_dp = 0;
                s_di = 0;
            }
            __syncthreads();
            const u64 p0 = lp[l.base];
            const int x0 = li[l.base];
            const int len = (int)l.len;
            u64 dp = 0;
            uint32_t di = 0;
            for (int j = threadIdx.x; j < len; j += SEL_T) {
                const u64 p = lp[l.base + j];
                const int id = li[l.base + j];
                sp[j] = p;
                si[j] = id;
                dp |= p ^ p0;
                di |= (uint32_t)(id ^ x0);
            }
            if (dp) atomicOr(&s_dp, dp);
            if (di) atomicOr(&s_di, di);
            __syncthreads();
            dp = s_dp;
            di = s_di;
            long long r = l.r, left = len;  // keys that agree with the digits so far
            for (int pass = 2; pass < 8; pass++) {
                SelBin f;
                if (key_digit(dp, (int)di, pass) == 0) {
                    f.bin = (int)key_digit(p0, x0, pass);
                    f.cum = 0;
                    f.cnt = (unsigned long long)left;
                } else {
                    for (int x = threadIdx.x; x < 4096; x += SEL_T) h[x] = 0;
                    __syncthreads();
                    for (int j = threadIdx.x; j < len; j += SEL_T) {
                        bool ok = true;
                        for (int q = 2; q < pass; q++)
                            ok = ok && key_digit(sp[j], si[j], q) == pre[q];
                        if (ok) atomicAdd(&h[key_digit(sp[j], si[j], pass)], 1u);
                    }
                    __syncthreads();
                    f = sel_bin([&](int b) { return h[b]; }, r);
                }
                if (threadIdx.x == 0) sel_settle<SEG>(rd, seg, l.i, f, r, pass);
                if (f.bin < 0 || (long long)(f.cum + f.cnt) == r) break;
                pre[pass] = (uint32_t)f.bin;
                r -= (long long)f.cum;
                left = (long long)f.cnt;
            }
        }
    }
    // the long ones: the whole cluster's.  Every block sees the same ones: only the
    // part above settles short lists, and a long one is settled behind a barrier.
    for (int i = i0; i < i0 + per && i < nseg; i++) {
        const SelList l = sel_list<SEG>(rd, seg, i);
        if (l.done || l.len <= SEL_SMEM) continue;
        long long r = l.r;
        for (int pass = 2; pass < 8; pass++) {
            __syncthreads();  // a short list's readers are done
            for (int x = threadIdx.x; x < 4096; x += SEL_T) h[x] = 0;
            cl.sync();  // every histogram is clear before counts are added to block 0's
            for (long long j = br * SEL_T + threadIdx.x; j < l.len; j += nb * SEL_T) {
                const u64 p = lp[l.base + j];
                const int id = li[l.base + j];
                bool ok = true;
                for (int q = 2; q < pass; q++) ok = ok && key_digit(p, id, q) == pre[q];
                if (ok) atomicAdd(&h[key_digit(p, id, pass)], 1u);
            }
            __syncthreads();
            if (br > 0) {
                uint32_t* h0 = cl.map_shared_rank(h, 0);
                for (int x = threadIdx.x; x < 4096; x += SEL_T)
                    if (h[x]) atomicAdd(&h0[x], h[x]);
            }
            cl.sync();
            if (br == 0) {
                const SelBin f = sel_bin([&](int b) { return h[b]; }, r);
                if (threadIdx.x == 0) {
                    s_f = f;
                    sel_settle<SEG>(rd, seg, i, f, r, pass);
                }
            }
            cl.sync();  // block 0's result
            const SelBin f = *cl.map_shared_rank(&s_f, 0);
            cl.sync();  // read by all before the next digit's (or block 0's exit)
            if (f.bin < 0 || (long long)(f.cum + f.cnt) == r) break;
            pre[pass] = (uint32_t)f.bin;
            r -= (long long)f.cum;
        }
    }
}

template <bool SEG>
static cudaError_t launch_rest(const u64* lp, const int* li, RoundDev* rd, SegDev* seg, int nseg,
                               cudaStream_t st) {
    // many scans: a block each, eight to a cluster
    const int per = nseg > SEL_CLUSTER_MAX ? SEL_CLUSTER : 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)((nseg + per - 1) / per * SEL_CLUSTER));
    c.blockDim = dim3(SEL_T);
    c.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = SEL_CLUSTER;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 2;
    note_launch();
    return cudaLaunchKernelEx(&c, sel_rest_kernel<SEG>, lp, li, rd, seg, nseg, per);
}

cudaError_t round_launch_select(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n,
                                SelBuffers& b, bool long_list, RoundDev* rd, cudaStream_t st) {
    int64_t blocks = (n + 4 * SEL_T - 1) / (4 * SEL_T);
    const int64_t lim = (int64_t)device_sms() * 4;
    if (blocks > lim) blocks = lim;
    if (blocks < 1) blocks = 1;
    const unsigned g = (unsigned)blocks;
    launch_chained(sel_pass_kernel<0, false>, g, SEL_T, 0, st, prim, alive, n, b.hist, rd,
                   nullptr, nullptr);
    launch_chained(sel_pass_kernel<1, false>, g, SEL_T, 0, st, prim, alive, n, b.hist, rd,
                   nullptr, nullptr);
    launch_chained(sel_list_kernel<false>, g, SEL_T, 0, st, prim, pos, alive, n, b.p, b.i, rd,
                   nullptr, nullptr);
    for (int i = 0; i < 3; i++) note_launch();
    if (long_list) {
        for (int pass = 2; pass < 8; pass++) {
            launch_chained(sel_digit_kernel, g, SEL_T, 0, st, b.p, b.i, pass, b.hist, rd);
            note_launch();
        }
        return cudaGetLastError();
    }
    const cudaError_t e = cudaGetLastError();
    return e ? e : launch_rest<false>(b.p, b.i, rd, nullptr, 1, st);
}

cudaError_t seg_launch_select(const u64* prim, const int4* pos, const uint8_t* alive, int64_t ng,
                              SelBuffers& b, uint32_t* hist, RoundDev* rd, SegDev* seg,
                              const int* items, int nseg, cudaStream_t st) {
    if (nseg < 1 || nseg > PD_SEG_MAX) return cudaErrorInvalidValue;
    // work items: at most ng / CHUNK + nseg; the launch size depends on the
    // layout only, so a captured round replays it unchanged
    int64_t blocks = ng / PD_SEG_CHUNK + nseg;
    const int64_t lim = (int64_t)device_sms() * 8;
    if (blocks > lim) blocks = lim;
    const unsigned g = (unsigned)blocks;
    launch_chained(sel_pass_kernel<0, true>, g, SEL_T, 0, st, prim, alive, ng, hist, rd, seg,
                   items);
    launch_chained(sel_pass_kernel<1, true>, g, SEL_T, 0, st, prim, alive, ng, hist, rd, seg,
                   items);
    launch_chained(sel_list_kernel<true>, g, SEL_T, 0, st, prim, pos, alive, ng, b.p, b.i, rd,
                   seg, items);
    for (int i = 0; i < 3; i++) note_launch();
    const cudaError_t e = cudaGetLastError();
    return e ? e : launch_rest<true>(b.p, b.i, rd, seg, nseg, st);
}

}  // namespace pd
