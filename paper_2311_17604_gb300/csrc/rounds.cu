// rounds.cu -- device-side removal rounds that reproduce the sequential greedy.
//
// The sequential greedy (section "Computing per-sample costs"; section
// "Sub-sampling algorithm", step 2: removing a point never raises a cost)
// pops the live point of largest key (cost, input index).  A round removes a
// set P at once; P is chosen so that the sequential run pops exactly the
// points of P among its next `need` pops and, apart from them, behaves as the
// run on the cloud without P:
//   (R2) key(p) >= K*, the need-th largest live key, so p is popped within
//        the next `need` pops once its key cannot change;
//   (A)  key(p) does not change when every point of larger key is removed,
//        so it stays fixed until p is popped;
//   (B)  p can never change the key of a point x that is popped before p
//        while x is not itself in P.
// k = 1: (A) holds iff p has no neighbour or some point at distance d1(p)
//        (the "shell") has a smaller key; (B) holds iff every shell member
//        of larger input index is itself in P (a fixpoint over P).
// k >= 2: (A) is checked by a neighbour search restricted to smaller keys;
//        (B) by counting, for every larger-key point x near p, the points of
//        key below key(p) that are closer to x than p is: p can enter x's k
//        nearest only if fewer than k of them exist (again a fixpoint).
// Before the rounds, coincident points (infinite cost) are removed in one
// step: all but the smallest input index of each coincident class are the
// first pops of the sequential run, in decreasing index order.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define FULLM 0xffffffffu

// ------------------------------------------------------------------ duplicates
__global__ void dup_flag_kernel(const u64* __restrict__ code, const int4* __restrict__ pos,
                                int64_t n, uint8_t* dup, unsigned long long* count) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned c = 0;
    if (s < n) {
        // coincident points share a code; where cells are wider than 1 mm (clouds
        // beyond 2^21 mm) so do other points, which may lie between them
        uint8_t f = 0;
        const u64 c0 = code[s];
        if (s > 0 && code[s - 1] == c0) {
            const int4 a = pos[s];
            for (int64_t j = s - 1; j >= 0 && !f && code[j] == c0; j--) {
                const int4 b = pos[j];
                f = a.x == b.x && a.y == b.y && a.z == b.z;
            }
        }
        dup[s] = f;
        c = f;
    }
    block_add(count, c);
}

// remove flagged duplicates whose input index is >= idx_min
__global__ void dup_remove_kernel(const uint8_t* __restrict__ dup, const int4* __restrict__ pos,
                                  int64_t n, int idx_min, uint8_t* alive) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    alive[s] = !(dup[s] && pos[s].w >= idx_min);
}

// ------------------------------------------------------------------ selection
// By the host, digit by digit: the largest key of a round that the device did not
// settle, and the coincident points to remove.  The rounds' own is select.cu.
__device__ inline bool prefix_match(u64 prim, int idx, int npass, const uint32_t* pre) {
    for (int p = 0; p < npass; p++)
        if (key_digit(prim, idx, p) != pre[p]) return false;
    return true;
}

struct SelPrefix {
    uint32_t d[8];
};

// Histogram of digit `pass`.  Grid mode (lp == NULL, pass 0 only): every
// alive grid point.  List mode: compacted (prim, idx) pairs that match the
// digits chosen so far.
__global__ void sel_hist_kernel(const u64* __restrict__ prim, const uint8_t* __restrict__ alive,
                                int64_t n, const u64* __restrict__ lp, const int* __restrict__ li,
                                int64_t llen, int pass, SelPrefix pre, uint32_t* hist) {
    __shared__ uint32_t h[4096];
    for (int x = threadIdx.x; x < 4096; x += blockDim.x) h[x] = 0;
    __syncthreads();
    int64_t len = lp ? llen : n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (lp) {
            u64 p = lp[i];
            int id = li[i];
            if (!prefix_match(p, id, pass, pre.d)) continue;
            atomicAdd(&h[key_digit(p, id, pass)], 1u);
        } else {
            if (!alive[i]) continue;
            atomicAdd(&h[(uint32_t)(prim[i] >> 52)], 1u);
        }
    }
    __syncthreads();
    for (int x = threadIdx.x; x < 4096; x += blockDim.x)
        if (h[x]) atomicAdd(&hist[x], h[x]);
}

// Keep the entries whose digits 0..pass equal pre[0..pass].
__global__ void sel_compact_kernel(const u64* __restrict__ prim, const int4* __restrict__ pos,
                                   const uint8_t* __restrict__ alive, int64_t n,
                                   const u64* __restrict__ lp, const int* __restrict__ li,
                                   int64_t llen, int pass, SelPrefix pre, u64* op, int* oi,
                                   int* ocount) {
    int64_t len = lp ? llen : n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < len;
         i += (int64_t)gridDim.x * blockDim.x) {
        u64 p;
        int id;
        if (lp) {
            p = lp[i];
            id = li[i];
            if (!prefix_match(p, id, pass + 1, pre.d)) continue;
        } else {
            if (!alive[i]) continue;
            p = prim[i];
            if ((uint32_t)(p >> 52) != pre.d[0]) continue;
            id = pos[i].w;
        }
        int slot = atomicAdd(ocount, 1);
        op[slot] = p;
        oi[slot] = id;
    }
}

// (B) for k = 1: a shell member of larger input index must be in P.  The
// shell is the first flg >> 2 stored neighbours.
__global__ void k1_fix_kernel(const int* __restrict__ cand, const int* __restrict__ ncand,
                              const int4* __restrict__ pos, const int* __restrict__ nbr,
                              const uint8_t* __restrict__ flg, int S,
                              const uint8_t* __restrict__ inP, uint8_t* rej, int* changed) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= *ncand) return;
    int s = cand[t];
    if (rej[s]) return;
    int is = pos[s].w;
    int shell = flg[s] >> 2;
    for (int i = 0; i < shell; i++) {
        int x = nbr[(int64_t)s * S + i];
        if (x < 0) continue;
        if (pos[x].w > is && (!inP[x] || rej[x])) {
            rej[s] = 1;
            *changed = 1;
            return;
        }
    }
}

#define DG_CAP 512
#define DG_SCAN 64   // larger octree nodes are entered by their children
#define DG_WARPS 2
#define DG_BLOCKS_PER_SM 14  // resident blocks per SM (registers capped to fit)
#define PD_DG_SMAX 8  // stored neighbours used as shields (S up to 8)

// The first level from L0 whose 3x3x3 cells around a point hold every point
// closer than sqrt(lam).
__device__ inline int cover_level(const GridView& g, int ux, int uy, int uz, int L0, u64 lam) {
    for (int L = L0; L < g.B; L++) {
        const int sh = L + g.shift;
        const int q[3] = {ux, uy, uz};
        const int m[3] = {g.umax.x, g.umax.y, g.umax.z};
        int best = 0x7fffffff;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int c = q[a] >> sh;  // faces are below 2^25 + 2 * 2^25: ints
            const int lo = (c - 1) * (1 << sh), hi = (c + 2) * (1 << sh);
            if (lo > 0) best = min(best, q[a] - lo + 1);
            if (hi <= m[a]) best = min(best, hi - q[a]);
        }
        if (best == 0x7fffffff || lam <= (u64)((long long)best * best)) return L;
    }
    return g.B;
}

// Danger pairs (condition (B), k >= 2).  One warp per source x (key above
// tau, lam = k-th squared distance from x to keys below tau):
//   1. collect the candidates p (in P so far, key below x's) with d^2(x,p) < lam,
//      from the candidates' bitmap over the ranges' positions (in Morton order
//      within a range, the ranges in kCellOrder);
//   2. for 32 candidates at a time stream every live point y with
//      d^2(x,y) < lam and count, per candidate, the y != p with
//      d^2(x,y) <= d^2(x,p) and key(y) < key(p), stopping once all 32 counts
//      reach k; a count below k means p could enter x's k nearest before p is
//      popped: record (x, p).
// Candidates beyond the list capacity are rejected without counting.
// A source's time is a chain of dependent loads, so the ranges are laid end to
// end (32 bitmap words, then 32 points a step, the next step's loads issued
// before this step's are used) instead of walked one by one, and octree nodes
// above DG_SCAN points are entered by their children (9.8M outdoor points, k =
// 4, 287 rounds: 95.6 -> 47.3 ms).  Candidates that the shields at hand leave open
// are gathered before the ball is streamed, so that it is streamed once per 32 of
// them (1.0M room points, k = 4, 112 rounds at 2 %: 9.7 -> 7.2 ms).
struct DangerSmem {
    int c_j[DG_WARPS][DG_CAP];
    u64 c_d[DG_WARPS][DG_CAP];
    union {
        struct {  // staged points within the batch's farthest candidate:
            u64 d[32], k[32];  // d^2 to the source, key, input index, Morton position
            int o[32], j[32];
        } st;
        int raw[192];  // candidate positions before the distance test
    } u[DG_WARPS];
};

// The range that holds item x of ranges laid end to end (inc: this lane's
// inclusive prefix count); every lane must call it.
__device__ __forceinline__ int range_of(uint32_t inc, uint32_t x) {
    int r = 0;
#pragma unroll
    for (int step = 16; step; step >>= 1) {
        const uint32_t v = __shfl_sync(FULLM, inc, r + step - 1);
        if (v <= x) r += step;
    }
    return r;
}
__device__ void danger_one(const GridView& g, int x, const u64* __restrict__ prim,
                           const uint8_t* __restrict__ alive, const uint32_t* __restrict__ inPb,
                           uint8_t* rej, const u64* __restrict__ lam, const int* __restrict__ nbr,
                           int S, int k, int2* pairs, int* npairs, int pair_cap, int* overflow,
                           unsigned long long* diag, DangerSmem& sm, int w, int lane) {
    int(&c_j)[DG_CAP] = sm.c_j[w];
    u64(&c_d)[DG_CAP] = sm.c_d[w];
    auto& u = sm.u[w];
    __syncwarp();
    int4 xp = g.pos[x];
    u64 px = prim[x];
    u64 lx = lam[x];
    if (lx == ~0ull) {  // fewer than k low points in the cloud: host falls back
        if (lane == 0) *overflow = 1;
        return;
    }
    int ux = xp.x - g.origin.x, uy = xp.y - g.origin.y, uz = xp.z - g.origin.z;
    const int L = cover_level(g, ux, uy, uz, g.leaf[x], lx);
    // nodes entirely beyond lam (or beyond the candidates being counted) are skipped
    WarpNode cell = warp_cells(g, L, g.code[x], ux, uy, uz, lane);
    const uint32_t rb = cell.b, re = cell.e;
    const bool rt = cell.count() > 0 && cell.box < lx;
    // 1. candidates
    int nc = 0;
    {
        const uint32_t w0 = rb >> 5, words = rt ? ((re - 1) >> 5) - w0 + 1 : 0;
        const uint32_t inc = warp_inclusive(words, lane);
        const uint32_t total = __shfl_sync(FULLM, inc, 31);
        for (uint32_t base = 0; base < total; base += 32) {
            const uint32_t t = base + lane;
            const int r = range_of(inc, t < total ? t : total - 1);
            const uint32_t b = __shfl_sync(FULLM, rb, r), e = __shfl_sync(FULLM, re, r);
            const uint32_t wb = __shfl_sync(FULLM, w0, r) +
                                (t - (__shfl_sync(FULLM, inc, r) - __shfl_sync(FULLM, words, r)));
            uint32_t bits = 0;
            if (t < total) {
                bits = inPb[wb];
                if (wb == (b >> 5)) bits &= 0xffffffffu << (b & 31);
                if (wb == (e - 1) >> 5) bits &= 0xffffffffu >> (31 - ((e - 1) & 31));
            }
            const uint32_t end = warp_inclusive((uint32_t)__popc(bits), lane);
            const uint32_t tot = __shfl_sync(FULLM, end, 31);
            uint32_t at = end - (uint32_t)__popc(bits);  // place of this lane's next bit
            for (uint32_t win = 0; win < tot; win += 192) {
                __syncwarp();
                while (bits && at < win + 192) {
                    u.raw[at - win] = (int)(wb * 32 + (uint32_t)__ffs(bits) - 1);
                    bits &= bits - 1;
                    at++;
                }
                __syncwarp();
                const uint32_t m = min(192u, tot - win);
                for (uint32_t c = 0; c < m; c += 32) {
                    bool take = false;
                    u64 d2 = 0;
                    int j = 0;
                    if (c + lane < m) {
                        j = u.raw[c + lane];
                        const int4 v = g.pos[j];
                        d2 = sqd(v, xp);
                        take = j != x && d2 < lx && key_gt(px, xp.w, prim[j], v.w);
                    }
                    const unsigned bal = __ballot_sync(FULLM, take);
                    const int slot = nc + __popc(bal & ((1u << lane) - 1u));
                    if (take) {
                        if (slot < DG_CAP) {
                            c_j[slot] = j;
                            c_d[slot] = d2;
                        } else {
                            rej[j] = 1;
                        }
                    }
                    nc += __popc(bal);
                }
            }
        }
    }
    if (diag && lane == 0) {
        if (nc > DG_CAP) atomicAdd(diag, (unsigned long long)(nc - DG_CAP));
    }
    nc = min(nc, DG_CAP);
    __syncwarp();
    if (nc == 0) return;
    // x's stored neighbours are live points near x: the cheapest shields, one
    // per lane
    int sn_j = -1, sn_i = 0;
    u64 sn_d = ~0ull, sn_k = 0;
    if (nbr && lane < S) {
        sn_j = nbr[(int64_t)x * S + lane];
        if (sn_j >= 0) {
            const int4 v = g.pos[sn_j];
            sn_d = sqd(v, xp);
            sn_k = prim[sn_j];
            sn_i = v.w;
        }
    }
    // 2. counting, 32 candidates at a time: this lane's
    int p = -1, ip = 0, cnt = 0;
    u64 dp = 0, pp = 0, dmax = 0, kmax = 0;
    bool done = true;
    auto take = [&](int at, int nlist) {
        done = at >= nlist;
        p = done ? -1 : c_j[at];
        dp = done ? 0 : c_d[at];
        pp = done ? 0 : prim[p];
        ip = done ? 0 : g.pos[p].w;
        cnt = 0;
    };
    // the farthest distance and the largest key of the open candidates
    auto reach = [&]() {
        dmax = done ? 0 : dp;
        kmax = done ? 0 : pp;
        for (int o = 16; o; o >>= 1) {
            const u64 d = __shfl_xor_sync(FULLM, dmax, o), q = __shfl_xor_sync(FULLM, kmax, o);
            dmax = d > dmax ? d : dmax;
            kmax = q > kmax ? q : kmax;
        }
    };
    // the open candidates move to the front of the list, from place `to` on
    auto keep_open = [&](int to) -> int {
        const unsigned m = __ballot_sync(FULLM, !done);
        __syncwarp();  // this batch was read
        if (!done) {
            const int at = to + __popc(m & ((1u << lane) - 1u));
            c_j[at] = p;
            c_d[at] = dp;
        }
        __syncwarp();
        return to + __popc(m);
    };
    // Streams the lanes' ranges [b, b + len): true once every count reached k.
    auto stream = [&](uint32_t b, uint32_t len) -> bool {
        const uint32_t inc = warp_inclusive(len, lane);
        const uint32_t total = __shfl_sync(FULLM, inc, 31);
        uint32_t jn = 0;  // a step's point: its fields loaded one step ahead
        int4 vn = make_int4(0, 0, 0, 0);
        u64 kn = 0;
        uint8_t an = 0;
        auto load = [&](uint32_t t) {
            const int r = range_of(inc, t < total ? t : total - 1);
            jn = __shfl_sync(FULLM, b, r) +
                 (t - (__shfl_sync(FULLM, inc, r) - __shfl_sync(FULLM, len, r)));
            an = 0;
            if (t < total) {
                an = alive[jn];
                vn = g.pos[jn];
                kn = prim[jn];
            }
        };
        if (total) load(lane);
        for (uint32_t base = 0; base < total; base += 32) {
            const uint32_t j = jn;
            const int4 v = vn;
            const u64 ky = kn;
            const uint8_t al = an;
            load(base + 32 + lane);
            // only points within the farthest open candidate and of smaller
            // key than the largest can shield: they are compacted into the
            // staging buffer
            const u64 d2 = sqd(v, xp);
            const bool near = al && (int)j != x && d2 <= dmax && ky <= kmax;
            const unsigned nb = __ballot_sync(FULLM, near);
            if (!nb) continue;
            if (near) {
                const int slot = __popc(nb & ((1u << lane) - 1u));
                u.st.d[slot] = d2;
                u.st.k[slot] = ky;
                u.st.o[slot] = v.w;
                u.st.j[slot] = (int)j;
            }
            __syncwarp();
            const int mm = __popc(nb);
            if (!done) {
                for (int tt = 0; tt < mm; tt++) {
                    if (u.st.j[tt] == p) continue;
                    if (u.st.d[tt] <= dp && key_gt(pp, ip, u.st.k[tt], u.st.o[tt])) {
                        if (++cnt >= k) {
                            done = true;
                            break;
                        }
                    }
                }
            }
            __syncwarp();
            if (__all_sync(FULLM, done)) return true;
        }
        return false;
    };
    // x's stored neighbours as shields
    int no = 0;
    for (int a0 = 0; a0 < nc; a0 += 32) {
        take(a0 + lane, nc);
        for (int i = 0; i < PD_DG_SMAX; i++) {
            const int yj = __shfl_sync(FULLM, sn_j, i), yi = __shfl_sync(FULLM, sn_i, i);
            const u64 yd = __shfl_sync(FULLM, sn_d, i), yk = __shfl_sync(FULLM, sn_k, i);
            if (yj >= 0 && yj != p && yd <= dp && key_gt(pp, ip, yk, yi)) cnt++;
        }
        if (cnt >= k) done = true;
        no = keep_open(no);
    }
    // many left: the points of the nearest cells as shields.  A candidate is
    // dangerous only if its key is among the k smallest of all points closer to
    // x, so few survive a hundred shields, and only batches of survivors stream
    // the whole ball.
    if (no > 32) {
        const int m = no;
        no = 0;
        for (int a0 = 0; a0 < m; a0 += 32) {
            take(a0 + lane, m);
            reach();
            const bool in = rt && lane < 7 && cell.count() <= DG_SCAN && cell.box <= dmax;
            stream(cell.b, in ? cell.count() : 0);
            no = keep_open(no);
        }
    }
    for (int a0 = 0; a0 < no; a0 += 32) {
        take(a0 + lane, no);
        reach();
        // small nodes at once, then the large ones by their children, nearest first
        WarpNode n = cell;
        const bool in = rt && n.box <= dmax;
        bool held = in && n.count() > DG_SCAN && n.lv > 0;
        bool fin = stream(n.b, in && !held ? n.count() : 0);
        while (!fin) {
            u64 next = held ? (n.box << 5) | lane : ~0ull;
            if (__all_sync(FULLM, next == ~0ull)) break;
            for (int o2 = 16; o2; o2 >>= 1) {
                const u64 v = __shfl_xor_sync(FULLM, next, o2);
                next = v < next ? v : next;
            }
            const int from = (int)(next & 31);
            const WarpNode c = warp_children(g, n, from, ux, uy, uz, lane);
            if (lane == from) held = false;
            bool now = c.count() > 0 && c.box <= dmax;
            bool keep = now && c.count() > DG_SCAN && c.lv > 0;
            const bool was = keep;
            warp_keep(n, held, c, keep, lane);
            if (was && !keep) now = false;
            fin = stream(c.b, now ? c.count() : 0);
        }
        if (!done) {
            int ps = atomicAdd(npairs, 1);
            if (ps < pair_cap) pairs[ps] = make_int2(x, p);
            else *overflow = 1;
        }
    }
}

__global__ void __launch_bounds__(DG_WARPS * 32, DG_BLOCKS_PER_SM)
    danger_kernel(GridView g, const int* __restrict__ src, const int* __restrict__ nsrc,
                  const u64* __restrict__ prim, const uint8_t* __restrict__ alive,
                  const uint32_t* __restrict__ inPb, uint8_t* rej, const u64* __restrict__ lam,
                  const int* __restrict__ nbr, int S, int k, int2* pairs, int* npairs,
                  int pair_cap, int* overflow, unsigned long long* diag, int* next) {
    __shared__ DangerSmem sm;
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int ns = *nsrc;
    // sources differ in time by two orders of magnitude: taken one by one (9.8M
    // outdoor points, k = 4, 2.6 sources a warp and round: 132 -> 125 ms)
    const int step = gridDim.x * DG_WARPS;
    for (int t = blockIdx.x * DG_WARPS + w; t < ns; t = step + warp_take(next, lane))
        danger_one(g, src[t], prim, alive, inPb, rej, lam, nbr, S, k, pairs, npairs, pair_cap,
                   overflow, diag, sm, w, lane);
}

// Fallback: accept every live point with key >= tau (tau = the top key).
__global__ void accept_above_kernel(const u64* __restrict__ prim, const int4* __restrict__ pos,
                                    const uint8_t* __restrict__ alive, int64_t n, u64 tp, int ti,
                                    uint8_t* inP, int* cand, int* ncand) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n || !alive[s]) return;
    if (key_gt(tp, ti, prim[s], pos[s].w)) return;
    inP[s] = 1;
    cand[atomicAdd(ncand, 1)] = (int)s;
}

// (B) fixpoint over pairs: p is rejected while its source x is not in P.
__global__ void pair_fix_kernel(const int2* __restrict__ pairs, const int* __restrict__ npairs,
                                int pair_cap, const uint8_t* __restrict__ inP, uint8_t* rej,
                                int* changed) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    int np = min(*npairs, pair_cap);
    if (t >= np) return;
    int2 pr = pairs[t];
    if (rej[pr.y]) return;
    if (!inP[pr.x] || rej[pr.x]) {
        rej[pr.y] = 1;
        *changed = 1;
    }
}

// ------------------------------------------------------------------ removal
__global__ void remove_kernel(const int* __restrict__ cand, const int* __restrict__ ncand,
                              uint8_t* inP, uint8_t* rej, uint8_t* alive,
                              unsigned long long* removed) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    unsigned c = 0;
    if (t < *ncand) {
        int s = cand[t];
        if (inP[s] && !rej[s]) {
            alive[s] = 0;
            c = 1;
        }
        inP[s] = 0;
        rej[s] = 0;
    }
    block_add(removed, c);
}

__global__ void keep_kernel(const int4* __restrict__ pos, const uint8_t* __restrict__ alive,
                            int64_t n, uint8_t* keep) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    if (alive[s]) keep[pos[s].w] = 1;
}

// cost / neighbour output in input order (pd_knn_cost)
__global__ void knn_out_kernel(const int4* pos, const double* cost_s, const int* nbr, int64_t n,
                               int S, int k, double* cost, int32_t* knn) {
    chain();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int i = pos[s].w;
    if (cost) cost[i] = cost_s[s];
    if (knn) {
        for (int j = 0; j < k; j++) {
            int x = nbr[s * S + j];
            knn[(int64_t)i * k + j] = x >= 0 ? pos[x].w : -1;
        }
    }
}

// remap stored neighbours after a compaction of the live points
__global__ void remap_kernel(const int* __restrict__ live_list, int64_t nl, const int* old_nbr,
                             int* new_nbr, const int* __restrict__ newpos, int64_t nold, int S) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= nl) return;
    int s = live_list[t];
    for (int i = 0; i < S; i++) {
        int x = old_nbr[(int64_t)s * S + i];
        new_nbr[t * S + i] = (x >= 0 && x < nold) ? newpos[x] : -1;
    }
}

template <typename T>
__global__ void take_kernel(const int* __restrict__ list, int64_t nl, const T* __restrict__ src,
                            T* dst) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < nl) dst[t] = src[list[t]];
}

__global__ void newpos_kernel(const int* __restrict__ list, int64_t nl, int* newpos) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t < nl) newpos[list[t]] = (int)t;
}

// ------------------------------------------------------------------ launchers
#define GRID1(n) (unsigned)(((n) + 255) / 256), 256

cudaError_t launch_dup_flag(const u64* code, const int4* pos, int64_t n, uint8_t* dup,
                            unsigned long long* count, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), st);
    if (e) return e;
    dup_flag_kernel<<<GRID1(n), 0, st>>>(code, pos, n, dup, count); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_dup_remove(const uint8_t* dup, const int4* pos, int64_t n, int idx_min,
                              uint8_t* alive, cudaStream_t st) {
    dup_remove_kernel<<<GRID1(n), 0, st>>>(dup, pos, n, idx_min, alive); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_sel_hist(const u64* prim, const uint8_t* alive, int64_t n, const u64* lp,
                            const int* li, int64_t llen, int pass, const uint32_t* pre,
                            uint32_t* hist, cudaStream_t st) {
    SelPrefix sp;
    for (int i = 0; i < 8; i++) sp.d[i] = i < pass ? pre[i] : 0;
    cudaError_t e = cudaMemsetAsync(hist, 0, 4096 * sizeof(uint32_t), st);
    if (e) return e;
    int64_t len = lp ? llen : n;
    int blocks = (int)((len + 255) / 256);
    if (blocks > device_sms() * 4) blocks = device_sms() * 4;
    if (blocks < 1) blocks = 1;
    sel_hist_kernel<<<blocks, 256, 0, st>>>(prim, alive, n, lp, li, llen, pass, sp, hist); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_sel_compact(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n,
                               const u64* lp, const int* li, int64_t llen, int pass,
                               const uint32_t* pre, u64* op, int* oi, int* ocount,
                               cudaStream_t st) {
    SelPrefix sp;
    for (int i = 0; i < 8; i++) sp.d[i] = i <= pass ? pre[i] : 0;
    cudaError_t e = cudaMemsetAsync(ocount, 0, sizeof(int), st);
    if (e) return e;
    int64_t len = lp ? llen : n;
    int blocks = (int)((len + 255) / 256);
    if (blocks > device_sms() * 8) blocks = device_sms() * 8;
    if (blocks < 1) blocks = 1;
    sel_compact_kernel<<<blocks, 256, 0, st>>>(prim, pos, alive, n, lp, li, llen, pass, sp, op,
                                               oi, ocount); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_k1_fix(const int* cand, const int* ncand, int max_cand, const int4* pos,
                          const int* nbr, const uint8_t* flg, int S, const uint8_t* inP,
                          uint8_t* rej, int* changed, cudaStream_t st) {
    if (max_cand <= 0) return cudaSuccess;
    k1_fix_kernel<<<GRID1(max_cand), 0, st>>>(cand, ncand, pos, nbr, flg, S, inP, rej, changed); note_launch();
    return cudaGetLastError();
}
cudaError_t round_launch_danger(const GridView& g, const int* src, const u64* prim,
                                const uint8_t* alive, const uint32_t* inPb, uint8_t* rej,
                                const u64* lam, const int* nbr, int S, int k, int2* pairs,
                                int pair_cap, int64_t n, RoundDev* rd, cudaStream_t st) {
    danger_kernel<<<list_blocks(n, 128, DG_BLOCKS_PER_SM), DG_WARPS * 32, 0, st>>>(
        g, src, &rd->nsrc, prim, alive, inPb, rej, lam, S <= PD_DG_SMAX ? nbr : nullptr, S, k,
        pairs, &rd->npairs, pair_cap, &rd->overflow, &rd->cap_over, &rd->take_src); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_accept_above(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n,
                                u64 tp, int ti, uint8_t* inP, int* cand, int* ncand,
                                cudaStream_t st) {
    accept_above_kernel<<<GRID1(n), 0, st>>>(prim, pos, alive, n, tp, ti, inP, cand, ncand); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_pair_fix(const int2* pairs, const int* npairs, int max_pairs, int pair_cap,
                            const uint8_t* inP, uint8_t* rej, int* changed, cudaStream_t st) {
    if (max_pairs <= 0) return cudaSuccess;
    pair_fix_kernel<<<GRID1(max_pairs), 0, st>>>(pairs, npairs, pair_cap, inP, rej, changed); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_remove(const int* cand, const int* ncand, int max_cand, uint8_t* inP,
                          uint8_t* rej, uint8_t* alive, unsigned long long* removed,
                          cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(removed, 0, sizeof(unsigned long long), st);
    if (e || max_cand <= 0) return e;
    remove_kernel<<<GRID1(max_cand), 0, st>>>(cand, ncand, inP, rej, alive, removed); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_keep(const int4* pos, const uint8_t* alive, int64_t n, uint8_t* keep,
                        cudaStream_t st) {
    keep_kernel<<<GRID1(n), 0, st>>>(pos, alive, n, keep); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_knn_out(const int4* pos, const double* cost_s, const int* nbr, int64_t n, int S,
                           int k, double* cost, int32_t* knn, cudaStream_t st) {
    launch_chained(knn_out_kernel, GRID1(n), 0, st, pos, cost_s, nbr, n, S, k, cost, knn);
    note_launch();
    return cudaGetLastError();
}
cudaError_t launch_newpos(const int* list, int64_t nl, int* newpos, cudaStream_t st) {
    newpos_kernel<<<GRID1(nl), 0, st>>>(list, nl, newpos); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_remap(const int* list, int64_t nl, const int* old_nbr, int* new_nbr,
                         const int* newpos, int64_t nold, int S, cudaStream_t st) {
    remap_kernel<<<GRID1(nl), 0, st>>>(list, nl, old_nbr, new_nbr, newpos, nold, S); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_take_u64(const int* list, int64_t nl, const u64* src, u64* dst,
                            cudaStream_t st) {
    take_kernel<u64><<<GRID1(nl), 0, st>>>(list, nl, src, dst); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_take_i4(const int* list, int64_t nl, const int4* src, int4* dst,
                           cudaStream_t st) {
    take_kernel<int4><<<GRID1(nl), 0, st>>>(list, nl, src, dst); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_take_u8(const int* list, int64_t nl, const uint8_t* src, uint8_t* dst,
                           cudaStream_t st) {
    take_kernel<uint8_t><<<GRID1(nl), 0, st>>>(list, nl, src, dst); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_take_uc4(const int* list, int64_t nl, const uchar4* src, uchar4* dst,
                            cudaStream_t st) {
    take_kernel<uchar4><<<GRID1(nl), 0, st>>>(list, nl, src, dst); note_launch();
    return cudaGetLastError();
}
cudaError_t launch_take_f4(const int* list, int64_t nl, const float4* src, float4* dst,
                           cudaStream_t st) {
    take_kernel<float4><<<GRID1(nl), 0, st>>>(list, nl, src, dst); note_launch();
    return cudaGetLastError();
}

}  // namespace pd
