// rounds_dev.cu -- removal rounds driven from device memory.
//
// One round is a fixed sequence of launches whose sizes never depend on
// counts computed in the round: the threshold tau comes from an on-device
// radix select (select.cu), candidate / source / pair / query lists are appended
// with atomics and walked by grid-stride or persistent kernels, and the fixpoint
// runs a fixed number of launches.  The host reads the small RoundDev block once
// per round.
// The rules themselves (R2, A, B) are documented in rounds.cu.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define FULLM 0xffffffffu

// Appends s to list[*count ...] for every thread with want set, one atomic
// per block; every thread of the block must call it.
__device__ __forceinline__ void list_append(bool want, int s, int* count, int* list) {
    const int slot = block_append(want, count);
    if (want) list[slot] = s;
}

// ------------------------------------------------------------------ k = 1
__global__ void k1d_cand_kernel(const u64* prim, const int4* pos, const uint8_t* alive,
                                const int* nbr, const int* nbr0, const uint8_t* flg, int64_t n,
                                int S, RoundDev* rd, uint8_t* inP, int* cand, int* slow, int* dep) {
    chain();
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool c = false, sl = false, dp = false;
    const bool in = s < n;
    const uint8_t al = in ? alive[s] : 0;
    const u64 ps = in ? prim[s] : 0;  // loaded beside the alive flag, not after it
    if (al) {
        u64 tp = rd->tau_prim;  // packed batch: the least threshold over the scans
        if (ps >= tp) {  // below the threshold on the primary: no index needed
            int ti = rd->tau_idx;
            int is;
            if (rd->seg) {  // packed batch: the threshold of the point's own scan
                const int4 p4 = pos[s];
                is = p4.w;
                round_tau(rd, p4, tp, ti);
            } else {
                is = pos[s].w;
            }
            if (!key_gt(tp, ti, ps, is)) {
                const uint8_t fl = flg[s];
                if (fl & 2) {
                    sl = true;
                } else {
                    // the shell (points at the nearest distance) is the first
                    // fl >> 2 stored neighbours; none: a lone point
                    const int shell = fl >> 2;
                    bool ok = shell == 0, larger = false;
                    for (int i = 0; i < shell; i++) {
                        const int x = i == 0 && nbr0 ? nbr0[s] : nbr[s * S + i];
                        const int ix = pos[x].w;
                        if (key_gt(ps, is, prim[x], ix)) ok = true;
                        if (ix > is) larger = true;
                    }
                    c = ok;
                    dp = ok && larger;
                }
            }
        }
    }
    // list appends aggregated per block (every thread reaches them)
    if (c) inP[s] = 1;
    list_append(c, (int)s, &rd->ncand, cand);
    list_append(sl, (int)s, &rd->nslow, slow);
    list_append(dp, (int)s, &rd->ndep, dep);
}

// overflowing shells: accept iff every live point at distance d1 has a
// smaller key (grid-stride over the slow list)
__global__ void k1d_slow_kernel(GridView g, const u64* prim, const uint8_t* alive, const u64* rk2,
                                const int* slow, RoundDev* rd, uint8_t* inP, int* cand) {
    chain();
    int ns = rd->nslow;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < ns; t += gridDim.x * blockDim.x) {
        int s = slow[t];
        int4 qp = g.pos[s];
        u64 r2 = rk2[s];
        u64 ps = prim[s];
        int ux = qp.x - g.origin.x, uy = qp.y - g.origin.y, uz = qp.z - g.origin.z;
        u64 c0 = g.code[s];
        bool ok = true;
        for (int L = g.leaf[s]; L <= g.B; L++) {
            int cx = 0, cy = 0, cz = 0;
            if (L < g.B) {
                cx = (int)compact3(c0 >> (3 * L));
                cy = (int)compact3(c0 >> (3 * L + 1));
                cz = (int)compact3(c0 >> (3 * L + 2));
            }
            int sh = L + g.shift;
            long long q[3] = {ux, uy, uz};
            int c[3] = {cx, cy, cz};
            int m[3] = {g.umax.x, g.umax.y, g.umax.z};
            long long best = -1;
            for (int a = 0; a < 3; a++) {
                long long lo = (long long)(c[a] - 1) << sh, hi = (long long)(c[a] + 2) << sh;
                if (lo > 0 && (best < 0 || q[a] - lo + 1 < best)) best = q[a] - lo + 1;
                if (hi <= m[a] && (best < 0 || hi - q[a] < best)) best = hi - q[a];
            }
            bool covered = L >= g.B || best < 0 || r2 < (u64)best * (u64)best;
            if (!covered) continue;
            for (int o = 0; o < 27 && ok; o++) {
                int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
                uint32_t b, e;
                int lvl;
                if (!resolve_cell(g, L, cx + dx, cy + dy, cz + dz, b, e, &lvl)) continue;
                for (uint32_t j = b; j < e && ok; j++) {
                    if ((int)j == s || !alive[j]) continue;
                    int4 v = g.pos[j];
                    long long dx2 = v.x - qp.x, dy2 = v.y - qp.y, dz2 = v.z - qp.z;
                    u64 d2 = (u64)(dx2 * dx2 + dy2 * dy2 + dz2 * dz2);
                    if (d2 == r2 && key_gt(prim[j], v.w, ps, qp.w)) ok = false;
                }
            }
            break;
        }
        if (ok) {
            inP[s] = 1;
            cand[atomicAdd(&rd->ncand, 1)] = s;
        }
    }
}

// Condition (B) only ever rejects more, so the sweeps of its fixpoint may run in
// any order: a block repeats its own sweep until it changes nothing (at most
// PD_FIX_INNER times), seeing other blocks' rejections as they land.  A launch
// in which nothing changed anywhere has checked everything against one state:
// the fixpoint; the launches after it return at once.  (A launch per sweep, up
// to 32 a round, were 608 launches and 1.11 ms of the 200k-point room scan;
// now 114 and 0.28 ms.)
template <class Sweep>
__device__ __forceinline__ void fix_sweeps(RoundDev* rd, int iter, Sweep sweep) {
    if (iter > 0 && !rd->changed[iter - 1]) return;
    bool any = false;
    for (int s = 0; s < PD_FIX_INNER; s++) {
        const bool c = sweep();
        any = any || c;
        if (!__syncthreads_or(c)) break;
    }
    if (any) rd->changed[iter] = 1;
}

__global__ void k1d_fix_kernel(const int* cand, const int4* pos, const int* nbr,
                               const uint8_t* flg, int S, const uint8_t* inP, uint8_t* rej,
                               int iter, RoundDev* rd) {
    chain();
    const volatile uint8_t* vrej = rej;
    const int nc = rd->ndep;  // cand: the dep list (only its members can be rejected)
    fix_sweeps(rd, iter, [&]() {
        bool c = false;
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nc; t += gridDim.x * blockDim.x) {
            const int s = cand[t];
            if (vrej[s]) continue;
            const int is = pos[s].w;
            const int shell = flg[s] >> 2;
            for (int i = 0; i < shell; i++) {
                const int x = nbr[(int64_t)s * S + i];
                if (pos[x].w > is && (!inP[x] || vrej[x])) {
                    rej[s] = 1;
                    c = true;
                    break;
                }
            }
        }
        return c;
    });
}

__global__ void pairs_fix_kernel(const int2* __restrict__ pairs, int pair_cap,
                                 const uint8_t* __restrict__ inP, uint8_t* rej, int iter,
                                 RoundDev* rd) {
    const volatile uint8_t* vrej = rej;
    const int np = min(rd->npairs, pair_cap);
    fix_sweeps(rd, iter, [&]() {
        bool c = false;
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < np; t += gridDim.x * blockDim.x) {
            const int2 pr = pairs[t];
            if (vrej[pr.y]) continue;
            if (!inP[pr.x] || vrej[pr.x]) {
                rej[pr.y] = 1;
                c = true;
            }
        }
        return c;
    });
}

// ------------------------------------------------------------------ removal
// Removes the accepted candidates unless the round must be settled on the
// host (danger overflow, or a fixpoint that did not converge in the fixed
// number of sweeps); candidate marks are cleared in the normal case.
__global__ void removed_kernel(const int* cand, uint8_t* inP, uint8_t* rej, uint8_t* alive,
                               RoundDev* rd) {
    chain();
    __shared__ int hold;
    if (threadIdx.x == 0) {
        int fi = rd->fix_iters;
        if (fi < 1 || fi > PD_FIX_ITERS) fi = PD_FIX_ITERS;
        const int last = rd->changed[fi - 1];
        hold = rd->overflow || last;
        if (hold && blockIdx.x == 0) rd->fix_unconverged = last;
    }
    __syncthreads();
    if (hold) return;
    int nc = rd->ncand;
    unsigned c = 0;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nc; t += gridDim.x * blockDim.x) {
        int s = cand[t];
        if (inP[s] && !rej[s]) {
            alive[s] = 0;
            c++;
        }
        inP[s] = 0;
        rej[s] = 0;
    }
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(FULLM, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&rd->removed, (unsigned long long)c);
}

__global__ void dirtyd_kernel(const uint8_t* alive, const int* nbr, int64_t n, int S, int kchk,
                              int* list, RoundDev* rd) {
    chain();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool d = false;
    if (s < n && alive[s]) {
        for (int i = 0; i < kchk; i++) {
            int x = nbr[s * S + i];
            if (x >= 0 && !alive[x]) d = true;
        }
    }
    list_append(d, (int)s, &rd->nreq, list);
}

// ------------------------------------------------------------------ k = 1 buffer
// k = 1 density cost: every point stores its S nearest live points exactly,
// with the horizon h = the S-th squared distance at search time (any live
// point not stored lies at d^2 >= h; h = ~0 when all live points were
// stored).  After removals, the first live stored entry is the new nearest;
// its shell (the stored entries at that distance) is complete when that
// distance is below h, and the key follows without a search.  Otherwise, or
// when no stored entry is left, the point is searched again.

// 40 registers, 6 blocks of 256 per SM: the update waits on dependent loads,
// and more threads in flight measured faster (rules of the 100M-point scan
// 52.9 -> 51.5 ms)
__global__ void __launch_bounds__(256, 6)
    k1d_update_kernel(BufView b, const uint8_t* alive, int64_t n, int* list, RoundDev* rd) {
    chain();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool req = false;
    if (s < n) {
        // only a removed shell member changes the key or the shell; removed
        // entries past the shell stay stored (stale) until the shell changes
        // the point's flag, shell size and first entry are loaded together
        // (the first entry from its coalesced copy: most shells hold one
        // point), so that only the entry's alive flag waits on them
        bool shell_hit = false;
        const uint8_t al = alive[s];
        const int shell = b.flg[s] >> 2;
        const int x0 = b.nbr0 ? b.nbr0[s] : b.nbr[s * 8];
        if (al && shell > 0) {
            shell_hit = !alive[x0];
            for (int i = 1; i < shell && !shell_hit; i++) shell_hit = !alive[b.nbr[s * 8 + i]];
        }
        if (shell_hit) {
            int ids[8];
            load_nbr8(b.nbr, s, ids);
            const int r = keep_live8(alive, ids);
            const u64 h = b.hz[s];
            const int4 ps = b.pos[s];
            u64 d[8];
#pragma unroll
            for (int i = 0; i < 8; i++) d[i] = i < r ? sqd(ps, b.pos[ids[i]]) : ~0ull;
            if (r > 0 && (h == ~0ull || d[0] < h)) {
                int sh = 1;
#pragma unroll
                for (int i = 1; i < 8; i++) sh += i < r && d[i] == d[0];
                b.prim[s] = key_prim_d2(d[0]);
                b.rk2[s] = d[0];
                b.flg[s] = (uint8_t)((sh >= 2 ? 1 : 0) | (sh << 2));
                store_nbr8(b.nbr, s, ids);
                if (b.nbr0) b.nbr0[s] = ids[0];
            } else {
                req = true;
            }
        }
    }
    list_append(req, (int)s, &rd->nreq, list);
}

// ------------------------------------------------------------------ k+b buffer
// Every point stores its S nearest live points exactly, plus the horizon h =
// the S-th squared distance when they were searched: any point not stored
// lies at d^2 >= h.  After removals the live stored entries, in order, are
// still the nearest live points, so as long as k of them remain the new cost
// follows without a search (the paper's extended k+b neighbourhood, section
// "Sub-sampling algorithm").  Fewer than k left: the point is searched again.

// Nearly every point lost nothing, so a block first runs that test over
// UPD_SPAN points (a point's 8 entries as two 16-byte loads beside its live flag,
// then the entries' flags together) and lists the others in shared memory; its
// threads then take the listed points densely, each point's positions and
// weights loaded side by side.  With the recomputation inside the test, every
// warp that held one such point waited for its chain of loads and binary64
// divisions (all rounds: 9.8M outdoor points, k = 4, 32.4 -> 21.0 ms; a packed batch
// of 3.8M with colours 22.8 -> 15.3 ms).
#define UPD_SPAN 512

__global__ void __launch_bounds__(256, 4)
    kkd_update_kernel(BufView b, const uint8_t* __restrict__ alive, int64_t n, int k, int* list,
                      RoundDev* rd) {
    __shared__ int s_list[UPD_SPAN];
    __shared__ int s_n;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t base = blockIdx.x * (int64_t)UPD_SPAN;
    {
        bool hit[UPD_SPAN / 256];
        int x[UPD_SPAN / 256][8];
        uint8_t al[UPD_SPAN / 256];
#pragma unroll
        for (int j = 0; j < UPD_SPAN / 256; j++) {
            const int64_t s = base + j * 256 + threadIdx.x;
            al[j] = 0;
            if (s < n) {
                al[j] = alive[s];
                load_nbr8(b.nbr, s, x[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < UPD_SPAN / 256; j++) {
            hit[j] = false;
            if (al[j]) {
                const int s = (int)(base + j * 256 + threadIdx.x);
#pragma unroll
                for (int i = 0; i < 8; i++) hit[j] |= !alive[x[j][i] >= 0 ? x[j][i] : s];
            }
        }
#pragma unroll
        for (int j = 0; j < UPD_SPAN / 256; j++) {
            const unsigned m = __ballot_sync(FULLM, hit[j]);
            if (!m) continue;
            const int lane = threadIdx.x & 31;
            int at = 0;
            if (lane == __ffs(m) - 1) at = atomicAdd(&s_n, __popc(m));
            at = __shfl_sync(FULLM, at, __ffs(m) - 1);
            if (hit[j])
                s_list[at + __popc(m & ((1u << lane) - 1u))] =
                    (int)(base + j * 256 + threadIdx.x);
        }
    }
    __syncthreads();
    const int m = s_n;
    for (int e0 = 0; e0 < m; e0 += 256) {  // uniform over the block
        const int e = e0 + threadIdx.x;
        bool req = false;
        int s = 0;
        if (e < m) {
            s = s_list[e];
            int ids[8];
            load_nbr8(b.nbr, s, ids);
            const int4 ps = b.pos[s];
            const u64 h = b.hz[s];
            const int r = keep_live8(alive, ids);
            if (r >= k) {
                u64 d[8];
                double w[8];
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    d[i] = i < r && i <= k ? sqd(ps, b.pos[ids[i]]) : ~0ull;
                    w[i] = 1.0;
                    if (b.term && i < k) w[i] = term_weight(b.term, b.weight, b.rgb, b.nrm, s, ids[i]);
                }
                double c = 0.0;
                u64 dk = 0, dk1 = ~0ull;
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    if (i < k) {  // r >= k
                        c = __dadd_rn(c, __ddiv_rn(w[i], (double)d[i]));
                        dk = d[i];
                    }
                    if (i == k) dk1 = d[i];
                }
                const bool tie = (r > k && dk1 == dk) || (h != ~0ull && dk == h);
                b.prim[s] = key_prim_cost(c);
                b.rk2[s] = dk;
                b.flg[s] = tie ? 1 : 0;
                store_nbr8(b.nbr, s, ids);
            } else {
                req = true;
            }
        }
        list_append(req, s, &rd->nreq, list);
    }
}

// Candidate test (k >= 2) using the stored buffer where it suffices:
//   (A) the cost over smaller keys is the cost over the first k stored entries
//       of smaller key, when k of them are stored (any unstored point is at
//       least as far as every stored one); otherwise a filtered search.
//   lam (danger sources): the k-th stored squared distance of key below tau,
//       when k such entries are stored; otherwise a search.
// Alongside: the bitmap of the candidates and the least live key of every
// 32-position chunk.
// A block first streams CAND_SPAN points (live flag and key, 4 points a thread
// in one load each) and lists those above the threshold, one or two in a
// hundred, in shared memory; then its threads take the listed points densely,
// all gathers of a point (neighbour, key, position) issued together.  With a
// thread per point the few above the threshold ran their chain of dependent
// loads in nearly empty warps (9.8M outdoor points, k = 4, 287 rounds: 31.2 -> 10.9 ms).
#define CAND_SPAN 1024

// One point above the threshold on its primary key.
struct CandOut {
    bool isc, iss, fq, lq;
};
template <bool S8>
__device__ __forceinline__ CandOut cand_point(const BufView& b, int64_t s, int S, int k,
                                              const RoundDev* rd, u64* lam) {
    CandOut o = {false, false, false, false};
    const u64 ps = b.prim[s];
    const int4 qs = b.pos[s];
    const uint8_t fl = b.flg[s];
    const int is = qs.w;
    u64 tp = rd->tau_prim;
    int ti = rd->tau_idx;
    if (rd->seg) round_tau(rd, qs, tp, ti);
    bool lower = !(fl & 1), band_nbr = (fl & 1) != 0;
    int nfound = 0;
    if (S8) {
        int x[8];
        load_nbr8(b.nbr, s, x);
        u64 px[8];
        int4 p4[8];
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int y = x[i] >= 0 ? x[i] : (int)s;
            px[i] = b.prim[y];
            p4[i] = b.pos[y];
        }
        if (key_gt(tp, ti, ps, is)) return o;
        bool less[8], low[8];  // key below the point's, below tau
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const bool in = x[i] >= 0;
            less[i] = in && key_gt(ps, is, px[i], p4[i].w);
            low[i] = in && key_gt(tp, ti, px[i], p4[i].w);
            nfound += in;
            if (in && i < k) {
                if (!less[i]) lower = false;  // keys are distinct
                if (!low[i]) band_nbr = true;
            }
        }
        if (nfound < k) band_nbr = true;
        o.isc = lower;
        if (!lower) {
            // cost over the first k stored entries of smaller key
            double c = 0.0;
            int cnt = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                if (less[i] && cnt < k) {
                    const double w = term_weight(b.term, b.weight, b.rgb, b.nrm, (int)s, x[i]);
                    c = __dadd_rn(c, __ddiv_rn(w, (double)sqd(qs, p4[i])));
                    cnt++;
                }
            }
            if (cnt >= k) o.isc = key_prim_cost(c) == ps;
            else o.fq = true;
        }
        if (key_gt(ps, is, tp, ti) && band_nbr) {
            int cnt = 0;
            u64 l = ~0ull;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                if (low[i] && cnt < k) {
                    l = sqd(qs, p4[i]);
                    cnt++;
                }
            }
            if (cnt >= k) lam[s] = l;
            else o.lq = true;
            o.iss = true;
        }
        return o;
    }
    if (key_gt(tp, ti, ps, is)) return o;
    for (int i = 0; i < S; i++) {
        int x = b.nbr[s * S + i];
        if (x < 0) continue;
        nfound++;
        if (i >= k) continue;
        u64 px = b.prim[x];
        int ix = b.pos[x].w;
        if (key_gt(px, ix, ps, is)) lower = false;
        if (!key_gt(tp, ti, px, ix)) band_nbr = true;
    }
    if (nfound < k) band_nbr = true;
    o.isc = lower;
    if (!lower) {
        double c = 0.0;
        int cnt = 0;
        for (int i = 0; i < S && cnt < k; i++) {
            int x = b.nbr[s * S + i];
            if (x < 0) continue;
            int4 px4 = b.pos[x];
            if (!key_gt(ps, is, b.prim[x], px4.w)) continue;
            double w = term_weight(b.term, b.weight, b.rgb, b.nrm, (int)s, x);
            c = __dadd_rn(c, __ddiv_rn(w, (double)sqd(qs, px4)));
            cnt++;
        }
        if (cnt >= k) o.isc = key_prim_cost(c) == ps;
        else o.fq = true;
    }
    if (key_gt(ps, is, tp, ti) && band_nbr) {
        int cnt = 0;
        u64 l = ~0ull;
        for (int i = 0; i < S && cnt < k; i++) {
            int x = b.nbr[s * S + i];
            if (x < 0) continue;
            int4 px4 = b.pos[x];
            if (!key_gt(tp, ti, b.prim[x], px4.w)) continue;
            l = sqd(qs, px4);
            cnt++;
        }
        if (cnt >= k) lam[s] = l;
        else o.lq = true;
        o.iss = true;
    }
    return o;
}

template <bool S8>
__global__ void __launch_bounds__(256, 3)
    kkd_cand2_kernel(BufView b, const uint8_t* __restrict__ alive, int64_t n, int S, int k,
                     RoundDev* rd, uint8_t* inP, uint32_t* inPb, int* cand, int* fq_list,
                     int* lq_list, u64* lam, int* src, u64* cmin) {
    __shared__ int s_list[CAND_SPAN];
    __shared__ uint32_t s_bits[CAND_SPAN / 32];
    __shared__ int s_n;
    const int t = threadIdx.x;
    if (t == 0) s_n = 0;
    if (t < CAND_SPAN / 32) s_bits[t] = 0;
    __syncthreads();
    const int64_t base = blockIdx.x * (int64_t)CAND_SPAN, s0 = base + 4 * t;
    u64 p[4] = {~0ull, ~0ull, ~0ull, ~0ull};
    bool al[4] = {false, false, false, false};
    if (s0 + 3 < n) {  // both arrays start aligned and s0 is a multiple of 4
        const uchar4 a = *reinterpret_cast<const uchar4*>(alive + s0);
        const ulonglong2 u = *reinterpret_cast<const ulonglong2*>(b.prim + s0);
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(b.prim + s0 + 2);
        al[0] = a.x;
        al[1] = a.y;
        al[2] = a.z;
        al[3] = a.w;
        p[0] = u.x;
        p[1] = u.y;
        p[2] = v.x;
        p[3] = v.y;
    } else {
        for (int j = 0; j < 4; j++)
            if (s0 + j < n) {
                al[j] = alive[s0 + j];
                p[j] = b.prim[s0 + j];
            }
    }
    const u64 tp = rd->tau_prim;
    u64 low = ~0ull;
    int c = 0;
#pragma unroll
    for (int j = 0; j < 4; j++) {
        if (al[j] && p[j] < low) low = p[j];
        c += al[j] && p[j] >= tp;
    }
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        const u64 v = __shfl_xor_sync(FULLM, low, o);
        low = v < low ? v : low;
    }
    if ((t & 7) == 0 && s0 < n) cmin[s0 >> 5] = low;
    if (c) {
        bool in[4];
#pragma unroll
        for (int j = 0; j < 4; j++) in[j] = al[j] && p[j] >= tp;
        if (rd->seg) {
            // packed batch: tau_prim is the least threshold over the scans,
            // each point answers to its own scan's
            int4 q[4];
#pragma unroll
            for (int j = 0; j < 4; j++)
                if (in[j]) q[j] = b.pos[s0 + j];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (in[j]) {
                    u64 sp;
                    int si;
                    round_tau(rd, q[j], sp, si);
                    in[j] = p[j] >= sp;
                }
            }
        }
        c = in[0] + in[1] + in[2] + in[3];
        int at = c ? atomicAdd(&s_n, c) : 0;
#pragma unroll
        for (int j = 0; j < 4; j++)
            if (in[j]) s_list[at++] = (int)(s0 + j);
    }
    __syncthreads();
    const int m = s_n;
    for (int e0 = 0; e0 < m; e0 += 256) {  // uniform over the block
        const int e = e0 + t;
        CandOut o = {false, false, false, false};
        int s = 0;
        if (e < m) {
            s = s_list[e];
            o = cand_point<S8>(b, s, S, k, rd, lam);
            if (o.isc) {
                inP[s] = 1;
                const int r = s - (int)base;
                atomicOr(&s_bits[r >> 5], 1u << (r & 31));
            }
        }
        const bool want[4] = {o.isc, o.iss, o.fq, o.lq};
        int* const count[4] = {&rd->ncand, &rd->nsrc, &rd->nfq, &rd->nlq};
        int slot[4];
        block_append_n(want, count, slot);
        if (o.isc) cand[slot[0]] = s;
        if (o.iss) src[slot[1]] = s;
        if (o.fq) fq_list[slot[2]] = s;
        if (o.lq) lq_list[slot[3]] = s;
    }
    __syncthreads();
    if (t < CAND_SPAN / 32 && base + 32 * t < n) inPb[(base >> 5) + t] = s_bits[t];
}

// ------------------------------------------------------------------ launchers
#define GRID1(n) (unsigned)(((n) + 255) / 256), 256

cudaError_t round_launch_k1(const GridView& g, const u64* prim, const uint8_t* alive,
                            const int* nbr, const int* nbr0, const uint8_t* flg, const u64* rk2,
                            int64_t n, int S, RoundDev* rd, uint8_t* inP, uint8_t* rej, int* cand,
                            int* slow, int* dep, int fix_iters, cudaStream_t st) {
    if (fix_iters < 1 || fix_iters > PD_FIX_ITERS) return cudaErrorInvalidValue;
    launch_chained(k1d_cand_kernel, GRID1(n), 0, st, prim, g.pos, alive, nbr, nbr0, flg, n, S, rd,
                   inP, cand, slow, dep);
    note_launch();
    launch_chained(k1d_slow_kernel, list_blocks(n, 4096, 4), 128, 0, st, g, prim, alive, rk2,
                   slow, rd, inP, cand);
    note_launch();
    for (int it = 0; it < fix_iters; it++) {
        launch_chained(k1d_fix_kernel, list_blocks(n, 2048, 8), 256, 0, st, dep, g.pos, nbr, flg,
                       S, inP, rej, it, rd);
        note_launch();
    }
    return cudaGetLastError();
}

cudaError_t round_launch_pairs_fix(const int2* pairs, int pair_cap, const uint8_t* inP,
                                   uint8_t* rej, int64_t n, RoundDev* rd, cudaStream_t st) {
    for (int it = 0; it < PD_FIX_ITERS_KK; it++) {
        pairs_fix_kernel<<<list_blocks(n, 4096, 8), 256, 0, st>>>(pairs, pair_cap, inP, rej, it, rd);
        note_launch();
    }
    return cudaGetLastError();
}

cudaError_t round_launch_remove(const int* cand, uint8_t* inP, uint8_t* rej, uint8_t* alive,
                                int64_t n, RoundDev* rd, cudaStream_t st) {
    launch_chained(removed_kernel, list_blocks(n, 4096, 8), 256, 0, st, cand, inP, rej, alive, rd);
    note_launch();
    return cudaGetLastError();
}

cudaError_t round_launch_dirty(const uint8_t* alive, const int* nbr, int64_t n, int S, int kchk,
                               int* list, RoundDev* rd, cudaStream_t st) {
    launch_chained(dirtyd_kernel, GRID1(n), 0, st, alive, nbr, n, S, kchk, list, rd);
    note_launch();
    return cudaGetLastError();
}

}  // namespace pd

namespace pd {
cudaError_t round_launch_k1_update(const BufView& b, const uint8_t* alive, int64_t n, int S,
                                   int* list, RoundDev* rd, cudaStream_t st) {
    if (S != 8) return cudaErrorInvalidValue;
    launch_chained(k1d_update_kernel, GRID1(n), 0, st, b, alive, n, list, rd);
    note_launch();
    return cudaGetLastError();
}
cudaError_t round_launch_kk_update(const BufView& b, const uint8_t* alive, int64_t n, int S, int k,
                                   int* list, RoundDev* rd, cudaStream_t st) {
    if (S != 8) return cudaErrorInvalidValue;
    kkd_update_kernel<<<(unsigned)((n + UPD_SPAN - 1) / UPD_SPAN), 256, 0, st>>>(b, alive, n, k,
                                                                                list, rd); note_launch();
    return cudaGetLastError();
}
cudaError_t round_launch_kk_cand2(const BufView& b, const uint8_t* alive, int64_t n, int S, int k,
                                  RoundDev* rd, uint8_t* inP, uint32_t* inPb, int* cand, int* fq,
                                  int* lq, u64* lam, int* src, u64* cmin, cudaStream_t st) {
    const unsigned g = (unsigned)((n + CAND_SPAN - 1) / CAND_SPAN);
    if (S == 8)
        kkd_cand2_kernel<true><<<g, 256, 0, st>>>(b, alive, n, S, k, rd, inP, inPb, cand, fq, lq,
                                                  lam, src, cmin);
    else
        kkd_cand2_kernel<false><<<g, 256, 0, st>>>(b, alive, n, S, k, rd, inP, inPb, cand, fq, lq,
                                                   lam, src, cmin);
    note_launch();
    return cudaGetLastError();
}
}  // namespace pd
