// knn.cu -- exact k-nearest-neighbour search and cost (Eq. 10 / Eq. 11).
//
// Two kernels share the search.  The full passes run a warp per leaf group
// (<= 32 query points of one octree leaf), one level, with 32-bit keys; what
// that cannot settle, and the scattered searches of the removal rounds, run a
// warp per query, level by level.  A level resolves the 3x3x3 cells around the
// query's in the hashed cell table and keeps the S smallest (d^2, tie) pairs
// over their points.  Squared distances are exact integers.  Exactness: every
// point outside the searched cube lies at least g from the query (g = distance
// to the cube's faces); when the bound that matters is below g^2 the query is
// done, otherwise the search repeats one level up (a cube of twice the size).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define FULLM 0xffffffffu

// Squared distance from the query to the outside of the level-L cube of
// cells [c-1, c+1]; ~0 when the cube holds the whole cloud.
__device__ inline u64 gap2(const GridView& g, int ux, int uy, int uz, int L, int cx, int cy,
                           int cz) {
    const int sh = L + g.shift;
    const int q[3] = {ux, uy, uz};
    const int c[3] = {cx, cy, cz};
    const int m[3] = {g.umax.x, g.umax.y, g.umax.z};
    int best = 0x7fffffff;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        // faces are below 2^25 + 2 * 2^25: ints
        const int lo = (c[a] - 1) * (1 << sh), hi = (c[a] + 2) * (1 << sh);
        if (lo > 0) best = min(best, q[a] - lo + 1);
        if (hi <= m[a]) best = min(best, hi - q[a]);
    }
    return best == 0x7fffffff ? ~0ull : (u64)((long long)best * best);
}

__device__ inline double nbr_weight(const KnnArgs& a, int q, int j) {
    return term_weight(a.term, a.weight, a.rgb, a.nrm, q, j);
}

// Pairs scanned, to this SM's slot.
__device__ __forceinline__ void add_pairs(const KnnArgs& a, uint32_t pairs) {
    unsigned smid;
    asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
    atomicAdd(&a.pairs_out[smid % PD_PAIR_SLOTS], (unsigned long long)pairs);
}

// ------------------------------------------------------------------ one warp per leaf group
// The full pass: a thread (or several) per query of a leaf group, one level.
// The candidates of the 27 cells get local numbers in Morton order, so that a
// candidate is one 32-bit key, d^2 << bits | number, and the sorted list is a
// chain of 32-bit minima and maxima: batches of candidates are sorted and merged
// by networks without branches.  The arithmetic bounds this kernel; the 64-bit
// (d^2, position) chain it replaces took 556 warp instructions per query.
// Measured, this kernel and the list's: 100M site points, k = 1, 61.8 -> 35.8 ms;
// 1.0M room points, k = 6, 2.20 -> 0.49; 2.0M, 17 stored, 9.19 -> 3.61 (4 to 6 blocks
// per SM, batches of 8 keys and 512 candidates all within 3 %: the arithmetic is
// the bound).
// Where the largest distance does not fit beside a candidate's number (cells of a
// metre and more: sparse clouds, far returns), the keys hold its leading bits: 24 of
// them with 8 bits of number, so two distances share a key about once in 10^5, and
// the exact ones order such a run.  Left to the warp-per-query kernel, those groups
// made the pass of a cloud with 1 m between its points slower than the chain had
// (1.0M points, grid and pass: k = 6 1.91 ms with the chain, 3.99 a warp each, 1.06
// now; k = 1 1.61, 3.54, 0.95; 17 stored 5.53, 5.06, 1.96).
// Weighted costs of 7 neighbours and more need the 17th entry in order too, hence two
// successors of the list's 16 (1.0M room points with colours, k = 7: 4.40 ms with the
// chain, 4.48 a warp each, 2.58 now; k = 16 6.17, 5.08, 4.12).
// What one level cannot settle goes to a list that the warp-per-query kernel
// finishes: the S-th distance beyond the cube's faces, more than NEAR_MAX
// candidates, equal distances at the end of a list whose order they decide (W),
// equal leading bits there.
#define NEAR_MAX 1024  // candidates of a group
#define NEAR_WARPS 8

__device__ __forceinline__ void key_cx(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}
__device__ __forceinline__ void key_sort(uint32_t (&c)[4]) {
    key_cx(c[0], c[1]);
    key_cx(c[2], c[3]);
    key_cx(c[0], c[2]);
    key_cx(c[1], c[3]);
    key_cx(c[1], c[2]);
}
// Batcher's odd-even merge sort of 8
__device__ __forceinline__ void key_sort(uint32_t (&c)[8]) {
    key_cx(c[0], c[1]);
    key_cx(c[2], c[3]);
    key_cx(c[4], c[5]);
    key_cx(c[6], c[7]);
    key_cx(c[0], c[2]);
    key_cx(c[1], c[3]);
    key_cx(c[4], c[6]);
    key_cx(c[5], c[7]);
    key_cx(c[1], c[2]);
    key_cx(c[5], c[6]);
    key_cx(c[0], c[4]);
    key_cx(c[1], c[5]);
    key_cx(c[2], c[6]);
    key_cx(c[3], c[7]);
    key_cx(c[2], c[4]);
    key_cx(c[3], c[5]);
    key_cx(c[1], c[2]);
    key_cx(c[3], c[4]);
    key_cx(c[5], c[6]);
}

// The E least keys, sorted, and the NX (0, 1, 2) least of all others.
template <int E, int NX>
struct NearList {
    uint32_t k[E], nx, nx2;
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int i = 0; i < E; i++) k[i] = ~0u;
        nx = nx2 = ~0u;
    }
    // a key at or above it changes nothing
    __device__ __forceinline__ uint32_t last() const {
        return NX == 2 ? nx2 : (NX == 1 ? nx : k[E - 1]);
    }
    __device__ __forceinline__ void pass(uint32_t v) {
        if (NX == 2) nx2 = min(nx2, max(nx, v));
        if (NX) nx = min(nx, v);
    }
    // takes NB sorted keys
    template <int NB>
    __device__ __forceinline__ void merge(const uint32_t (&c)[NB]) {
#pragma unroll
        for (int i = 0; i < NB; i++) {
            const uint32_t a = k[E - 1 - i];
            k[E - 1 - i] = min(a, c[i]);
            pass(max(a, c[i]));
        }
#pragma unroll
        for (int j = E / 2; j > 0; j >>= 1) {
#pragma unroll
            for (int i = 0; i < E; i++)
                if ((i & j) == 0) key_cx(k[i], k[i + j]);
        }
    }
    // the lists of lanes that share a query
    __device__ __forceinline__ void merge_lane(int off) {
        uint32_t c[E];
#pragma unroll
        for (int i = 0; i < E; i++) c[i] = __shfl_xor_sync(FULLM, k[i], off);
        const uint32_t o = NX ? __shfl_xor_sync(FULLM, nx, off) : ~0u;
        const uint32_t o2 = NX == 2 ? __shfl_xor_sync(FULLM, nx2, off) : ~0u;
        if (NX) pass(o);
        if (NX == 2) pass(o2);
        merge(c);
    }
};

struct NearSmem {
    int4 c[32];                 // this step's candidates: x, y, z, number
    uint32_t first[32];         // ranges laid end to end: prefix counts (the rest: total)
    uint32_t start[32], num[32];  // first position and first number
    int pos[NEAR_MAX];          // Morton position of every number seen
};

// The lanes' ranges [b, b + cnt) (numbers from num on) against every query.
template <int E, int NX, int NB, bool WIDE>
__device__ __forceinline__ void near_scan(const GridView& g, const KnnArgs& a, NearSmem& sm,
                                          NearList<E, NX>& top, uint32_t b, uint32_t cnt,
                                          uint32_t num, int4 qp, uint32_t self, int bits, int cut,
                                          int sub, int lpq, int lane) {
    const unsigned act = __ballot_sync(FULLM, cnt > 0);
    if (!act) return;
    const uint32_t inc = warp_inclusive(cnt, lane);
    const uint32_t total = __shfl_sync(FULLM, inc, 31);
    __syncwarp();
    sm.first[lane] = total;
    __syncwarp();
    if (cnt) {
        const int at = __popc(act & ((1u << lane) - 1u));
        sm.first[at] = inc - cnt;
        sm.start[at] = b;
        sm.num[at] = num;
    }
    __syncwarp();
    int r = 0;
    uint32_t t = lane;
    int4 v = make_int4(0, 0, 0, 0);
    uint32_t j = 0, id = 0;
    bool ok = false;
    auto load = [&]() {  // t ascends from call to call
        ok = t < total;
        if (ok) {
            while (r < 31 && t >= sm.first[r + 1]) r++;
            const uint32_t o = t - sm.first[r];
            j = sm.start[r] + o;
            id = sm.num[r] + o;
            v = g.pos[j];
            if (a.alive) ok = a.alive[j];
        }
    };
    load();
    for (uint32_t base = 0; base < total; base += 32) {  // warp-uniform
        const unsigned in = __ballot_sync(FULLM, ok);
        if (ok) {
            const int at = __popc(in & ((1u << lane) - 1u));
            sm.c[at] = make_int4(v.x, v.y, v.z, (int)id);
            sm.pos[id] = (int)j;
        }
        __syncwarp();
        t += 32;
        load();
        const int m = __popc(in);
        for (int c0 = sub; c0 - sub < m; c0 += NB * lpq) {  // warp-uniform
            uint32_t key[NB];
#pragma unroll
            for (int u = 0; u < NB; u++) {
                const int i = c0 + u * lpq;
                const int4 c = sm.c[i & 31];
                const int dx = c.x - qp.x, dy = c.y - qp.y, dz = c.z - qp.z;
                const uint32_t d2 =
                    WIDE ? (uint32_t)(((u64)((long long)dx * dx) + (u64)((long long)dy * dy) +
                                       (u64)((long long)dz * dz)) >> cut)
                         : (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
                const bool skip = i >= m || (uint32_t)c.w == self;
                key[u] = skip ? ~0u : (d2 << bits) | (uint32_t)c.w;
            }
            uint32_t least = key[0];
#pragma unroll
            for (int u = 1; u < NB; u++) least = min(least, key[u]);
            if (__any_sync(FULLM, least < top.last())) {
                key_sort(key);
                top.merge(key);
            }
        }
        __syncwarp();
    }
}

// A leaf group's queries on the lanes of one warp.
struct NearGroup {
    int4 qp;                // this lane's query (an idle lane: the first one's)
    int q, nq, sub, lpq;    // its position (-1: idle); queries; lane `sub` of its `lpq`
    int ux, uy, uz, L;
    WarpNode n;             // this lane's cell
    uint32_t num, self;     // number of the cell's first candidate; the query's own
    u64 gbox;               // squared distance from the cell to the box of the queries
    int bits, cut;          // of a key: its number's bits, distance bits left out
};

// The search of a group's queries.  Returns the lane's query when it is left to
// the warp-per-query kernel, -1 otherwise.
// WIDE: the keys hold d^2 >> cut, so the S nearest are known where the next key's
// distance bits differ from the last one's, and their order from their positions.
// W: equal distances in the order of the input index (1: of the first 8 or 16,
// 2: of all S, which a weighted cost of 7 neighbours or more needs).
template <int S, int W, bool WIDE>
__device__ __forceinline__ int near_search(const GridView& g, const KnnArgs& a, NearSmem& sm,
                                           const NearGroup& G, int lane) {
    const int E = S == 8 ? 8 : 16, NB = S == 8 ? 4 : 8;
    const int T = W == 2 ? S : E;  // entries in order with W
    const int NX = WIDE ? S - E + 1 : (W ? T - E + 1 : S - E);
    const int bits = G.bits, cut = WIDE ? G.cut : 0, q = G.q;
    const bool on = q >= 0;
    const int4 qp = G.qp;
    const uint32_t cnt = G.n.count(), self = on ? G.self : ~0u;
    NearList<E, NX> top;
    top.init();
    // the cell and its face neighbours first; the other cells only where they
    // reach the largest S-th distance of the group
    near_scan<E, NX, NB, WIDE>(g, a, sm, top, G.n.b, lane < 7 ? cnt : 0, G.num, qp, self, bits,
                               cut, G.sub, G.lpq, lane);
    {
        uint32_t far = top.last();  // partial lists bound the merged one
        if (!on) far = 0;
        far = __reduce_max_sync(FULLM, far);
        const u64 bound = far == ~0u ? ~0ull : ((u64)((far >> bits) + 1) << cut) - 1;
        near_scan<E, NX, NB, WIDE>(g, a, sm, top, G.n.b, lane >= 7 && G.gbox <= bound ? cnt : 0,
                                   G.num, qp, self, bits, cut, G.sub, G.lpq, lane);
        if (a.pairs_out) {
            const uint32_t mine = lane < 7 || G.gbox <= bound ? cnt : 0;
            const uint32_t pairs = __reduce_add_sync(FULLM, mine) * (uint32_t)G.nq;
            if (lane == 0) add_pairs(a, pairs);
        }
    }
    for (int off = G.lpq >> 1; off >= 1; off >>= 1) top.merge_lane(off);
    if (!on || G.sub) return -1;
    // the S nearest: key i, and past the list its successor
    auto key = [&](int i) -> uint32_t { return i < E ? top.k[i < E ? i : 0] : top.nx; };
    auto same = [&](uint32_t x, uint32_t y) { return y != ~0u && x >> bits == y >> bits; };
    if (WIDE && same(key(S - 1), top.last())) return q;
    int id[S], ix[S];
    u64 wd[S];  // WIDE: exact distances
    int found = 0;
#pragma unroll
    for (int i = 0; i < S; i++) {
        const bool has = key(i) != ~0u;
        found += has;
        id[i] = has ? sm.pos[key(i) & ((1u << bits) - 1u)] : -1;
        if (WIDE) {
            const int4 v = g.pos[has ? id[i] : 0];
            wd[i] = has ? sqd(v, qp) : ~0ull;
            ix[i] = W ? v.w : id[i];
        }
    }
    if (WIDE) {
        // (distance, tie) within a run of equal keys
        bool again = true;
        while (again) {
            again = false;
#pragma unroll
            for (int i = 0; i + 1 < S; i++) {
                const bool sw = wd[i] > wd[i + 1] ||
                                (wd[i] == wd[i + 1] && wd[i] != ~0ull && ix[i] > ix[i + 1]);
                const u64 d = wd[i];
                const int x = ix[i], y = id[i];
                wd[i] = sw ? wd[i + 1] : d;
                ix[i] = sw ? ix[i + 1] : x;
                id[i] = sw ? id[i + 1] : y;
                wd[i + 1] = sw ? d : wd[i + 1];
                ix[i + 1] = sw ? x : ix[i + 1];
                id[i + 1] = sw ? y : id[i + 1];
                again = again || sw;
            }
        }
    }
    auto dist = [&](int i) -> u64 {
        return WIDE ? wd[i] : (key(i) == ~0u ? ~0ull : (u64)(key(i) >> bits));
    };
    const int R = a.r_exact > 0 && a.r_exact < S ? a.r_exact : S;
    const int sh = G.L + g.shift;
    const u64 gg = G.L >= g.B ? ~0ull
                              : gap2(g, G.ux, G.uy, G.uz, G.L, G.ux >> sh, G.uy >> sh, G.uz >> sh);
    u64 bound = 0;
#pragma unroll
    for (int i = 0; i < S; i++)
        if (i == R - 1) bound = dist(i);
    if (!(gg == ~0ull || bound < gg)) return q;
    if (!WIDE && W) {
        if (same(key(T - 1), T > E ? top.nx2 : top.nx)) return q;
        // equal distances in the order of the input index
        bool tie = false;
#pragma unroll
        for (int i = 0; i + 1 < T; i++) tie = tie || same(key(i), key(i + 1));
        if (tie) {
#pragma unroll
            for (int i = 0; i < T; i++) ix[i] = id[i] >= 0 ? g.pos[id[i]].w : 0x7fffffff;
            while (tie) {
                tie = false;
#pragma unroll
                for (int i = 0; i + 1 < T; i++) {
                    if (key(i) >> bits == key(i + 1) >> bits && ix[i] > ix[i + 1]) {
                        const int x = ix[i], y = id[i];
                        ix[i] = ix[i + 1];
                        id[i] = id[i + 1];
                        ix[i + 1] = x;
                        id[i + 1] = y;
                        tie = true;
                    }
                }
            }
        }
    }
    // results of the query
    if (S == 8) {
        store_nbr8(a.nbr, q, reinterpret_cast<int(&)[8]>(id));
    } else {
#pragma unroll
        for (int i = 0; i < S; i++) a.nbr[(int64_t)q * S + i] = id[i];
    }
    const u64 ds = dist(S - 1);
    if (a.density_k1) {
        // all S nearest are stored (the k+b buffer); the shell is the prefix at
        // the nearest distance d0, its size kept in flg >> 2
        const u64 d0 = dist(0);
        int shell = 0;
#pragma unroll
        for (int i = 0; i < E; i++) shell += dist(i) != ~0ull && dist(i) == d0;
        if (!W && a.nbr0_out) a.nbr0_out[q] = id[0];
        a.prim_out[q] = key_prim_d2(d0);
        a.rk2_out[q] = d0;
        a.flg_out[q] = (uint8_t)((shell >= 2 ? 1 : 0) | (shell == S ? 2 : 0) | (shell << 2));
        // the cells passed over lie beyond the S-th distance
        if (a.hz_out) a.hz_out[q] = gg < ds ? gg : ds;
        if (a.cost_out) a.cost_out[q] = d0 == ~0ull ? 0.0 : __ddiv_rn(1.0, (double)d0);
        return -1;
    }
    double c = 0.0;
    u64 dk = ~0ull, dn = ~0ull;
#pragma unroll
    for (int i = 0; i < S; i++) {
        const u64 d = dist(i);
        if (i < E && i < a.k && id[i] >= 0)
            c = __dadd_rn(c, __ddiv_rn(nbr_weight(a, q, id[i]), (double)d));
        if (i == a.k - 1) dk = d;
        if (i == a.k) dn = d;
    }
    a.prim_out[q] = key_prim_cost(c);
    a.rk2_out[q] = dk;
    a.flg_out[q] = (uint8_t)(found > a.k && dn == dk ? 1 : 0);
    if (a.hz_out) a.hz_out[q] = ds;
    if (a.cost_out) a.cost_out[q] = c;
    return -1;
}

// One leaf group (<= 32 queries) for one warp: sets the search up.
template <int S, int W>
__device__ __forceinline__ int near_group(const GridView& g, const KnnArgs& a, int gid,
                                          NearSmem& sm, int lane) {
    const int4 gr = a.groups[gid];
    NearGroup G;
    G.L = gr.z;
    int q = -1;
    if (lane < gr.y) {
        q = gr.x + lane;
        if (a.qflag && !a.qflag[q]) q = -1;
    }
    // the active queries packed onto the lanes: each gets lpq of them (a power
    // of two), which share the candidates and merge their lists
    const unsigned act = __ballot_sync(FULLM, q >= 0);
    if (!act) return -1;
    G.nq = __popc(act);
    int lpq = 32;
    while (G.nq * lpq > 32) lpq >>= 1;
    const int qi = lane / lpq;
    G.lpq = lpq;
    G.sub = lane - qi * lpq;
    {
        const int src = qi < G.nq ? (int)__fns(act, 0, qi + 1) : 0;
        const int qq = __shfl_sync(FULLM, q, src);
        q = qi < G.nq ? qq : -1;
    }
    G.q = q;
    // idle lanes follow the first query (its box and its bound)
    const int q0 = __shfl_sync(FULLM, q, 0);
    G.qp = g.pos[q >= 0 ? q : q0];
    G.ux = G.qp.x - g.origin.x;
    G.uy = G.qp.y - g.origin.y;
    G.uz = G.qp.z - g.origin.z;
    G.n = warp_cells(g, G.L, g.code[gr.x], G.ux, G.uy, G.uz, lane);
    const uint32_t cnt = G.n.count();
    // numbers in Morton order: candidates of the ranges that start before this one
    uint32_t num = 0, total = 0;
    for (int i = 0; i < 27; i++) {
        const uint32_t bi = __shfl_sync(FULLM, G.n.b, i), ci = __shfl_sync(FULLM, cnt, i);
        if (bi < G.n.b) num += ci;
        total += ci;
    }
    G.num = num;
    int bits = 1;
    while ((1u << bits) < total) bits++;
    G.bits = bits;
    // d^2 < 12 * 4^(widest cell), two of its edges per axis: what of it does not fit
    // beside the number
    const int edge = __reduce_max_sync(FULLM, cnt > 0 ? G.n.lv + g.shift : 0);
    G.cut = 2 * edge + bits - 28;
    if (total > NEAR_MAX) return G.sub == 0 ? q : -1;
    // the query's own number: its cell is lane 0's
    G.self = __shfl_sync(FULLM, num, 0) + (uint32_t)(q - (int)__shfl_sync(FULLM, G.n.b, 0));
    // squared distance from this lane's cell to the box of the group's queries
    {
        const int sh = G.n.lv + g.shift;
        const int u[3] = {G.ux, G.uy, G.uz}, c[3] = {G.n.x, G.n.y, G.n.z};
        G.gbox = 0;
#pragma unroll
        for (int x = 0; x < 3; x++) {
            const int lo = __reduce_min_sync(FULLM, u[x]), hi = __reduce_max_sync(FULLM, u[x]);
            const int cl = c[x] << sh, ch = cl + ((1 << sh) - 1);
            const int d = max(max(cl - hi, lo - ch), 0);
            G.gbox += (u64)((long long)d * d);
        }
    }
    return G.cut > 0 ? near_search<S, W, true>(g, a, sm, G, lane)
                     : near_search<S, W, false>(g, a, sm, G, lane);
}

template <int S, int W>
__global__ void __launch_bounds__(NEAR_WARPS * 32, S == 8 ? 4 : 2)
    knn_kernel(GridView g, KnnArgs a, int* rest, int* nrest) {
    chain();
    __shared__ NearSmem s_m[NEAR_WARPS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gid = blockIdx.x * NEAR_WARPS + w;
    const int q = gid < a.ngroups ? near_group<S, W>(g, a, gid, s_m[w], lane) : -1;
    const int slot = block_append(q >= 0, nrest);
    if (q >= 0) rest[slot] = q;
}

// ------------------------------------------------------------------ one warp per query
// The searches of the removal rounds: re-searches of points that lost too
// many stored neighbours, and the filtered searches of the candidate and
// danger tests.  A round has few of them, scattered over the cloud, so a
// round's search time is the latency of one query's chain of dependent loads,
// not the arithmetic: one warp serves one query.  Lanes 0..26 resolve the 27
// cells at once, the non-empty ranges are laid end to end, and every lane
// takes every 32nd candidate of that sequence, the next step's loads issued
// before this step's are used.  The 32 nearest so far are kept sorted across
// the lanes (lane i holds the i-th); a step's candidates below the S-th are
// inserted one by one, or, when there are many (the first step), sorted
// (bitonic) and merged.  Measured against the kernels it replaces (k = 1: 2
// lanes per query walking the ranges in turn; otherwise a warp per leaf group
// with a flagged point), all rounds of one decimation: 9.8M outdoor points,
// k = 4, re-searches 114 -> 16 ms, filtered and lambda searches 116 -> 18.6 ms;
// 100M site points, k = 1, 41.2 -> 33.7 ms; 200k room points, k = 1, 1.51 -> 0.25 ms.
template <bool PACK>
struct WarpKey {  // (d^2, tie), ordered; PACK: d^2 < 2^32, both in one word
    u64 d;
    uint32_t t;
    __device__ __forceinline__ static WarpKey make(u64 dd, uint32_t tie) {
        WarpKey k;
        k.d = PACK ? (dd << 32) | tie : dd;
        k.t = tie;
        return k;
    }
    __device__ __forceinline__ static WarpKey none() {
        WarpKey k;
        k.d = ~0ull;
        k.t = 0xffffffffu;
        return k;
    }
    __device__ __forceinline__ bool less(const WarpKey& o) const {
        return PACK ? d < o.d : (d < o.d || (d == o.d && t < o.t));
    }
    __device__ __forceinline__ bool has() const { return d != ~0ull; }
    __device__ __forceinline__ u64 dist() const { return PACK && has() ? d >> 32 : d; }
    __device__ __forceinline__ uint32_t tie() const { return PACK ? (uint32_t)d : t; }
    __device__ __forceinline__ WarpKey from(int src) const {
        WarpKey k;
        k.d = __shfl_sync(FULLM, d, src);
        k.t = PACK ? 0u : __shfl_sync(FULLM, t, src);
        return k;
    }
    __device__ __forceinline__ WarpKey across(int mask) const {
        WarpKey k;
        k.d = __shfl_xor_sync(FULLM, d, mask);
        k.t = PACK ? 0u : __shfl_xor_sync(FULLM, t, mask);
        return k;
    }
    __device__ __forceinline__ WarpKey before() const {
        WarpKey k;
        k.d = __shfl_up_sync(FULLM, d, 1);
        k.t = PACK ? 0u : __shfl_up_sync(FULLM, t, 1);
        return k;
    }
};

// A candidate's fields, loaded ahead of their use.
struct WarpLoad {
    int4 v;
    u64 key;
    uint8_t live;
};
// Whether it counts: live, not the query itself, below the threshold in a
// filtered search.
template <int FILT>
__device__ __forceinline__ bool warp_counts(const WarpLoad& c, uint32_t j, int q, u64 tp, int ti) {
    const bool ok = c.live && (int)j != q;
    return FILT == FILT_NONE ? ok : ok && key_gt(tp, ti, c.key, c.v.w);
}

// The 32 nearest so far, sorted across the lanes, in the order (d^2, tie): the
// tie is the input index with W, the Morton position otherwise.  More
// candidates than SORT_AT in one step are sorted and merged (about 170
// instructions) rather than inserted one by one (about 12 each).
template <bool W, bool PACK>
struct WarpList {
    static const int SORT_AT = 12;
    WarpKey<PACK> best, last, cap;  // last: the least of cap and the S-th key
    int bpid;
    // cap_d, cap_t: no key above this one is wanted (cap_d ~0: no cap); cap_t is
    // below 0xffffffff
    __device__ __forceinline__ void init(u64 cap_d, uint32_t cap_t) {
        best = WarpKey<PACK>::none();
        cap = best;
        if (cap_d != ~0ull) {
            cap = WarpKey<PACK>::make(cap_d, cap_t);
            if (PACK) cap.d++;
            else cap.t++;
        }
        last = cap;
        bpid = -1;
    }
    __device__ __forceinline__ u64 bound() const { return last.dist(); }
    __device__ __forceinline__ u64 dist() const { return best.dist(); }
    __device__ __forceinline__ bool has() const { return best.has(); }
    __device__ __forceinline__ int id() const { return W ? bpid : (int)best.tie(); }
    __device__ __forceinline__ uint32_t tie() const { return best.tie(); }
    __device__ __forceinline__ void take(bool ok, const int4& v, uint32_t j, const int4& qp, int S,
                                         int lane) {
        u64 dd;
        if (PACK) {
            const int dx = v.x - qp.x, dy = v.y - qp.y, dz = v.z - qp.z;
            dd = (u64)((uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz));
        } else {
            dd = sqd(v, qp);
        }
        WarpKey<PACK> c =
            ok ? WarpKey<PACK>::make(dd, W ? (uint32_t)v.w : j) : WarpKey<PACK>::none();
        int cpid = (int)j;
        unsigned m = __ballot_sync(FULLM, c.less(last));
        if (!m) return;
        if (__popc(m) > SORT_AT) {
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int i = k >> 1; i > 0; i >>= 1) {
                    const WarpKey<PACK> o = c.across(i);
                    const int op = W ? __shfl_xor_sync(FULLM, cpid, i) : 0;
                    const bool low = ((lane & k) == 0) == ((lane & i) == 0);
                    const bool sw = low ? o.less(c) : c.less(o);
                    c = sw ? o : c;
                    if (W) cpid = sw ? op : cpid;
                }
            }
            {   // the 32 least of both lists, a bitonic sequence
                const WarpKey<PACK> o = c.across(31);
                const int op = W ? __shfl_xor_sync(FULLM, cpid, 31) : 0;
                const bool sw = o.less(best);
                best = sw ? o : best;
                if (W) bpid = sw ? op : bpid;
            }
#pragma unroll
            for (int i = 16; i > 0; i >>= 1) {
                const WarpKey<PACK> o = best.across(i);
                const int op = W ? __shfl_xor_sync(FULLM, bpid, i) : 0;
                const bool sw = (lane & i) == 0 ? o.less(best) : best.less(o);
                best = sw ? o : best;
                if (W) bpid = sw ? op : bpid;
            }
        } else {
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const WarpKey<PACK> k = c.from(src);
                const int kp = W ? __shfl_sync(FULLM, cpid, src) : 0;
                const WarpKey<PACK> prev = best.before();
                const int pp = W ? __shfl_up_sync(FULLM, bpid, 1) : 0;
                if (k.less(best)) {
                    const bool here = lane == 0 || !k.less(prev);
                    best = here ? k : prev;
                    if (W) bpid = here ? kp : pp;
                }
            }
        }
        last = best.from(S - 1);
        if (cap.less(last)) last = cap;
    }
};

// The same without an order among equal distances (a density cost does not
// depend on it: whichever of several equally far points is stored, the others
// lie at the horizon), for levels with d^2 < 2^27: a step is sorted as one
// 32-bit key per lane (d^2 << 5 | lane), a third of the instructions, and the
// positions follow from the lane.
struct WarpList32 {
    static const int SORT_AT = 6;
    uint32_t best, last, cap;
    int bid;
    __device__ __forceinline__ void init(u64 cap_d, uint32_t) {
        best = ~0u;
        bid = -1;
        cap = cap_d < (1u << 27) ? (uint32_t)cap_d + 1 : ~0u;
        last = cap;
    }
    __device__ __forceinline__ u64 bound() const { return last == ~0u ? ~0ull : last; }
    __device__ __forceinline__ u64 dist() const { return best == ~0u ? ~0ull : best; }
    __device__ __forceinline__ bool has() const { return best != ~0u; }
    __device__ __forceinline__ int id() const { return bid; }
    // as a later level's cap: every key at this distance is wanted
    __device__ __forceinline__ uint32_t tie() const { return 0xfffffffeu; }
    __device__ __forceinline__ void merge(int o_, int lane) {
        const uint32_t o = __shfl_xor_sync(FULLM, best, o_);
        const int oi = __shfl_xor_sync(FULLM, bid, o_);
        const bool sw = (lane & o_) == 0 ? o < best : best < o;
        best = sw ? o : best;
        bid = sw ? oi : bid;
    }
    __device__ __forceinline__ void take(bool ok, const int4& v, uint32_t j, const int4& qp, int S,
                                         int lane) {
        const int dx = v.x - qp.x, dy = v.y - qp.y, dz = v.z - qp.z;
        const uint32_t dd = (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
        const bool in = ok && dd < last;
        unsigned m = __ballot_sync(FULLM, in);
        if (!m) return;
        if (__popc(m) > SORT_AT) {
            uint32_t key = in ? (dd << 5) | lane : ~0u;
#pragma unroll
            for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                for (int i = k >> 1; i > 0; i >>= 1) {
                    const uint32_t o = __shfl_xor_sync(FULLM, key, i);
                    const bool low = ((lane & k) == 0) == ((lane & i) == 0);
                    key = low ? min(key, o) : max(key, o);
                }
            }
            uint32_t d = key == ~0u ? ~0u : key >> 5;
            int id = __shfl_sync(FULLM, (int)j, (int)(key & 31));
            if (__shfl_sync(FULLM, best, 0) == ~0u) {  // the first points
                best = d;
                bid = id;
            } else {
                // the least of both lists, a bitonic sequence (8 or 32 lanes of it)
                const int f = S <= 8 ? 7 : 31;
                d = __shfl_xor_sync(FULLM, d, f);
                id = __shfl_xor_sync(FULLM, id, f);
                const bool sw = d < best;
                best = sw ? d : best;
                bid = sw ? id : bid;
                if (S > 8) {
                    merge(16, lane);
                    merge(8, lane);
                }
                merge(4, lane);
                merge(2, lane);
                merge(1, lane);
            }
        } else {
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const uint32_t k = __shfl_sync(FULLM, dd, src);
                const int kid = __shfl_sync(FULLM, (int)j, src);
                const uint32_t prev = __shfl_up_sync(FULLM, best, 1);
                const int pid = __shfl_up_sync(FULLM, bid, 1);
                if (k < best) {
                    const bool here = lane == 0 || k >= prev;
                    best = here ? k : prev;
                    bid = here ? kid : pid;
                }
            }
        }
        last = min(cap, __shfl_sync(FULLM, best, S - 1));
    }
};

struct WarpRanges {  // non-empty ranges laid end to end
    uint32_t first[33];  // prefix counts
    uint32_t start[32];
    uint32_t pairs;      // candidates of the query so far (where a.pairs_out asks)
};

template <int FILT>
__device__ __forceinline__ WarpLoad warp_load(const GridView& g, const KnnArgs& a, bool in,
                                              uint32_t j) {
    WarpLoad c;
    c.v = make_int4(0, 0, 0, 0);
    c.key = 0;
    c.live = 0;
    if (in) {
        c.v = g.pos[j];
        c.live = a.alive ? a.alive[j] : 1;
        if (FILT != FILT_NONE) c.key = a.prim[j];
    }
    return c;
}
// Nodes of at most this many points are scanned; larger ones are entered by
// their children, nearest box first, and only where the box reaches the S-th
// distance so far: a sparse point next to a dense region (far returns, scan
// edges) would otherwise read the whole region.  Filtered searches scan up to
// the second limit, 1024 positions a step, by the chunks' least keys.
#define WARP_SCAN 64
#define WARP_SCAN_FILT 2048

// The 32 nearest so far of one warp's query and how candidates join them.
template <int FILT, class List>
struct WarpSearch {
    const GridView& g;
    const KnnArgs& a;
    const int q, S, lane;
    const int4 qp;
    const u64 tp;
    const int ti;
    WarpRanges& wr;
    List top;

    __device__ __forceinline__ WarpSearch(const GridView& g_, const KnnArgs& a_, int q_, int S_,
                                          int lane_, int4 qp_, u64 tp_, int ti_, WarpRanges& wr_)
        : g(g_), a(a_), q(q_), S(S_), lane(lane_), qp(qp_), tp(tp_), ti(ti_), wr(wr_) {}
    __device__ __forceinline__ void take(const WarpLoad& c, uint32_t j) {
        top.take(warp_counts<FILT>(c, j, q, tp, ti), c.v, j, qp, S, lane);
    }
    // the lanes' ranges [b, b + cnt), laid end to end
    __device__ __forceinline__ void scan(uint32_t b, uint32_t cnt) {
        const unsigned act = __ballot_sync(FULLM, cnt > 0);
        if (!act) return;
        const uint32_t inc = warp_inclusive(cnt, lane);
        const uint32_t total = __shfl_sync(FULLM, inc, 31);
        __syncwarp();  // the previous scan's readers are done
        if (cnt) {
            const int at = __popc(act & ((1u << lane) - 1u));
            wr.first[at] = inc - cnt;
            wr.start[at] = b;
        }
        if (lane == 0) wr.first[__popc(act)] = total;
        if (FILT == FILT_NONE && a.pairs_out && lane == 0) wr.pairs += total;
        __syncwarp();
        int r = 0;
        uint32_t t = lane;
        auto place = [&](uint32_t x) -> uint32_t {  // x ascends from call to call
            while (x >= wr.first[r + 1]) r++;
            return wr.start[r] + (x - wr.first[r]);
        };
        uint32_t jn = t < total ? place(t) : 0;
        WarpLoad next = warp_load<FILT>(g, a, t < total, jn);
        for (uint32_t base = 0; base < total; base += 32) {  // warp-uniform
            const WarpLoad cur = next;
            const uint32_t j = jn;
            t += 32;
            jn = t < total ? place(t) : 0;
            next = warp_load<FILT>(g, a, t < total, jn);
            take(cur, j);
        }
    }
    // one long range, the chunks of 32 without a key below the threshold skipped
    __device__ __forceinline__ void scan_chunks(uint32_t b, uint32_t e) {
        for (uint32_t c0 = b >> 5; c0 <= (e - 1) >> 5; c0 += 32) {
            const uint32_t ch = c0 + lane;
            unsigned m = __ballot_sync(FULLM, ch <= (e - 1) >> 5 && a.cmin[ch] <= tp);
            while (m) {
                const uint32_t j = (c0 + (uint32_t)__ffs(m) - 1) * 32 + lane;
                m &= m - 1;
                take(warp_load<FILT>(g, a, j >= b && j < e, j), j);
            }
        }
    }
    // the points of the lanes' nodes (put: which lanes hold one to scan now)
    __device__ __forceinline__ void scan_nodes(const WarpNode& n, bool put) {
        const uint32_t cnt = put ? n.count() : 0;
        if (FILT == FILT_NONE) {
            scan(n.b, cnt);
        } else {
            scan(n.b, cnt <= WARP_SCAN ? cnt : 0);
            unsigned m = __ballot_sync(FULLM, cnt > WARP_SCAN);
            while (m) {
                const int src = __ffs(m) - 1;
                m &= m - 1;
                const u64 bx = __shfl_sync(FULLM, n.box, src);
                if (bx > top.bound()) continue;
                scan_chunks(__shfl_sync(FULLM, n.b, src), __shfl_sync(FULLM, n.e, src));
            }
        }
    }
    // every candidate of the cells in n that can be among the S nearest
    __device__ __forceinline__ void search(WarpNode n, int ux, int uy, int uz) {
        const uint32_t lim = FILT == FILT_NONE ? WARP_SCAN : WARP_SCAN_FILT;
        bool held = n.count() > lim && n.lv > 0;
        // the cell and its face neighbours first; their S-th distance then rules
        // out most of the edge and corner cells
        bool now = !held && n.count() > 0;
        scan_nodes(n, now && lane < 7);
        now = now && lane >= 7 && n.box <= top.bound();
        scan_nodes(n, now);
        for (;;) {
            held = held && n.box <= top.bound();
            u64 near = held ? (n.box << 5) | lane : ~0ull;  // box < 2^52
            if (__all_sync(FULLM, near == ~0ull)) break;
            for (int o = 16; o; o >>= 1) {
                const u64 v = __shfl_xor_sync(FULLM, near, o);
                near = v < near ? v : near;
            }
            const int src = (int)(near & 31);
            const WarpNode c = warp_children(g, n, src, ux, uy, uz, lane);
            if (lane == src) held = false;
            now = c.count() > 0 && c.box <= top.bound();
            bool keep = now && c.count() > lim && c.lv > 0;
            const bool was = keep;
            warp_keep(n, held, c, keep, lane);
            if (was && !keep) now = false;  // kept for later; no room: scanned now
            scan_nodes(c, now);
        }
    }
};

// One search level of one query; returns true when its R nearest are exact.
template <int FILT, bool W, class List>
__device__ __forceinline__ bool warp_level(const GridView& g, const KnnArgs& a, int q, int4 qp,
                                           int S, int R, u64 tp, int ti, WarpRanges& wr,
                                           const WarpNode& n, int ux, int uy, int uz, u64 gg,
                                           u64& cap_d, uint32_t& cap_t, int lane) {
    WarpSearch<FILT, List> ws(g, a, q, S, lane, qp, tp, ti, wr);
    ws.top.init(cap_d, cap_t);
    ws.search(n, ux, uy, uz);
    const List& top = ws.top;
    const u64 dl = top.dist();
    const u64 bound = __shfl_sync(FULLM, dl, R - 1);
    if (!(gg == ~0ull || bound < gg)) {
        cap_d = __shfl_sync(FULLM, dl, S - 1);
        cap_t = __shfl_sync(FULLM, top.tie(), S - 1);
        return false;
    }
    // lane i holds the i-th nearest
    const bool has = top.has() && lane < S;
    const u64 d = has ? dl : ~0ull;
    const int id = has ? top.id() : -1;
    const int found = __popc(__ballot_sync(FULLM, has));
    if (FILT == FILT_BELOW_TAU) {
        if (lane == 0) a.lam_out[q] = bound;  // R = k
        return true;
    }
    if (FILT == FILT_NONE && lane < S) a.nbr[(int64_t)q * S + lane] = id;
    if (FILT == FILT_NONE && a.density_k1) {
        const u64 d0 = __shfl_sync(FULLM, d, 0), ds = __shfl_sync(FULLM, d, S - 1);
        const int shell = __popc(__ballot_sync(FULLM, has && d == d0));
        if (lane == 0) {
            if (!W && a.nbr0_out) a.nbr0_out[q] = id;
            a.prim_out[q] = key_prim_d2(d0);
            a.rk2_out[q] = d0;
            a.flg_out[q] = (uint8_t)((shell >= 2 ? 1 : 0) | (shell == S ? 2 : 0) | (shell << 2));
            // every live point closer than the cube's faces and the S-th was seen
            if (a.hz_out) a.hz_out[q] = gg < ds ? gg : ds;
            if (a.cost_out) a.cost_out[q] = d0 == ~0ull ? 0.0 : __ddiv_rn(1.0, (double)d0);
        }
        return true;
    }
    // the terms side by side, the sum in order (each operation rounded)
    const double term =
        has && lane < a.k ? __ddiv_rn(nbr_weight(a, q, id), (double)d) : 0.0;
    double c = 0.0;
    for (int i = 0; i < a.k && i < found; i++) c = __dadd_rn(c, __shfl_sync(FULLM, term, i));
    const u64 prim = key_prim_cost(c);
    if (FILT == FILT_BELOW_SELF) {
        // condition (A): the cost over the smaller keys is the cost itself
        if (lane == 0 && prim == a.prim[q]) {
            a.inP[q] = 1;
            atomicOr(&a.inPb[q >> 5], 1u << (q & 31));
            a.cand[atomicAdd(a.ncand, 1)] = q;
        }
        return true;
    }
    const u64 dk = __shfl_sync(FULLM, d, a.k - 1);
    const u64 dn = __shfl_sync(FULLM, d, a.k), ds = __shfl_sync(FULLM, d, S - 1);
    if (lane == 0) {
        a.prim_out[q] = prim;
        a.rk2_out[q] = dk;
        a.flg_out[q] = (uint8_t)(found > a.k && dn == dk ? 1 : 0);
        if (a.hz_out) a.hz_out[q] = ds;
        if (a.cost_out) a.cost_out[q] = c;
    }
    return true;
}

// The list of a level whose distances fit 32 bits (27 if unordered).
template <bool W, bool ORDER>
struct WarpLists {
    typedef WarpList<W, true> Near;
};
template <>
struct WarpLists<false, false> {
    typedef WarpList32 Near;
};

template <int FILT, bool W, bool ORDER>
__device__ __forceinline__ void warp_query(const GridView& g, const KnnArgs& a, int q,
                                           WarpRanges& wr, int lane) {
    const int4 qp = g.pos[q];
    const u64 c0 = g.code[q];
    int L = g.leaf[q];
    const int S = FILT == FILT_NONE ? a.S : a.k;
    const int R = FILT == FILT_NONE && a.r_exact > 0 && a.r_exact < S ? a.r_exact : S;
    const int ux = qp.x - g.origin.x, uy = qp.y - g.origin.y, uz = qp.z - g.origin.z;
    u64 tp = 0;
    int ti = 0;
    if (FILT == FILT_BELOW_SELF) {
        tp = a.prim[q];
        ti = qp.w;
    } else if (FILT == FILT_BELOW_TAU) {
        round_tau(a.rd, qp, tp, ti);  // packed batch: the query's own scan's
        // fewer than k lower keys are stored, and every live point closer than
        // the horizon is: start where the cell edge reaches it
        const u64 h = a.hz_out[q];
        if (h != ~0ull)
            while (L < g.B && (1ull << (2 * (L + g.shift))) < h) L++;
    }
    u64 cap_d = ~0ull;  // the S-th key found so far bounds the next level's search
    uint32_t cap_t = 0;
    if (FILT == FILT_NONE && lane == 0) wr.pairs = 0;
    for (;; L++) {
        const WarpNode n = warp_cells(g, L, c0, ux, uy, uz, lane);
        const int sh = L + g.shift;
        const u64 gg = L >= g.B ? ~0ull : gap2(g, ux, uy, uz, L, ux >> sh, uy >> sh, uz >> sh);
        // every coordinate difference is below 3 cells: d^2 < 27 * 4^(level)
        const bool near = __all_sync(FULLM, n.lv + g.shift <= (ORDER ? 13 : 11));
        const bool done =
            near ? warp_level<FILT, W, typename WarpLists<W, ORDER>::Near>(
                       g, a, q, qp, S, R, tp, ti, wr, n, ux, uy, uz, gg, cap_d, cap_t, lane)
                 : warp_level<FILT, W, WarpList<W, false>>(g, a, q, qp, S, R, tp, ti, wr, n, ux,
                                                           uy, uz, gg, cap_d, cap_t, lane);
        if (done || L >= g.B) break;
    }
    if (FILT == FILT_NONE && a.pairs_out && lane == 0) add_pairs(a, wr.pairs);
}

// Queries per warp up to which a list is taken one by one: 9.8M outdoor points, k = 4,
// 129 ms with 0 and 4, 126 with 16, 64 and no limit; packed and room scans within 1 %.
#define TAKE_MOST 16

// FILTERED: qlist holds the points whose cost over smaller keys is wanted
// (condition (A)), qlist2 the danger sources whose lambda is wanted.  ORDER:
// equal distances in the order of the tie (input index with W, Morton position
// without), which the weights and the neighbour output need.
// 10 blocks per SM (48 registers) without order, 8 with: the chain of
// dependent loads wants warps in flight (100M-point scan, searches of all rounds:
// 40.6 ms at 8 blocks, 33.7 at 10, 34 at 12 with more spilled).
template <bool FILTERED, bool W, bool ORDER>
__global__ void __launch_bounds__(PD_WARPS * 32, ORDER ? 8 : 10)
    knn_query_kernel(GridView g, KnnArgs a) {
    chain();
    __shared__ WarpRanges s_r[PD_WARPS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!FILTERED && a.finish && blockIdx.x == 0 && threadIdx.x == 0) round_finish(a.finish);
    const int n1 = *a.qcount, n2 = FILTERED ? *a.qcount2 : 0;
    const int step = gridDim.x * PD_WARPS;
    // a short list is taken one by one: its queries' times differ tenfold, and a
    // fixed share of two or three of them left the launch waiting for the
    // unluckiest warp (9.8M outdoor points, k = 4: 125 -> 121 ms); a long one evens
    // out by itself
    int* take = a.take && n1 + n2 <= TAKE_MOST * step ? a.take : nullptr;
    for (int t = blockIdx.x * PD_WARPS + w; t < n1 + n2;
         t = take ? step + warp_take(take, lane) : t + step) {
        if (!FILTERED) warp_query<FILT_NONE, W, ORDER>(g, a, a.qlist[t], s_r[w], lane);
        else if (t < n1) warp_query<FILT_BELOW_SELF, W, ORDER>(g, a, a.qlist[t], s_r[w], lane);
        else warp_query<FILT_BELOW_TAU, W, ORDER>(g, a, a.qlist2[t - n1], s_r[w], lane);
    }
}

cudaError_t launch_knn_queries(const GridView& g, const KnnArgs& a, int64_t cap, cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    const bool filtered = a.qlist2 != nullptr;
    const dim3 gr(list_blocks(cap, 128, 10)), bl(PD_WARPS * 32);
    if (filtered) {
        if (a.term != 0) launch_chained(knn_query_kernel<true, true, true>, gr, bl, 0, st, g, a);
        else launch_chained(knn_query_kernel<true, false, false>, gr, bl, 0, st, g, a);
    } else if (a.term != 0) {
        launch_chained(knn_query_kernel<false, true, true>, gr, bl, 0, st, g, a);
    } else if (a.ordered) {
        launch_chained(knn_query_kernel<false, false, true>, gr, bl, 0, st, g, a);
    } else {
        launch_chained(knn_query_kernel<false, false, false>, gr, bl, 0, st, g, a);
    }
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_knn(const GridView& g, const KnnArgs& a, int64_t n, int* rest, int* nrest,
                       cudaStream_t st) {
    if (a.ngroups <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(nrest, 0, sizeof(int), st);
    if (e) return e;
    const unsigned blocks = (unsigned)((a.ngroups + NEAR_WARPS - 1) / NEAR_WARPS);
    const dim3 gr(blocks), bl(NEAR_WARPS * 32);
    if (a.S == 8) {
        if (a.term != 0) launch_chained(knn_kernel<8, 1>, gr, bl, 0, st, g, a, rest, nrest);
        else launch_chained(knn_kernel<8, 0>, gr, bl, 0, st, g, a, rest, nrest);
    } else if (a.S == 17) {
        if (a.term == PD_TERM_INDEX_TIE)
            launch_chained(knn_kernel<17, 1>, gr, bl, 0, st, g, a, rest, nrest);
        else if (a.term != 0) launch_chained(knn_kernel<17, 2>, gr, bl, 0, st, g, a, rest, nrest);
        else launch_chained(knn_kernel<17, 0>, gr, bl, 0, st, g, a, rest, nrest);
    } else {
        return cudaErrorInvalidValue;
    }
    note_launch();
    e = cudaGetLastError();
    if (e) return e;
    KnnArgs b = a;
    b.qlist = rest;
    b.qcount = nrest;
    b.qlist2 = nullptr;
    b.ordered = 1;
    b.take = nullptr;
    return launch_knn_queries(g, b, n, st);
}

}  // namespace pd
