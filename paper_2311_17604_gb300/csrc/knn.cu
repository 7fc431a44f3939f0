// knn.cu -- exact k-nearest-neighbour search and cost (Eq. 10 / Eq. 11).
//
// One warp serves one group of <= 32 query points that share an octree leaf
// of level L.  The warp resolves the 3x3x3 level-L cells around the leaf in
// the hashed cell table (the own cell first), then scans their points in
// chunks of 32: every lane loads one candidate (a coalesced 16-byte int4
// load of {x, y, z, index}), the chunk is staged in shared memory, and every
// lane streams the whole chunk against its own query, keeping the S smallest
// (d^2, position) pairs in registers.  Squared distances are exact integers:
// uint32 at levels whose resolved cells are at most 2^13 mm wide (every
// coordinate difference within the 3x3x3 cells is then below 3 * 2^13, so
// d^2 < 2^32), uint64 otherwise.  A cell is skipped when its box is farther than
// the current bound for every lane.  Exactness: every point outside the
// searched cube lies at least g from the query (g = distance to the cube's
// faces); when the bound that matters is below g^2 the lane is done,
// otherwise the search repeats one level up (a cube of twice the size).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define FULLM 0xffffffffu

// The S smallest (d^2, input index) pairs; id holds the Morton position.
// Equal distances are ordered by input index, as in the definition's reading
// (it matters only when neighbour weights differ, i.e. colour/orientation).
template <int S, bool W>
struct TopList;

// Density costs: any order among equal distances gives the same cost, so the
// Morton position serves as the tie order (no extra registers).
template <int S>
struct TopList<S, false> {
    u64 d[S];
    int id[S];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int i = 0; i < S; i++) {
            d[i] = ~0ull;
            id[i] = 0x7fffffff;
        }
    }
    __device__ __forceinline__ int tie(int i) const { return id[i]; }
    __device__ __forceinline__ bool beats_last(u64 dd, int j, int) const {
        return dd < d[S - 1] || (dd == d[S - 1] && j < id[S - 1]);
    }
    __device__ __forceinline__ void insert(u64 dd, int j, int) {
        d[S - 1] = dd;
        id[S - 1] = j;
#pragma unroll
        for (int i = S - 1; i > 0; i--) {
            bool sw = d[i] < d[i - 1] || (d[i] == d[i - 1] && id[i] < id[i - 1]);
            u64 a = d[i], b = d[i - 1];
            int x = id[i], y = id[i - 1];
            d[i - 1] = sw ? a : b;
            d[i] = sw ? b : a;
            id[i - 1] = sw ? x : y;
            id[i] = sw ? y : x;
        }
    }
    __device__ __forceinline__ u64 at(int r) const {
        u64 v = d[0];
#pragma unroll
        for (int i = 1; i < S; i++)
            if (i == r) v = d[i];
        return v;
    }
    __device__ __forceinline__ u64 dist(int i) const { return d[i]; }
    __device__ __forceinline__ int ident(int i) const { return id[i]; }
    __device__ __forceinline__ bool has(int i) const { return d[i] != ~0ull; }
    // merge the list of lane (lane ^ off) into this lane's (active lanes only)
    __device__ __forceinline__ void merge_xor(int off, bool active) {
        u64 od[S];
        int oj[S], oo[S];
#pragma unroll
        for (int i = 0; i < S; i++) {
            od[i] = __shfl_xor_sync(0xffffffffu, d[i], off);
            oj[i] = __shfl_xor_sync(0xffffffffu, id[i], off);
            oo[i] = __shfl_xor_sync(0xffffffffu, tie(i), off);
        }
        if (active) {
#pragma unroll
            for (int i = 0; i < S; i++)
                if (od[i] != ~0ull && beats_last(od[i], oj[i], oo[i])) insert(od[i], oj[i], oo[i]);
        }
    }
};

template <int S>
struct TopList<S, true> {
    u64 d[S];
    int id[S];
    int oi[S];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int i = 0; i < S; i++) {
            d[i] = ~0ull;
            id[i] = 0x7fffffff;
            oi[i] = 0x7fffffff;
        }
    }
    __device__ __forceinline__ int tie(int i) const { return oi[i]; }
    __device__ __forceinline__ bool beats_last(u64 dd, int, int o) const {
        return dd < d[S - 1] || (dd == d[S - 1] && o < oi[S - 1]);
    }
    __device__ __forceinline__ void insert(u64 dd, int j, int o) {
        d[S - 1] = dd;
        id[S - 1] = j;
        oi[S - 1] = o;
#pragma unroll
        for (int i = S - 1; i > 0; i--) {
            bool sw = d[i] < d[i - 1] || (d[i] == d[i - 1] && oi[i] < oi[i - 1]);
            u64 a = d[i], b = d[i - 1];
            int x = id[i], y = id[i - 1];
            int u = oi[i], v = oi[i - 1];
            d[i - 1] = sw ? a : b;
            d[i] = sw ? b : a;
            id[i - 1] = sw ? x : y;
            id[i] = sw ? y : x;
            oi[i - 1] = sw ? u : v;
            oi[i] = sw ? v : u;
        }
    }
    __device__ __forceinline__ u64 at(int r) const {
        u64 v = d[0];
#pragma unroll
        for (int i = 1; i < S; i++)
            if (i == r) v = d[i];
        return v;
    }
    __device__ __forceinline__ u64 dist(int i) const { return d[i]; }
    __device__ __forceinline__ int ident(int i) const { return id[i]; }
    __device__ __forceinline__ bool has(int i) const { return d[i] != ~0ull; }
    // merge the list of lane (lane ^ off) into this lane's (active lanes only)
    __device__ __forceinline__ void merge_xor(int off, bool active) {
        u64 od[S];
        int oj[S], oo[S];
#pragma unroll
        for (int i = 0; i < S; i++) {
            od[i] = __shfl_xor_sync(0xffffffffu, d[i], off);
            oj[i] = __shfl_xor_sync(0xffffffffu, id[i], off);
            oo[i] = __shfl_xor_sync(0xffffffffu, tie(i), off);
        }
        if (active) {
#pragma unroll
            for (int i = 0; i < S; i++)
                if (od[i] != ~0ull && beats_last(od[i], oj[i], oo[i])) insert(od[i], oj[i], oo[i]);
        }
    }
};


// The same lists when every squared distance of the search level is below
// 2^32: one 64-bit key (d^2 << 32 | tie) per entry, so that a compare-exchange
// stage is one 64-bit compare and select.  The order is the same as above
// ((d^2, tie) lexicographic), so results are identical.  W = false: the tie is
// the Morton position, which is also the neighbour; W = true: the tie is the
// input index and the Morton position is kept beside it.
template <int S, bool W>
struct TopPack {
    u64 key[S];
    int pid[W ? S : 1];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int i = 0; i < S; i++) key[i] = ~0ull;
        if (W) {
#pragma unroll
            for (int i = 0; i < S; i++) pid[W ? i : 0] = 0x7fffffff;
        }
    }
    __device__ __forceinline__ static u64 pack(u64 dd, int j, int o) {
        return (dd << 32) | (uint32_t)(W ? o : j);
    }
    __device__ __forceinline__ int tie(int i) const { return (int)(uint32_t)key[i]; }
    __device__ __forceinline__ bool beats_last(u64 dd, int j, int o) const {
        return pack(dd, j, o) < key[S - 1];
    }
    __device__ __forceinline__ void insert(u64 dd, int j, int o) {
        key[S - 1] = pack(dd, j, o);
        if (W) pid[W ? S - 1 : 0] = j;
#pragma unroll
        for (int i = S - 1; i > 0; i--) {
            u64 a = key[i], b = key[i - 1];
            bool sw = a < b;
            key[i - 1] = sw ? a : b;
            key[i] = sw ? b : a;
            if (W) {
                int x = pid[W ? i : 0], y = pid[W ? i - 1 : 0];
                pid[W ? i - 1 : 0] = sw ? x : y;
                pid[W ? i : 0] = sw ? y : x;
            }
        }
    }
    __device__ __forceinline__ bool has(int i) const { return key[i] != ~0ull; }
    __device__ __forceinline__ u64 dist(int i) const {
        return key[i] == ~0ull ? ~0ull : (key[i] >> 32);
    }
    __device__ __forceinline__ int ident(int i) const {
        return W ? pid[W ? i : 0] : (int)(uint32_t)key[i];
    }
    __device__ __forceinline__ u64 at(int r) const {
        u64 v = key[0];
#pragma unroll
        for (int i = 1; i < S; i++)
            if (i == r) v = key[i];
        return v == ~0ull ? ~0ull : (v >> 32);
    }
    __device__ __forceinline__ void merge_xor(int off, bool active) {
        u64 ok[S];
        int op[W ? S : 1];
#pragma unroll
        for (int i = 0; i < S; i++) {
            ok[i] = __shfl_xor_sync(0xffffffffu, key[i], off);
            if (W) op[W ? i : 0] = __shfl_xor_sync(0xffffffffu, pid[W ? i : 0], off);
        }
        if (active) {
#pragma unroll
            for (int i = 0; i < S; i++) {
                if (ok[i] != ~0ull && ok[i] < key[S - 1]) {
                    key[S - 1] = ok[i];
                    if (W) pid[W ? S - 1 : 0] = op[W ? i : 0];
#pragma unroll
                    for (int t = S - 1; t > 0; t--) {
                        u64 a = key[t], b = key[t - 1];
                        bool sw = a < b;
                        key[t - 1] = sw ? a : b;
                        key[t] = sw ? b : a;
                        if (W) {
                            int x = pid[W ? t : 0], y = pid[W ? t - 1 : 0];
                            pid[W ? t - 1 : 0] = sw ? x : y;
                            pid[W ? t : 0] = sw ? y : x;
                        }
                    }
                }
            }
        }
    }
};

// box_d2 in 32-bit arithmetic, for levels whose cell edge is at most
// 2^13 mm: the box is the query's own or an adjacent cell's leaf, so every
// coordinate gap is below 2 * 2^13 and the sum below 2^30.
__device__ inline u64 box_d2_32(int ux, int uy, int uz, int bx, int by, int bz, int sh) {
    const int q[3] = {ux, uy, uz};
    const int c[3] = {bx, by, bz};
    uint32_t s = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int lo = c[a] * (1 << sh);
        const int hi = (c[a] + 1) * (1 << sh) - 1;
        const int d = q[a] < lo ? lo - q[a] : (q[a] > hi ? q[a] - hi : 0);
        s += (uint32_t)(d * d);
    }
    return (u64)s;
}

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
    if (a.term == 1) {  // colour deviation
        uchar4 p = a.rgb[q], r = a.rgb[j];
        double dr = (double)p.x - (double)r.x;
        double dg = (double)p.y - (double)r.y;
        double db = (double)p.z - (double)r.z;
        double s = __dmul_rn(dr, dr);
        s = __dadd_rn(s, __dmul_rn(dg, dg));
        s = __dadd_rn(s, __dmul_rn(db, db));
        double dist = __dsqrt_rn(s);
        double scale = __dmul_rn(255.0, __dsqrt_rn(3.0));
        return __dsub_rn(1.0, __dmul_rn(a.weight, __ddiv_rn(dist, scale)));
    }
    if (a.term == 2) {  // orientation, Eq. 13 with |n_p . n_q|
        float4 p = a.nrm[q], r = a.nrm[j];
        double d = __dmul_rn((double)p.x, (double)r.x);
        d = __dadd_rn(d, __dmul_rn((double)p.y, (double)r.y));
        d = __dadd_rn(d, __dmul_rn((double)p.z, (double)r.z));
        return __dsub_rn(1.0, __dmul_rn(a.weight, __dsub_rn(1.0, fabs(d))));
    }
    return 1.0;
}

template <int S, class TL>
__device__ inline double cost_sum(const KnnArgs& a, int q, const TL& top, int k) {
    double c = 0.0;
#pragma unroll
    for (int i = 0; i < S; i++) {
        if (i < k && top.has(i)) {
            double w = nbr_weight(a, q, top.ident(i));
            c = __dadd_rn(c, __ddiv_rn(w, (double)top.dist(i)));
        }
    }
    return c;
}

// Stream one range [b, e) of Morton positions against every lane's query.
template <int S, bool W, class TL, typename D>
__device__ __forceinline__ void scan_range(const GridView& g, const KnnArgs& a, uint32_t b,
                                           uint32_t e, int q, int4 qp, bool todo, TL& top,
                                           int4* sp, int* so, int lane, int sub, int lpq) {
    for (uint32_t c = b; c < e; c += 32) {
        uint32_t j = c + lane;
        int4 v = make_int4(0, 0, 0, -1);
        if (j < e) {
            v = g.pos[j];
            bool ok = !a.alive || a.alive[j];
            if (W) so[lane] = v.w;
            v.w = ok ? (int)j : -1;
        }
        sp[lane] = v;
        __syncwarp();
        int m = (int)min(32u, e - c);
        if (todo) {
            for (int t = sub; t < m; t += lpq) {
                int4 cv = sp[t];
                if (cv.w < 0 || cv.w == q) continue;
                int dx = cv.x - qp.x, dy = cv.y - qp.y, dz = cv.z - qp.z;
                D dd;
                if (sizeof(D) == 4) {
                    dd = (D)(dx * dx) + (D)(dy * dy) + (D)(dz * dz);
                } else {
                    dd = (D)((long long)dx * dx) + (D)((long long)dy * dy) + (D)((long long)dz * dz);
                }
                int co = W ? so[t] : cv.w;
                if (top.beats_last((u64)dd, cv.w, co)) top.insert((u64)dd, cv.w, co);
            }
        }
        __syncwarp();
    }
}

// Results of a query whose list is exact (one lane per query).
// hzv: squared distance below which every live point is in the list (the
// searched cube's gap and the skipped cells' boxes; the S-th distance when
// the list is full).
template <int S, bool W, class TL>
__device__ __forceinline__ void write_result(const KnnArgs& a, int q, const TL& top, u64 hzv) {
    int found = 0;
#pragma unroll
    for (int i = 0; i < S; i++) found += top.has(i);
    if (a.density_k1) {
        // all S nearest are stored (the k+b buffer); the shell is the
        // prefix at the nearest distance d0, its size kept in flg >> 2
        u64 d0 = top.dist(0);
        int shell = 0;
#pragma unroll
        for (int i = 0; i < S; i++) {
            bool h = top.has(i);
            shell += (h && top.dist(i) == d0) ? 1 : 0;
            a.nbr[(int64_t)q * S + i] = h ? top.ident(i) : -1;
        }
        if (!W && a.nbr0_out) a.nbr0_out[q] = top.has(0) ? top.ident(0) : -1;
        a.prim_out[q] = key_prim_d2(d0);
        a.rk2_out[q] = d0;
        a.flg_out[q] = (uint8_t)((shell >= 2 ? 1 : 0) | (shell == S ? 2 : 0) | (shell << 2));
        if (a.hz_out) {
            u64 h = top.has(S - 1) ? top.dist(S - 1) : ~0ull;
            a.hz_out[q] = hzv < h ? hzv : h;
        }
        if (a.cost_out) a.cost_out[q] = d0 == ~0ull ? 0.0 : __ddiv_rn(1.0, (double)d0);
    } else {
        int k = a.k;
#pragma unroll
        for (int i = 0; i < S; i++) a.nbr[(int64_t)q * S + i] = top.has(i) ? top.ident(i) : -1;
        double c = cost_sum<S>(a, q, top, k);
        a.prim_out[q] = key_prim_cost(c);
        u64 dk = top.at(k - 1);
        a.rk2_out[q] = dk;
        bool tie = found > k && top.at(k) == dk;
        a.flg_out[q] = (uint8_t)(tie ? 1 : 0);
        if (a.hz_out) a.hz_out[q] = top.dist(S - 1);
        if (a.cost_out) a.cost_out[q] = c;
    }
}

// One search level for the warp: scan the resolved 3x3x3 ranges, merge each
// query's partial lists, and finish the queries whose R-th distance is
// closer than the searched cube's faces.  PACK: every range of this level
// has squared distances below 2^32 (packed lists, 32-bit distances).
template <int S, bool W, class TL, bool PACK>
__device__ __forceinline__ void knn_level(const GridView& g, const KnnArgs& a, int L, int R,
                                          int q, int4 qp, int ux, int uy, int uz, bool& todo,
                                          int lane, int sub, int lpq, int rt, uint32_t rb,
                                          uint32_t re, int rl, int bx, int by, int bz, int cx,
                                          int cy, int cz, int4* sp, int* so,
                                          unsigned long long& wpairs) {
    TL top;
    top.init();
    u64 hzl = ~0ull;  // smallest box distance of a range this lane did not scan
    for (int r = 0; r < 27; r++) {
        int tr = __shfl_sync(FULLM, rt, r);
        if (!tr) continue;
        uint32_t b = __shfl_sync(FULLM, rb, r), e = __shfl_sync(FULLM, re, r);
        int lv = __shfl_sync(FULLM, rl, r);
        int bxr = __shfl_sync(FULLM, bx, r), byr = __shfl_sync(FULLM, by, r),
            bzr = __shfl_sync(FULLM, bz, r);
        bool skip = true;
        u64 bd = ~0ull;
        if (todo) {
            u64 bound = top.at(R - 1);
            bd = PACK ? box_d2_32(ux, uy, uz, bxr, byr, bzr, lv + g.shift)
                      : box_d2(ux, uy, uz, bxr, byr, bzr, lv + g.shift);
            skip = bound != ~0ull && bd > bound;
        }
        // every lane of the warp scans a range unless none needs it: the
        // lanes that do not still fill their stored entries beyond the R
        // nearest from it (measured: skipping per lane halves the candidates
        // a lane takes but leaves sparser buffers, whose extra re-searches in
        // the removal rounds cost more than the pass saves)
        if (__all_sync(FULLM, skip)) {
            if (bd < hzl) hzl = bd;
            continue;
        }
        if (a.pairs_out) {  // warp-uniform count of the pairs this range costs
            int nqt = __popc(__ballot_sync(FULLM, todo && sub == 0));
            wpairs += (unsigned long long)(e - b) * (unsigned long long)nqt;
        }
        if (PACK || lv + g.shift <= 13)
            scan_range<S, W, TL, uint32_t>(g, a, b, e, q, qp, todo, top, sp, so, lane, sub, lpq);
        else
            scan_range<S, W, TL, u64>(g, a, b, e, q, qp, todo, top, sp, so, lane, sub, lpq);
    }
    // merge the partial lists of each query's lanes (butterfly)
    for (int off = lpq >> 1; off >= 1; off >>= 1) top.merge_xor(off, todo);
    if (todo) {
        u64 gg = L >= g.B ? ~0ull : gap2(g, ux, uy, uz, L, cx, cy, cz);
        u64 bound = top.at(R - 1);
        if (gg == ~0ull || bound < gg) {
            todo = false;
            if (sub == 0) write_result<S, W>(a, q, top, hzl < gg ? hzl : gg);
        }
    }
}

// One leaf group (<= 32 queries) for one warp.
template <int S, bool W>
__device__ __forceinline__ void knn_group(const GridView& g, const KnnArgs& a, int gid, int4* sp,
                                          int* so, int lane) {
    int4 G = a.groups[gid];
    int cnt = G.y;
    int L = G.z;
    int q = -1;
    if (lane < cnt) {
        q = G.x + lane;
        if (a.qflag && !a.qflag[q]) q = -1;
    }
    // pack the active queries onto the 32 lanes: with nq queries each gets
    // lpq = 32 / nq (power of two) lanes that split every staged chunk; their
    // partial lists are merged before the exactness test
    unsigned act = __ballot_sync(FULLM, q >= 0);
    if (!act) return;
    int nq = __popc(act);
    int lpq = 32;
    while (lpq > 1 && nq * lpq > 32) lpq >>= 1;
    int qi = lane / lpq, sub = lane - qi * lpq;
    {
        int srcl = qi < nq ? (int)__fns(act, 0, qi + 1) : 0;
        int qq = __shfl_sync(FULLM, q, srcl);
        q = qi < nq ? qq : -1;
    }
    u64 c0 = g.code[G.x];
    int4 qp = q >= 0 ? g.pos[q] : make_int4(0, 0, 0, 0);
    int ux = qp.x - g.origin.x, uy = qp.y - g.origin.y, uz = qp.z - g.origin.z;
    // exactness bound: the R-th smallest distance must be exact: all S stored
    // neighbours (the k+b neighbour buffer, so a removal can be absorbed
    // without a new search; for the k = 1 density cost the nearest shell is
    // then complete), or the first r_exact of them
    const int R = a.r_exact > 0 && a.r_exact < S ? a.r_exact : S;
    bool todo = q >= 0;
    unsigned long long wpairs = 0;
    while (__any_sync(FULLM, todo)) {
        int sh = 3 * L;
        int cx = (int)compact3(c0 >> sh), cy = (int)compact3(c0 >> (sh + 1)),
            cz = (int)compact3(c0 >> (sh + 2));
        if (L >= g.B) cx = cy = cz = 0;
        int o = lane < 27 ? kCellOrder[lane] : 13;
        int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
        uint32_t rb = 0, re = 0;
        int rl = L, rt = 0;
        u64 prefix = L < g.B ? c0 >> sh : 0;
        if (lane < 27 && prefix_offset(prefix, g.B - L, dx, dy, dz))
            rt = resolve_prefix(g, L, prefix, rb, re, &rl);
        // a coarse leaf reached from two cells is scanned once
        const unsigned same = __match_any_sync(FULLM, rt == 2 ? rb : 0x80000000u + lane);
        if (rt == 2 && __ffs(same) - 1 != lane) rt = 0;
        int bx = 0, by = 0, bz = 0;
        if (rt) {
            bx = (cx + dx) >> (rl - L);
            by = (cy + dy) >> (rl - L);
            bz = (cz + dz) >> (rl - L);
        }
        // 32-bit distances and packed lists when every range of this level is
        // within 3 cells of 2^13 mm (squared distances < 3 * 24576^2 < 2^32)
        bool pack = __all_sync(FULLM, !rt || rl + g.shift <= 13);
        if (pack)
            knn_level<S, W, TopPack<S, W>, true>(g, a, L, R, q, qp, ux, uy, uz, todo, lane, sub,
                                                 lpq, rt, rb, re, rl, bx, by, bz, cx, cy, cz, sp,
                                                 so, wpairs);
        else
            knn_level<S, W, TopList<S, W>, false>(g, a, L, R, q, qp, ux, uy, uz, todo, lane, sub,
                                                  lpq, rt, rb, re, rl, bx, by, bz, cx, cy, cz, sp,
                                                  so, wpairs);
        L++;
    }
    // spread over PD_PAIR_SLOTS counters by SM (one address would serialise
    // in L2; the SM id is read here, so it holds no register during the search)
    if (a.pairs_out && lane == 0 && wpairs) {
        unsigned smid;
        asm volatile("mov.u32 %0, %%smid;" : "=r"(smid));
        atomicAdd(&a.pairs_out[smid % PD_PAIR_SLOTS], wpairs);
    }
}

// The first full pass of the density path (S = 8, no weights) is held to 64
// registers for 8 blocks per SM: more warps in flight measured faster than
// the few bytes it spills (first pass of the 100M-point scan 70.4 -> 67.1 ms).
template <int S, bool W>
__global__ void __launch_bounds__(PD_WARPS * 32, (S == 8 && !W) ? 8 : 1)
    knn_kernel(GridView g, KnnArgs a) {
    __shared__ int4 s_p[PD_WARPS][32];
    __shared__ int s_o[PD_WARPS][32];
    int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int gid = blockIdx.x * PD_WARPS + w;
    if (gid < a.ngroups) knn_group<S, W>(g, a, gid, s_p[w], s_o[w], lane);
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
    // cap_d, cap_t: no key above this one is wanted (cap_d ~0: no cap)
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
    __device__ __forceinline__ uint32_t tie() const { return 0; }
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
        c.live = a.alive[j];
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
            a.hz_out[q] = gg < ds ? gg : ds;
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
        a.hz_out[q] = ds;
    }
    return true;
}

template <bool W>
struct WarpLists {
    typedef WarpList32 Near;
};
template <>
struct WarpLists<true> {
    typedef WarpList<true, true> Near;
};

template <int FILT, bool W>
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
    for (;; L++) {
        const WarpNode n = warp_cells(g, L, c0, ux, uy, uz, lane);
        const int sh = L + g.shift;
        const u64 gg = L >= g.B ? ~0ull : gap2(g, ux, uy, uz, L, ux >> sh, uy >> sh, uz >> sh);
        // every coordinate difference is below 3 cells: d^2 < 27 * 4^(level)
        const bool near = __all_sync(FULLM, n.lv + g.shift <= (W ? 13 : 11));
        const bool done =
            near ? warp_level<FILT, W, typename WarpLists<W>::Near>(
                       g, a, q, qp, S, R, tp, ti, wr, n, ux, uy, uz, gg, cap_d, cap_t, lane)
                 : warp_level<FILT, W, WarpList<W, false>>(g, a, q, qp, S, R, tp, ti, wr, n, ux,
                                                           uy, uz, gg, cap_d, cap_t, lane);
        if (done || L >= g.B) break;
    }
}

// FILTERED: qlist holds the points whose cost over smaller keys is wanted
// (condition (A)), qlist2 the danger sources whose lambda is wanted.
template <bool FILTERED, bool W>
// 10 blocks per SM (48 registers) without weights, 8 with: the chain of
// dependent loads wants warps in flight (100M-point scan, searches of all rounds:
// 40.6 ms at 8 blocks, 33.7 at 10, 34 at 12 with more spilled).
__global__ void __launch_bounds__(PD_WARPS * 32, W ? 8 : 10) knn_query_kernel(GridView g, KnnArgs a) {
    __shared__ WarpRanges s_r[PD_WARPS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (!FILTERED && a.finish && blockIdx.x == 0 && threadIdx.x == 0) round_finish(a.finish);
    const int n1 = *a.qcount, n2 = FILTERED ? *a.qcount2 : 0;
    const int step = gridDim.x * PD_WARPS;
    for (int t = blockIdx.x * PD_WARPS + w; t < n1 + n2; t += step) {
        if (!FILTERED) warp_query<FILT_NONE, W>(g, a, a.qlist[t], s_r[w], lane);
        else if (t < n1) warp_query<FILT_BELOW_SELF, W>(g, a, a.qlist[t], s_r[w], lane);
        else warp_query<FILT_BELOW_TAU, W>(g, a, a.qlist2[t - n1], s_r[w], lane);
    }
}

cudaError_t launch_knn_queries(const GridView& g, const KnnArgs& a, int64_t cap, cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    const bool filtered = a.qlist2 != nullptr;
    const dim3 gr(list_blocks(cap, 128, 10)), bl(PD_WARPS * 32);
    if (filtered) {
        if (a.term != 0) knn_query_kernel<true, true><<<gr, bl, 0, st>>>(g, a);
        else knn_query_kernel<true, false><<<gr, bl, 0, st>>>(g, a);
    } else {
        if (a.term != 0) knn_query_kernel<false, true><<<gr, bl, 0, st>>>(g, a);
        else knn_query_kernel<false, false><<<gr, bl, 0, st>>>(g, a);
    }
    note_launch();
    return cudaGetLastError();
}

template <int S>
static cudaError_t launch_knn_s(const GridView& g, const KnnArgs& a, cudaStream_t st) {
    if (a.ngroups <= 0) return cudaSuccess;
    const unsigned blocks = (unsigned)((a.ngroups + PD_WARPS - 1) / PD_WARPS);
    if (a.term != 0) knn_kernel<S, true><<<blocks, PD_WARPS * 32, 0, st>>>(g, a);
    else knn_kernel<S, false><<<blocks, PD_WARPS * 32, 0, st>>>(g, a);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_knn(const GridView& g, const KnnArgs& a, cudaStream_t st) {
    switch (a.S) {
        case 8: return launch_knn_s<8>(g, a, st);
        case 17: return launch_knn_s<17>(g, a, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pd
