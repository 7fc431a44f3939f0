// pd_internal.cuh -- shared device definitions of libpd (sm_103a).
//
// Layout of one resident cloud (all arrays indexed by the point's position s
// in Morton order, 0 <= s < n):
//   pos[s]    int4 {x, y, z, input index}     16 B, read by every neighbour scan
//   code[s]   uint64 Morton code of (x,y,z) - origin, >> shift
//   leaf[s]   uint8 level of the octree leaf that holds s
//   alive[s]  uint8 1 while the point is retained
//   prim[s]   uint64 primary key, larger = higher cost (see key_prim_*)
//   nbr[s*S+i] int32 Morton positions of the S nearest live points
//   rk2[s]    uint64 squared distance of the k-th nearest (UINT64_MAX if none)
//   flg[s]    uint8 bit0: a further point ties the k-th distance
//                   bit1: (k = 1) the stored nearest-distance shell may be incomplete
// A cell of level L is the set of points whose codes share the prefix
// code >> 3L; it is a contiguous range of the Morton order.  The octree keeps
// splitting cells holding more than T points; its nodes (internal and leaf)
// are stored in an open-addressing hash keyed by (level, prefix).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#define PD_WARPS 4                 // warps per block in warp-per-group kernels
#define PD_MAXLEVEL 21             // Morton bits per axis
#define PD_EMPTY_KEY 0ull

namespace pd {

struct HashSlot {
    unsigned long long key;        // marker-bit encoded (level, prefix); 0 = empty
    uint32_t b, e;                 // [b, e) in Morton order
};

struct GridView {
    const int4* pos;
    const unsigned long long* code;
    const uint8_t* leaf;
    const HashSlot* hash;
    unsigned long long hmask;
    int B;         // Morton bits per axis of the root cell
    int shift;     // coordinates are (x - origin) >> shift before interleaving
    int T;         // largest leaf
    int3 origin;
    int3 umax;     // largest (x - origin) per axis
};

// ---------------------------------------------------------------- Morton
__host__ __device__ inline unsigned long long spread3(uint32_t v) {
    unsigned long long x = v & 0x1fffffu;
    x = (x | (x << 32)) & 0x1f00000000ffffull;
    x = (x | (x << 16)) & 0x1f0000ff0000ffull;
    x = (x | (x << 8)) & 0x100f00f00f00f00full;
    x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
    x = (x | (x << 2)) & 0x1249249249249249ull;
    return x;
}
__host__ __device__ inline uint32_t compact3(unsigned long long x) {
    x &= 0x1249249249249249ull;
    x = (x ^ (x >> 2)) & 0x10c30c30c30c30c3ull;
    x = (x ^ (x >> 4)) & 0x100f00f00f00f00full;
    x = (x ^ (x >> 8)) & 0x1f0000ff0000ffull;
    x = (x ^ (x >> 16)) & 0x1f00000000ffffull;
    x = (x ^ (x >> 32)) & 0x1fffffull;
    return (uint32_t)x;
}
__host__ __device__ inline unsigned long long morton3(uint32_t x, uint32_t y, uint32_t z) {
    return spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
}

// (level, prefix) -> hash key: a marker bit just above the prefix's 3(B-L) bits.
__device__ inline unsigned long long cell_key(unsigned long long prefix, int L, int B) {
    return (1ull << (3 * (B - L))) | prefix;
}
// Slot of a key: the upper half of a multiplication by 2^64 over the golden
// ratio (Fibonacci hashing, Knuth, TAOCP vol. 3, 6.4).  A search resolves 27
// cells and the ancestors of the empty ones, so the hash is most of its set-up:
// one 64-bit multiplication instead of a two-multiplication finaliser.
__device__ inline unsigned long long hash_slot(unsigned long long k, unsigned long long mask) {
    return ((k * 0x9e3779b97f4a7c15ull) >> 32) & mask;
}
__device__ inline bool hash_find(const HashSlot* tab, unsigned long long mask,
                                 unsigned long long key, uint32_t& b, uint32_t& e) {
    unsigned long long h = hash_slot(key, mask);
    for (unsigned long long i = 0; i <= mask; i++) {
        unsigned long long k = tab[h].key;
        if (k == key) {
            b = tab[h].b;
            e = tab[h].e;
            return true;
        }
        if (k == PD_EMPTY_KEY) return false;
        h = (h + 1) & mask;
    }
    return false;
}

// Range of the level-L cell with this Morton prefix.  Returns 0 = empty, 1 =
// the cell is an octree node (its exact range), 2 = the cell lies inside a
// coarser leaf (the whole leaf's range is returned; *lvl_out = that leaf's level).
__device__ inline int resolve_prefix(const GridView& g, int L, unsigned long long prefix,
                                     uint32_t& b, uint32_t& e, int* lvl_out) {
    if (hash_find(g.hash, g.hmask, cell_key(prefix, L, g.B), b, e)) {
        *lvl_out = L;
        return 1;
    }
    for (int L2 = L + 1; L2 <= g.B; L2++) {
        prefix >>= 3;
        if (hash_find(g.hash, g.hmask, cell_key(prefix, L2, g.B), b, e)) {
            if (e - b > (uint32_t)g.T) return 0;  // internal node: that child is empty
            *lvl_out = L2;
            return 2;
        }
    }
    return 0;
}
// The same for the cell (cx,cy,cz); 0 outside the grid.
__device__ inline int resolve_cell(const GridView& g, int L, int cx, int cy, int cz,
                                   uint32_t& b, uint32_t& e, int* lvl_out) {
    int lim = 1 << (g.B - L);
    if (cx < 0 || cy < 0 || cz < 0 || cx >= lim || cy >= lim || cz >= lim) return 0;
    return resolve_prefix(g, L, morton3((uint32_t)cx, (uint32_t)cy, (uint32_t)cz), b, e, lvl_out);
}
// The prefix of the cell at offset (dx, dy, dz), each in -1..1, from the cell
// with prefix p of 3 nb bits: additions on the interleaved bits of each axis.
// False outside the grid.
__device__ inline bool prefix_offset(unsigned long long& p, int nb, int dx, int dy, int dz) {
    const unsigned long long full = (1ull << (3 * nb)) - 1;
    const int d[3] = {dx, dy, dz};
    unsigned long long out = 0;
    bool in = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const unsigned long long m = (0x1249249249249249ull << a) & full;
        const unsigned long long v = p & m;
        if (d[a] > 0) in = in && v != m;
        if (d[a] < 0) in = in && v != 0;
        out |= (d[a] > 0 ? (p | ~m) + 1 : (d[a] < 0 ? v - 1 : v)) & m;
    }
    p = out;
    return in;
}

// ---------------------------------------------------------------- keys
// Larger key = removed first: (cost, input index) compared lexicographically.
// k = 1 density cost: order by d1^2 ascending, encoded as the complement of
// the IEEE bits of (double)d1^2 (exact: d^2 < 2^53).  Other costs: the IEEE
// bits of the non-negative binary64 cost (+inf for coincident points).
__device__ inline unsigned long long key_prim_d2(unsigned long long d2) {
    double v = d2 == ~0ull ? __longlong_as_double(0x7ff0000000000000ll) : (double)d2;
    return ~(unsigned long long)__double_as_longlong(v);
}
__device__ inline unsigned long long key_prim_cost(double c) {
    return (unsigned long long)__double_as_longlong(c);
}
__device__ inline bool key_gt(unsigned long long pa, int ia, unsigned long long pb, int ib) {
    return pa > pb || (pa == pb && ia > ib);
}
// Digit `pass` (12 bits) of the 96-bit key (prim << 32 | input index), most
// significant first: passes 0-4 read prim, 5 straddles, 6-7 read the index.
__device__ inline uint32_t key_digit(unsigned long long prim, int idx, int pass) {
    const int lo = 84 - 12 * pass;  // lowest bit of the digit
    const uint32_t ui = (uint32_t)idx;
    if (lo >= 32) return (uint32_t)(prim >> (lo - 32)) & 0xfffu;
    if (lo + 12 <= 32) return (ui >> lo) & 0xfffu;
    // straddle: bits [lo, 32) of idx and [0, lo + 12 - 32) of prim
    return ((uint32_t)(prim << (32 - lo)) | (ui >> lo)) & 0xfffu;
}

// Per-neighbour weight of the optional cost terms (section "Additional cost
// terms"): 1 - a * ||rgb_p - rgb_q|| / (255 sqrt 3) for colour, 1 - a * (1 -
// |n_p . n_q|) for orientation (Eq. 13), 1 otherwise.  Every operation is a
// separately rounded binary64 operation (no contraction).
__device__ inline double term_weight(int term, double a, const uchar4* rgb, const float4* nrm,
                                     int q, int j) {
    if (term == 1) {
        uchar4 p = rgb[q], r = rgb[j];
        double dr = (double)p.x - (double)r.x;
        double dg = (double)p.y - (double)r.y;
        double db = (double)p.z - (double)r.z;
        double s = __dmul_rn(dr, dr);
        s = __dadd_rn(s, __dmul_rn(dg, dg));
        s = __dadd_rn(s, __dmul_rn(db, db));
        double dist = __dsqrt_rn(s);
        double scale = __dmul_rn(255.0, __dsqrt_rn(3.0));
        return __dsub_rn(1.0, __dmul_rn(a, __ddiv_rn(dist, scale)));
    }
    if (term == 2) {
        float4 p = nrm[q], r = nrm[j];
        double d = __dmul_rn((double)p.x, (double)r.x);
        d = __dadd_rn(d, __dmul_rn((double)p.y, (double)r.y));
        d = __dadd_rn(d, __dmul_rn((double)p.z, (double)r.z));
        return __dsub_rn(1.0, __dmul_rn(a, __dsub_rn(1.0, fabs(d))));
    }
    return 1.0;
}

__device__ inline unsigned long long sqd(int4 a, int4 b) {
    long long dx = (long long)a.x - b.x, dy = (long long)a.y - b.y, dz = (long long)a.z - b.z;
    return (unsigned long long)(dx * dx + dy * dy + dz * dz);
}

// ---------------------------------------------------------------- stored neighbours
// The 8 stored neighbours of a point, two 16-byte accesses (a scalar access per
// entry touches every line of the warp's kilobyte 8 times).
__device__ __forceinline__ void load_nbr8(const int* __restrict__ nbr, long long s, int (&x)[8]) {
    const int4* p = reinterpret_cast<const int4*>(nbr + s * 8);
    const int4 a = p[0], b = p[1];
    x[0] = a.x;
    x[1] = a.y;
    x[2] = a.z;
    x[3] = a.w;
    x[4] = b.x;
    x[5] = b.y;
    x[6] = b.z;
    x[7] = b.w;
}
__device__ __forceinline__ void store_nbr8(int* nbr, long long s, const int (&x)[8]) {
    int4* p = reinterpret_cast<int4*>(nbr + s * 8);
    p[0] = make_int4(x[0], x[1], x[2], x[3]);
    p[1] = make_int4(x[4], x[5], x[6], x[7]);
}
// Moves the live entries to the front, in order, and sets the rest to -1 (in
// registers: every index is a compile-time one); returns their number.
__device__ __forceinline__ int keep_live8(const uint8_t* __restrict__ alive, int (&x)[8]) {
    bool live[8];
#pragma unroll
    for (int i = 0; i < 8; i++) live[i] = x[i] >= 0 && alive[x[i]];
    int r = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int v = x[i];
        x[i] = -1;
#pragma unroll
        for (int j = 0; j <= i; j++)
            if (live[i] && j == r) x[j] = v;
        r += live[i];
    }
    return r;
}

// ---------------------------------------------------------------- launches
// Number of kernels this library has launched (process-wide, host counter).
extern long long g_launch_count;
inline void note_launch() { __atomic_fetch_add(&g_launch_count, 1, __ATOMIC_RELAXED); }

// Programmatic dependent launch: a chained launch may be set up while the kernel
// ahead of it in the stream still runs, and its blocks take the places that the
// last blocks of that kernel leave free.  Every kernel launched this way begins
// with chain(): the launch after it may start, then it waits until the kernel
// ahead has completed (that one waited for its own predecessor, so all before it
// have).  Nothing comes before the wait; the kernels' pointers are not
// __restrict__, which would let the compiler take their loads for constants and
// move them there.  A small or ordinary call is tens to hundreds of short launches:
// static pass of 7.4k points 237 -> 213 us, decimation of 200k points, k = 1, 2.65 ->
// 2.52 ms, w_up of 700k points 9.5 -> 7.8 ms.  The long kernels of the k >= 2 rounds
// (buffer update, candidate test, danger test, pair fixpoint) are launched plainly:
// blocks that wait take places from those that work (9.8M outdoor points, k = 4, 133
// ms, 140 with all of them chained; a packed batch of 3.8M 130 and 135).
__device__ __forceinline__ void chain() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                  cudaStream_t st, A... args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Block-level aggregation of counters and list appends: one global atomic
// per block instead of one per warp (atomics on one address serialise in L2,
// and a full-grid kernel over a billion points has 31M warps).  Every thread
// of the block must make the call (blockDim.x a multiple of 32, <= 1024).
__device__ __forceinline__ void block_add(unsigned long long* dst, unsigned long long v) {
    __shared__ unsigned long long s_part[32];
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();  // s_part may still be read by a previous call
    if (lane == 0) s_part[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) t += s_part[i];
        if (t) atomicAdd(dst, t);
    }
}
// Appends for every thread with want set; returns the thread's slot in the
// list (meaningful where want is set).
__device__ __forceinline__ int block_append(bool want, int* count) {
    __shared__ int s_w[33];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, want);
    __syncthreads();  // s_w may still be read by a previous call
    if (lane == 0) s_w[w] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) {
            int c = s_w[i];
            s_w[i] = acc;
            acc += c;
        }
        s_w[32] = acc ? atomicAdd(count, acc) : 0;
    }
    __syncthreads();
    return s_w[32] + s_w[w] + __popc(m & ((1u << lane) - 1u));
}

// Appends to N lists at once: two block barriers for all of them instead of
// three per list.  slot[i] is meaningful where want[i] is set.
template <int N>
__device__ __forceinline__ void block_append_n(const bool (&want)[N], int* const (&count)[N],
                                               int (&slot)[N]) {
    __shared__ int s_w[N][33];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned m[N];
#pragma unroll
    for (int i = 0; i < N; i++) m[i] = __ballot_sync(0xffffffffu, want[i]);
    __syncthreads();  // s_w may still be read by a previous call
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < N; i++) s_w[i][w] = __popc(m[i]);
    }
    __syncthreads();
    if (threadIdx.x < N) {
        int acc = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) {
            const int c = s_w[threadIdx.x][i];
            s_w[threadIdx.x][i] = acc;
            acc += c;
        }
        int* dst = count[0];
#pragma unroll
        for (int i = 1; i < N; i++)
            if ((int)threadIdx.x == i) dst = count[i];
        s_w[threadIdx.x][32] = acc ? atomicAdd(dst, acc) : 0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; i++)
        slot[i] = s_w[i][32] + s_w[i][w] + __popc(m[i] & ((1u << lane) - 1u));
}

// The next item of a list that the warps of a launch share; every lane calls it.
__device__ __forceinline__ int warp_take(int* next, int lane) {
    int t = 0;
    if (lane == 0) t = atomicAdd(next, 1);
    return __shfl_sync(0xffffffffu, t, 0);
}

// Streaming multiprocessors of the current device (queried once per device
// and cached); persistent and grid-stride launches size their grids from it.
int device_sms();

// ---------------------------------------------------------------- warp utils
// The 3x3x3 cells around a query cell in the order they are scanned: the
// cell itself, the 6 face neighbours, the 12 edge and the 8 corner neighbours
// (cell o = (dx+1) + 3 (dy+1) + 9 (dz+1)).  Nearer cells first tighten the
// k-th distance bound early, which prunes more of the farther cells.
static __device__ __constant__ const unsigned char kCellOrder[27] = {13, 4, 10, 12, 14, 16, 22, 1, 3, 5, 7, 9, 11, 15, 17, 19, 21, 23, 25, 0, 2, 6, 8, 18, 20, 24, 26};


// Squared distance from a point (relative to the grid's origin) to the box of
// cell (bx, by, bz) with edge 2^sh; 0 inside.
__device__ __forceinline__ unsigned long long box_d2(int ux, int uy, int uz, int bx, int by,
                                                     int bz, int sh) {
    const int q[3] = {ux, uy, uz};
    const int c[3] = {bx, by, bz};
    unsigned long long s = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        // coordinates and cell faces are below 2^27, so the gap is an int
        const int lo = c[a] << sh, hi = lo + ((1 << sh) - 1);
        const int d = max(max(lo - q[a], q[a] - hi), 0);
        s += (unsigned long long)((long long)d * d);
    }
    return s;
}

// ---------------------------------------------------------------- one warp, one point
// An octree node held by one lane: positions [b, e), its level and cell, and
// the squared distance from the warp's point to its box.  b == e: none.
struct WarpNode {
    uint32_t b, e;
    int lv, x, y, z;
    unsigned long long box;
    __device__ __forceinline__ uint32_t count() const { return e - b; }
};

// Lane i < 27 takes the level-L cell kCellOrder[i] of the cube around the cell
// of the point (ux, uy, uz) with Morton code c0; a coarser leaf reached from
// several cells is kept once.
__device__ __forceinline__ WarpNode warp_cells(const GridView& g, int L, unsigned long long c0,
                                               int ux, int uy, int uz, int lane) {
    WarpNode n;
    const int o = lane < 27 ? kCellOrder[lane] : 13;
    const int dx = o % 3 - 1, dy = (o / 3) % 3 - 1, dz = o / 9 - 1;
    n.lv = L;
    n.b = n.e = 0;
    n.x = n.y = n.z = 0;
    n.box = ~0ull;
    unsigned long long prefix = L < g.B ? c0 >> (3 * L) : 0;
    int rt = 0;
    if (lane < 27 && prefix_offset(prefix, g.B - L, dx, dy, dz))
        rt = resolve_prefix(g, L, prefix, n.b, n.e, &n.lv);
    const unsigned same = __match_any_sync(0xffffffffu, rt == 2 ? n.b : 0x80000000u + lane);
    if (rt == 2 && __ffs(same) - 1 != lane) rt = 0;
    if (rt) {
        const int sh = L + g.shift, up = n.lv - L;
        n.x = ((ux >> sh) + dx) >> up;
        n.y = ((uy >> sh) + dy) >> up;
        n.z = ((uz >> sh) + dz) >> up;
        n.box = box_d2(ux, uy, uz, n.x, n.y, n.z, n.lv + g.shift);
    } else {
        n.b = n.e = 0;
        n.lv = L;
    }
    return n;
}

// Lane i < 8 takes child i of lane src's node (above level 0).
__device__ __forceinline__ WarpNode warp_children(const GridView& g, const WarpNode& n, int src,
                                                  int ux, int uy, int uz, int lane) {
    WarpNode c;
    c.lv = __shfl_sync(0xffffffffu, n.lv, src) - 1;
    c.x = 2 * __shfl_sync(0xffffffffu, n.x, src) + (lane & 1);
    c.y = 2 * __shfl_sync(0xffffffffu, n.y, src) + ((lane >> 1) & 1);
    c.z = 2 * __shfl_sync(0xffffffffu, n.z, src) + ((lane >> 2) & 1);
    c.b = c.e = 0;
    c.box = ~0ull;
    if (lane < 8 &&
        hash_find(g.hash, g.hmask,
                  cell_key(morton3((uint32_t)c.x, (uint32_t)c.y, (uint32_t)c.z), c.lv, g.B), c.b,
                  c.e))
        c.box = box_d2(ux, uy, uz, c.x, c.y, c.z, c.lv + g.shift);
    else
        c.b = c.e = 0;
    return c;
}

// The free lanes of `held` (no node kept) take the nodes of the lanes with
// `put` set, in lane order; put is cleared where a node was taken.
__device__ __forceinline__ void warp_keep(WarpNode& n, bool& held, const WarpNode& c, bool& put,
                                          int lane) {
    const unsigned pm = __ballot_sync(0xffffffffu, put), fm = __ballot_sync(0xffffffffu, !held);
    if (!pm) return;
    const int np = __popc(pm), nf = __popc(fm);
    const unsigned below = (1u << lane) - 1u;
    const int rank = __popc(fm & below);
    const bool take = !held && rank < np;
    const int src = take ? (int)__fns(pm, 0, rank + 1) : 0;
    WarpNode t;
    t.b = __shfl_sync(0xffffffffu, c.b, src);
    t.e = __shfl_sync(0xffffffffu, c.e, src);
    t.lv = __shfl_sync(0xffffffffu, c.lv, src);
    t.x = __shfl_sync(0xffffffffu, c.x, src);
    t.y = __shfl_sync(0xffffffffu, c.y, src);
    t.z = __shfl_sync(0xffffffffu, c.z, src);
    t.box = __shfl_sync(0xffffffffu, c.box, src);
    if (take) {
        n = t;
        held = true;
    }
    if (put && __popc(pm & below) < nf) put = false;
}

// Inclusive prefix sum over the lanes.
__device__ __forceinline__ uint32_t warp_inclusive(uint32_t v, int lane) {
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, v, s);
        if (lane >= s) v += y;
    }
    return v;
}

}  // namespace pd
