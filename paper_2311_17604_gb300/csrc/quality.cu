// quality.cu -- kernels of the quality report of a decimated cloud.
//
// Section "Results and Discussion" (the cube experiment) judges a decimated
// cloud by the number of its points that fall within a growing neighbourhood
// of each retained point: with an even 2-D distribution the count grows
// linearly with the neighbourhood's area pi r^2, the regression slope is the
// density estimate, and R^2, RMSE and the spread of the fractile bands
// measure how even it is.  Eq. 2's quantity, the smallest nearest-neighbour
// spacing, is the Poisson-disk radius of the result.
//
//   radius_counts_kernel  a block per leaf group (<= 32 retained points, one or
//                         more lanes each): the octree nodes within the largest
//                         radius of the group, then every point of them against
//                         every point of the group (exact integers), counted
//                         per radius: N_j(p) = #{q != p : d^2(p,q) <= r_j^2}.
//                         Per radius: exact integer sums of N and N^2 and a
//                         histogram of N.
//   spacing_kernel        per-block minimum and sum of sqrt of the nearest
//                         squared distance (the k = 1 search's result), block
//                         partials added in block order on the host.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

// A scan's density spans four orders of magnitude (the scanner's poles), so a
// thread per point left the launch waiting for the few threads in the dense
// spots, each walking its 27 cells alone.  Here a block shares one group's
// candidates: 8 warps take 32 candidates each in turn, staged in shared memory and
// compared by every lane.  Nodes are entered by their children for up to
// QUALITY_STEPS levels below the cell whose edge reaches the largest radius, and
// kept where their box is within that radius of the group's box, which leaves
// about a quarter of the 27 cells' points.  Measured (250k retained room points, 7 radii to
// 200 mm): 14.2 -> 1.88 ms.
#define QB 256          // threads per block
#define QW (QB / 32)
#define QNODES 512      // nodes of a group's neighbourhood
#define QUALITY_STEPS 3

struct QNode {
    uint32_t b, e;
    int lv, x, y, z;
};

// Squared distance between a cell's box and the box [lo, hi] (both relative to
// the grid's origin).
__device__ inline u64 box_box_d2(const int lo[3], const int hi[3], int x, int y, int z, int sh) {
    const int c[3] = {x, y, z};
    u64 s = 0;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int cl = c[a] << sh, ch = cl + ((1 << sh) - 1);
        const int d = max(max(cl - hi[a], lo[a] - ch), 0);
        s += (u64)((long long)d * d);
    }
    return s;
}

// NR: most radii (8 or PD_QUALITY_MAXR).  near_radius: the largest radius is at
// most 2^13 mm; a group whose nodes are no wider either has every coordinate
// difference below 3 * 2^13 and its squared distances in 32 bits.
template <int NR>
__global__ void __launch_bounds__(QB)
    radius_counts_kernel(GridView g, const int4* __restrict__ groups, int ngroups, int L,
                         const u64* __restrict__ r2, int nr, u64* __restrict__ sum_n,
                         u64* __restrict__ sum_n2, uint32_t* __restrict__ hist, int H, bool near_radius,
                         int* next) {
    __shared__ union {
        QNode node[2][QNODES];
        uint32_t cnt[QW][32][NR];  // once the nodes are done with
    } sm;
    QNode(&s_node)[2][QNODES] = sm.node;
    __shared__ u64 s_r2[NR];
    __shared__ uint32_t s_first[QNODES + 1];
    __shared__ int4 s_c[QW][32];
    __shared__ int s_n[2], s_group;
    __shared__ uint32_t s_scan[QW];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    uint32_t rr[NR];
#pragma unroll
    for (int j = 0; j < NR; j++) {
        const u64 v = j < nr ? r2[j] : 0;
        rr[j] = v < 0xffffffffull ? (uint32_t)v : 0xffffffffu;
    }
    for (int j = t; j < NR; j += QB) s_r2[j] = j < nr ? r2[j] : 0;
    const u64 rmax2 = r2[nr - 1];
    const uint32_t rmax32 = rmax2 < 0xffffffffull ? (uint32_t)rmax2 : 0xffffffffu;
    u64 acc = 0, acc2 = 0;  // thread j < nr: sums of radius j over this block's groups
    for (;;) {
        __syncthreads();  // the previous group's readers are done
        if (t == 0) {
            s_group = atomicAdd(next, 1);
            s_n[0] = s_n[1] = 0;
        }
        __syncthreads();
        const int gi = s_group;
        if (gi >= ngroups) break;
        const int4 G = groups[gi];
        // as many lanes per point as fit: they share its candidates
        int lpq = 32;
        while (lpq * G.y > 32) lpq >>= 1;
        const int qi = lane / lpq, sub = lane - qi * lpq;
        const bool on = qi < G.y;
        const int4 p = g.pos[G.x + (on ? qi : 0)];
        int lo[3], hi[3];
        {
            const int u[3] = {p.x - g.origin.x, p.y - g.origin.y, p.z - g.origin.z};
#pragma unroll
            for (int a = 0; a < 3; a++) {
                lo[a] = __reduce_min_sync(0xffffffffu, u[a]);
                hi[a] = __reduce_max_sync(0xffffffffu, u[a]);
            }
        }
        // the cells around the group's, at a level that holds the group in one
        const int L0 = max(L, G.z);
        if (t < 27) {
            QNode n;
            const int sh = L0 + g.shift;
            n.x = (L0 < g.B ? lo[0] >> sh : 0) + t % 3 - 1;
            n.y = (L0 < g.B ? lo[1] >> sh : 0) + (t / 3) % 3 - 1;
            n.z = (L0 < g.B ? lo[2] >> sh : 0) + t / 9 - 1;
            const int rt = resolve_cell(g, L0, n.x, n.y, n.z, n.b, n.e, &n.lv);
            bool keep = rt != 0;
            if (rt == 2) {
                // a coarser leaf reached from several cells is kept by the first
                // of them (the least corner of the leaf within the cube)
                const int up = n.lv - L0;
                const int c[3] = {n.x, n.y, n.z};
                const int q[3] = {lo[0] >> sh, lo[1] >> sh, lo[2] >> sh};
                for (int a = 0; a < 3; a++)
                    keep = keep && c[a] == max((c[a] >> up) << up, q[a] - 1);
                n.x >>= up;
                n.y >>= up;
                n.z >>= up;
            }
            if (keep && box_box_d2(lo, hi, n.x, n.y, n.z, n.lv + g.shift) <= rmax2)
                s_node[0][atomicAdd(&s_n[0], 1)] = n;
        }
        __syncthreads();
        int cur = 0;
        for (int step = 0; step < QUALITY_STEPS; step++) {
            const int m = s_n[cur];
            for (int i = t; i < 8 * m; i += QB) {
                QNode n = s_node[cur][i >> 3];
                const int c = i & 7;
                bool keep;
                if (n.e - n.b <= 32 || n.lv == 0) {
                    keep = c == 0;  // a small node stays whole
                } else {
                    n.lv--;
                    n.x = 2 * n.x + (c & 1);
                    n.y = 2 * n.y + ((c >> 1) & 1);
                    n.z = 2 * n.z + (c >> 2);
                    keep = hash_find(g.hash, g.hmask,
                                     cell_key(morton3((uint32_t)n.x, (uint32_t)n.y, (uint32_t)n.z),
                                              n.lv, g.B),
                                     n.b, n.e) &&
                           box_box_d2(lo, hi, n.x, n.y, n.z, n.lv + g.shift) <= rmax2;
                }
                if (keep) {
                    const int at = atomicAdd(&s_n[cur ^ 1], 1);
                    if (at < QNODES) s_node[cur ^ 1][at] = n;
                }
            }
            __syncthreads();
            if (s_n[cur ^ 1] > QNODES) break;  // too many: the coarser nodes stand
            cur ^= 1;
            __syncthreads();
            if (t == 0) s_n[cur ^ 1] = 0;
            __syncthreads();
        }
        // candidates of the nodes laid end to end
        const int m = s_n[cur];
        bool near;
        {
            const int per = QNODES / QB;
            uint32_t c[per], sum = 0;
            bool wide = !near_radius || G.z + g.shift > 13;
#pragma unroll
            for (int j = 0; j < per; j++) {
                const int i = t * per + j;
                c[j] = 0;
                if (i < m) {
                    c[j] = s_node[cur][i].e - s_node[cur][i].b;
                    wide = wide || s_node[cur][i].lv + g.shift > 13;
                }
                sum += c[j];
            }
            near = !__syncthreads_or(wide);
            const uint32_t inc = warp_inclusive(sum, lane);
            if (lane == 31) s_scan[w] = inc;
            __syncthreads();
            uint32_t off = inc - sum;
            for (int i = 0; i < w; i++) off += s_scan[i];
#pragma unroll
            for (int j = 0; j < per; j++) {
                s_first[t * per + j] = off;
                off += c[j];
            }
            if (t == QB - 1) s_first[QNODES] = off;
        }
        __syncthreads();
        const uint32_t total = s_first[QNODES];
        uint32_t cnt[NR];
#pragma unroll
        for (int j = 0; j < NR; j++) cnt[j] = 0;
        for (uint32_t c0 = w * 32; c0 < total; c0 += QB) {
            const uint32_t x = c0 + lane;
            int4 v = make_int4(0, 0, 0, 0);
            if (x < total) {
                int a = 0;  // the last node that starts at or before x
#pragma unroll
                for (int step = QNODES / 2; step; step >>= 1)
                    if (s_first[a + step] <= x) a += step;
                v = g.pos[s_node[cur][a].b + (x - s_first[a])];
            }
            __syncwarp();
            s_c[w][lane] = v;
            __syncwarp();
            const int mm = (int)min(32u, total - c0);
            if (near) {
                for (int i = sub; i < mm; i += lpq) {
                    const int4 q = s_c[w][i];
                    const int dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
                    const uint32_t d2 =
                        (uint32_t)(dx * dx) + (uint32_t)(dy * dy) + (uint32_t)(dz * dz);
                    if (d2 <= rmax32) {
#pragma unroll
                        for (int j = 0; j < NR; j++) cnt[j] += d2 <= rr[j];
                    }
                }
            } else {
                for (int i = sub; i < mm; i += lpq) {
                    const u64 d2 = sqd(s_c[w][i], p);
                    if (d2 <= rmax2) {
#pragma unroll
                        for (int j = 0; j < NR; j++) cnt[j] += d2 <= s_r2[j];
                    }
                }
            }
        }
        __syncthreads();  // the nodes are done with
#pragma unroll
        for (int j = 0; j < NR; j++) sm.cnt[w][lane][j] = cnt[j];
        __syncthreads();
        // thread (radius j, point i): the point's count, without itself
        for (int i = t; i < 32 * nr; i += QB) {
            const int j = i >> 5, q = i & 31;  // a warp per radius
            uint32_t c = 0;
            if (q < G.y) {
                for (int ww = 0; ww < QW; ww++)
                    for (int k = 0; k < lpq; k++) c += sm.cnt[ww][q * lpq + k][j];
                c -= 1;
                atomicAdd(&hist[(int64_t)j * H + (c < (uint32_t)H ? c : (uint32_t)(H - 1))], 1u);
            }
            u64 s1 = c, s2 = (u64)c * c;
            for (int o = 16; o; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            if (lane == (j >> 3)) {  // lane j / 8 of warp j % 8 keeps radius j
                acc += s1;
                acc2 += s2;
            }
        }
    }
    const int j = lane * QW + w;
    if (j < nr) {
        if (acc) atomicAdd(&sum_n[j], acc);
        if (acc2) atomicAdd(&sum_n2[j], acc2);
    }
}

cudaError_t launch_radius_counts(const GridView& g, const int4* groups, int ngroups, int L,
                                 int rmax, const u64* r2, int nr, u64* sum_n, u64* sum_n2,
                                 uint32_t* hist, int H, int* next, cudaStream_t st) {
    if (ngroups <= 0) return cudaSuccess;
    if (nr < 1 || nr > PD_QUALITY_MAXR) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(next, 0, sizeof(int), st);
    if (e) return e;
    const int lim = device_sms() * 4;
    const int blocks = ngroups < lim ? ngroups : lim;
    const bool near = rmax <= (1 << 13);
    if (nr <= 8)
        radius_counts_kernel<8><<<blocks, QB, 0, st>>>(g, groups, ngroups, L, r2, nr, sum_n,
                                                       sum_n2, hist, H, near, next);
    else
        radius_counts_kernel<PD_QUALITY_MAXR><<<blocks, QB, 0, st>>>(
            g, groups, ngroups, L, r2, nr, sum_n, sum_n2, hist, H, near, next);
    note_launch();
    return cudaGetLastError();
}

// Per block: the least nearest squared distance and the sum of the nearest
// distances (binary64, in a fixed order within the block).  ~0 = no neighbour.
__global__ void spacing_kernel(const u64* __restrict__ rk2, int64_t n, u64* __restrict__ bmin,
                               double* __restrict__ bsum) {
    __shared__ u64 s_min[256];
    __shared__ double s_sum[256];
    const int t = threadIdx.x;
    const int64_t s = blockIdx.x * (int64_t)256 + t;
    u64 v = s < n ? rk2[s] : ~0ull;
    s_min[t] = v;
    s_sum[t] = v == ~0ull ? 0.0 : __dsqrt_rn((double)v);
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (t < o) {
            s_min[t] = s_min[t + o] < s_min[t] ? s_min[t + o] : s_min[t];
            s_sum[t] = __dadd_rn(s_sum[t], s_sum[t + o]);
        }
        __syncthreads();
    }
    if (t == 0) {
        bmin[blockIdx.x] = s_min[0];
        bsum[blockIdx.x] = s_sum[0];
    }
}

cudaError_t launch_spacing(const u64* rk2, int64_t n, u64* bmin, double* bsum, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    spacing_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(rk2, n, bmin, bsum);
    note_launch();
    return cudaGetLastError();
}

// Rows of an n x 3 int32 array at the listed positions (ascending input order).
__global__ void take_xyz_kernel(const int* __restrict__ list, const int* __restrict__ count,
                                const int32_t* __restrict__ xyz, int32_t* __restrict__ out) {
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= *count) return;
    const int64_t i = list[t];
    out[3 * t] = xyz[3 * i];
    out[3 * t + 1] = xyz[3 * i + 1];
    out[3 * t + 2] = xyz[3 * i + 2];
}

cudaError_t launch_take_xyz(const int* list, const int* count, int64_t cap, const int32_t* xyz,
                            int32_t* out, cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    take_xyz_kernel<<<(unsigned)((cap + 255) / 256), 256, 0, st>>>(list, count, xyz, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace pd
