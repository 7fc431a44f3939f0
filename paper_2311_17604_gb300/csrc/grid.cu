// grid.cu -- voxel-grid build: extent, Morton codes, stable LSD radix sort,
// gather into Morton order, adaptive octree leaf levels and the hashed table
// of octree cells (the paper's voxelisation, section "Sub-sampling algorithm",
// rebuilt as one sort that serves every power-of-two cell size).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

// ------------------------------------------------------------------ extent
__global__ void bbox_kernel(const int32_t* __restrict__ xyz, int64_t n, int* out6) {
    int mn[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, mx[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
#pragma unroll 4
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int v = xyz[3 * i + a];
            mn[a] = min(mn[a], v);
            mx[a] = max(mx[a], v);
        }
    }
    // six atomics a block: per warp they queued at the six addresses (1.0M points
    // 40 -> 4 us)
    __shared__ int s_v[6][8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const int lo = __reduce_min_sync(0xffffffffu, mn[a]);
        const int hi = __reduce_max_sync(0xffffffffu, mx[a]);
        if (lane == 0) {
            s_v[a][w] = lo;
            s_v[3 + a][w] = hi;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        int v = s_v[threadIdx.x][0];
        for (int i = 1; i < 8; i++)
            v = threadIdx.x < 3 ? min(v, s_v[threadIdx.x][i]) : max(v, s_v[threadIdx.x][i]);
        if (threadIdx.x < 3) atomicMin(&out6[threadIdx.x], v);
        else atomicMax(&out6[threadIdx.x], v);
    }
}

cudaError_t launch_bbox(const int32_t* xyz, int64_t n, int* out6, cudaStream_t st) {
    int init[6] = {INT32_MAX, INT32_MAX, INT32_MAX, INT32_MIN, INT32_MIN, INT32_MIN};
    cudaError_t e = cudaMemcpyAsync(out6, init, sizeof(init), cudaMemcpyHostToDevice, st);
    if (e) return e;
    int blocks = (int)((n + 255) / 256);
    if (blocks > device_sms() * 4) blocks = device_sms() * 4;
    if (blocks < 1) blocks = 1;
    bbox_kernel<<<blocks, 256, 0, st>>>(xyz, n, out6); note_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ Morton order
// Morton codes sorted with their input indices: a stable LSD radix sort of 8-bit
// digits that reads and writes every pair once per pass.  The digits' totals
// over the cloud do not depend on the order, so the code kernel counts all of
// them at once; a pass then needs, for a tile, only the counts of the tiles
// before it, which the tiles publish and look up while they run (the decoupled
// look-back of Merrill and Garland, "Single-pass Parallel Prefix Scan with
// Decoupled Look-back", NVIDIA NVR-2016-002; in a radix sort: Adinets and
// Merrill, "Onesweep", arXiv 2206.01784).  Bound: the scattered writes and the
// ranking.  A histogram launch, a scan of the tiles' counts (three to five
// launches) and a scatter per pass read every key twice and were launch-bound
// below a million points: neighbours and costs of 1.0M points 1016 -> 951 us, of
// 7.4k 307 -> 262, the decimation of 200k 2.90 -> 2.77 ms, of 100M 134.0 -> 131.9.
#define RS_T 256
#define RS_MAXP 8  // passes of at most 3 PD_MAXLEVEL = 63 bits
#define RS_SPIN 20000

struct SortState {
    uint32_t total[RS_MAXP][256];  // of each digit over the cloud
    uint32_t ticket[RS_MAXP];      // next tile of a pass
};

__global__ void __launch_bounds__(256)
    morton_kernel(const int32_t* xyz, int64_t n, int3 o, int shift, u64* keys, int passes,
                  SortState* ss) {
    chain();
    __shared__ uint32_t h[RS_MAXP][256];
    const int lane = threadIdx.x & 31;
    for (int p = 0; p < passes; p++) h[p][threadIdx.x] = 0;
    __syncthreads();
    const int64_t step = (int64_t)gridDim.x * 256;
    for (int64_t b = blockIdx.x * (int64_t)256; b < n; b += step) {  // uniform over the block
        const int64_t i = b + threadIdx.x;
        const bool in = i < n;
        u64 k = 0;
        if (in) {
            const uint32_t ux = (uint32_t)(xyz[3 * i] - o.x) >> shift;
            const uint32_t uy = (uint32_t)(xyz[3 * i + 1] - o.y) >> shift;
            const uint32_t uz = (uint32_t)(xyz[3 * i + 2] - o.z) >> shift;
            k = morton3(ux, uy, uz);
            keys[i] = k;
        }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (!m) continue;
        // neighbours in the scan share their leading digits: one addition then
        for (int p = 0; p < passes; p++) {
            const uint32_t d = (uint32_t)(k >> (8 * p)) & 255;
            const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);  // lane 0 is in
            if (__all_sync(0xffffffffu, !in || d == d0)) {
                if (lane == 0) atomicAdd(&h[p][d0], (uint32_t)__popc(m));
            } else if (in) {
                atomicAdd(&h[p][d], 1u);
            }
        }
    }
    __syncthreads();
    for (int p = 0; p < passes; p++)
        if (h[p][threadIdx.x]) atomicAdd(&ss->total[p][threadIdx.x], h[p][threadIdx.x]);
}

// Exclusive prefix sums of a and b over the 256 threads of a block.
__device__ __forceinline__ void scan256(uint32_t& a, uint32_t& b, uint32_t (&ws)[2][8]) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = a, y = b;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, x, o), v = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) {
            x += u;
            y += v;
        }
    }
    if (lane == 31) {
        ws[0][w] = x;
        ws[1][w] = y;
    }
    __syncthreads();
    x -= a;
    y -= b;
    for (int i = 0; i < w; i++) {
        x += ws[0][i];
        y += ws[1][i];
    }
    a = x;
    b = y;
}

// One pass over tiles of 256 x PER keys, a warp ranking 32 x PER consecutive
// ones.  The tile's pairs are placed in digit order in shared memory and written
// from there, so that neighbouring threads write neighbouring addresses of a
// digit's run.  status[tile][digit]: (tag, count), the tag 2 pass + 1 for the
// tile's own count and 2 pass + 2 for the sum up to and including it (a pass
// thus never takes an earlier one's words).  Tiles are handed out in order, so a
// tile only waits for tiles that run; after RS_SPIN polls it counts the other
// tile's digit itself, so that no wait is without end.
template <int PER>
__global__ void __launch_bounds__(RS_T, 2)
    radix_pass_kernel(const u64* kin, const uint32_t* vin, u64* kout, uint32_t* vout, int64_t n,
                      int pass, SortState* ss, u64* status) {
    chain();
    const int TILE = RS_T * PER;
    __shared__ u64 sk[RS_T * PER];     // the tile's keys, then its values
    __shared__ uint32_t wc[8][256];    // counts of a warp, then of the warps before it
    __shared__ uint32_t first[256];    // first slot of a digit in the tile
    __shared__ uint32_t to[256];       // where slot x of a digit goes: to[digit] + x
    __shared__ uint32_t ws[2][8];
    __shared__ int s_tile;
    const int t = threadIdx.x, w = t >> 5, lane = t & 31, shift = 8 * pass;
    if (t == 0) s_tile = (int)atomicAdd(&ss->ticket[pass], 1u);
#pragma unroll
    for (int i = 0; i < 8; i++) wc[i][t] = 0;
    __syncthreads();
    const int tile = s_tile;
    const int64_t base = (int64_t)tile * TILE;
    const int tn = (int)min((int64_t)TILE, n - base);
    u64 k[PER];
    uint32_t v[PER];
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const int x = w * 32 * PER + j * 32 + lane;
        // past the end: digit 255, behind every key of the cloud
        k[j] = x < tn ? kin[base + x] : ~0ull;
        v[j] = x < tn ? (vin ? vin[base + x] : (uint32_t)(base + x)) : 0u;
    }
    // slot of each key: its rank among the warp's keys of its digit for now
    uint32_t slot[PER];
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const uint32_t d = (uint32_t)(k[j] >> shift) & 255;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = wc[w][d];
        __syncwarp();
        if (lane == __ffs(peers) - 1) wc[w][d] = before + __popc(peers);
        __syncwarp();
        slot[j] = before + __popc(peers & ((1u << lane) - 1u));
    }
    __syncthreads();
    // thread t: digit t
    uint32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const uint32_t c = wc[i][t];
        wc[i][t] = cnt;
        cnt += c;
    }
    uint32_t lo = cnt, gbase = ss->total[pass][t];
    if (t == 255) cnt -= (uint32_t)(TILE - tn);
    const uint32_t own = 2 * pass + 1, sum = own + 1;
    volatile u64* mine = status + (int64_t)tile * 256 + t;
    *mine = ((u64)(tile ? own : sum) << 32) | cnt;
    scan256(lo, gbase, ws);
    first[t] = lo;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const uint32_t d = (uint32_t)(k[j] >> shift) & 255;
        slot[j] += first[d] + wc[w][d];
        sk[slot[j]] = k[j];
    }
    // the digit's keys in the tiles before: eight of their words at a time
    uint32_t before = 0;
    bool found = false;
    for (int p = tile - 1; p >= 0 && !found; p -= 8) {
        u64 s[8];
#pragma unroll
        for (int i = 0; i < 8; i++)
            s[i] = p - i >= 0 ? *(volatile u64*)(status + (int64_t)(p - i) * 256 + t) : 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            if (p - i < 0 || found) continue;
            u64 x = s[i];
            for (int spin = 0; (uint32_t)(x >> 32) < own && spin < RS_SPIN; spin++)
                x = *(volatile u64*)(status + (int64_t)(p - i) * 256 + t);
            if ((uint32_t)(x >> 32) < own) {
                uint32_t c = 0;
                const int64_t b = (int64_t)(p - i) * TILE;  // a full tile: it is not the last
                for (int y = 0; y < TILE; y++) c += ((uint32_t)(kin[b + y] >> shift) & 255) == t;
                x = c;
            }
            before += (uint32_t)x;
            found = (uint32_t)(x >> 32) == sum;
        }
    }
    if (tile) *mine = ((u64)sum << 32) | (before + cnt);
    to[t] = gbase + before - lo;
    __syncthreads();
    uint32_t at[PER];
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const int x = j * RS_T + t;
        if (x < tn) {
            const u64 q = sk[x];
            at[j] = to[(uint32_t)(q >> shift) & 255] + (uint32_t)x;
            kout[at[j]] = q;
        }
    }
    __syncthreads();
    uint32_t* sv = reinterpret_cast<uint32_t*>(sk);
#pragma unroll
    for (int j = 0; j < PER; j++) sv[slot[j]] = v[j];
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; j++) {
        const int x = j * RS_T + t;
        if (x < tn) vout[at[j]] = sv[x];
    }
}

cudaError_t sort_points(const int32_t* xyz, int64_t n, int3 origin, int shift, int bits, u64* keys,
                        uint32_t* vals, const Scratch& s, cudaStream_t st) {
    const int passes = (bits + 7) / 8;
    if (n < 1 || passes < 1 || passes > RS_MAXP) return cudaErrorInvalidValue;
    // half tiles where full ones would leave SMs without one: grid build of 7.4k
    // points 0.153 ms against 0.171, of 98k 0.174 against 0.179; of 1.0M 0.291
    // against 0.268, of 100M 14.6 against 11.8
    const bool half = n < (int64_t)device_sms() * RS_T * 16;
    const int tile = RS_T * (half ? 8 : 16);
    const int64_t tiles = (n + tile - 1) / tile;
    const size_t words = (size_t)tiles * 256;
    u64* k2 = (u64*)s.get(n * sizeof(u64));
    uint32_t* v2 = (uint32_t*)s.get(n * sizeof(uint32_t));
    u64* status = (u64*)s.get(words * sizeof(u64));
    // apart: a small block stays in device memory, where its atomics belong
    SortState* ss = (SortState*)s.get(sizeof(SortState));
    cudaError_t e = cudaSuccess;
    if (!k2 || !v2 || !status || !ss) e = cudaErrorMemoryAllocation;
    if (!e) e = cudaMemsetAsync(status, 0, words * sizeof(u64), st);
    if (!e) e = cudaMemsetAsync(ss, 0, sizeof(SortState), st);
    if (!e) {
        // the last pass writes keys and vals
        int64_t blocks = (n + 255) / 256;
        const int64_t lim = (int64_t)device_sms() * 8;
        if (blocks > lim) blocks = lim;
        launch_chained(morton_kernel, (unsigned)blocks, 256, 0, st, xyz, n, origin, shift,
                       passes & 1 ? k2 : keys, passes, ss);
        note_launch();
        e = cudaGetLastError();
    }
    for (int p = 0; p < passes && !e; p++) {
        const bool last = ((passes - p) & 1) != 0;  // this pass writes keys, the next one k2
        const u64* ki = last ? k2 : keys;
        const uint32_t* vi = p == 0 ? nullptr : last ? v2 : vals;
        u64* ko = last ? keys : k2;
        uint32_t* vo = last ? vals : v2;
        if (half)
            launch_chained(radix_pass_kernel<8>, (unsigned)tiles, RS_T, 0, st, ki, vi, ko, vo, n,
                           p, ss, status);
        else
            launch_chained(radix_pass_kernel<16>, (unsigned)tiles, RS_T, 0, st, ki, vi, ko, vo, n,
                           p, ss, status);
        note_launch();
        e = cudaGetLastError();
    }
    s.put(ss);
    s.put(status);
    s.put(v2);
    s.put(k2);
    return e;
}

// ------------------------------------------------------------------ scan
// Exclusive prefix sum of uint32 (block = 256 threads x 4 items = 1024).
__global__ void scan_block_kernel(uint32_t* data, int64_t len, uint32_t* sums) {
    __shared__ uint32_t wsum[8];
    int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int64_t base = (int64_t)blockIdx.x * 1024 + t * 4;
    uint32_t v[4];
    uint32_t acc = 0;
    for (int j = 0; j < 4; j++) {
        v[j] = base + j < len ? data[base + j] : 0;
        acc += v[j];
    }
    uint32_t inc = acc;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < 8 ? wsum[lane] : 0;
        for (int o = 1; o < 8; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < 8) wsum[lane] = s;
    }
    __syncthreads();
    uint32_t off = (w ? wsum[w - 1] : 0) + inc - acc;
    for (int j = 0; j < 4; j++) {
        if (base + j < len) data[base + j] = off;
        off += v[j];
    }
    if (t == 255 && sums) sums[blockIdx.x] = wsum[7];
}

__global__ void scan_add_kernel(uint32_t* data, int64_t len, const uint32_t* sums) {
    int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
    uint32_t add = sums[blockIdx.x];
    for (int j = 0; j < 4; j++, i += 256)
        if (i < len) data[i] += add;
}

cudaError_t exclusive_scan_u32(uint32_t* data, int64_t len, const Scratch& s, cudaStream_t st) {
    if (len <= 0) return cudaSuccess;
    int64_t nb = (len + 1023) / 1024;
    if (nb == 1) {
        scan_block_kernel<<<1, 256, 0, st>>>(data, len, nullptr); note_launch();
        return cudaGetLastError();
    }
    uint32_t* sums = (uint32_t*)s.get(nb * sizeof(uint32_t));
    if (!sums) return cudaErrorMemoryAllocation;
    scan_block_kernel<<<(unsigned)nb, 256, 0, st>>>(data, len, sums); note_launch();
    cudaError_t e = exclusive_scan_u32(sums, nb, s, st);
    if (!e) scan_add_kernel<<<(unsigned)nb, 256, 0, st>>>(data, len, sums); note_launch();
    s.put(sums);
    return e ? e : cudaGetLastError();
}

// ------------------------------------------------------------------ gather
__global__ void gather_kernel(const int32_t* xyz, const uint8_t* rgb, const float* nrm,
                              const uint32_t* perm, int64_t n, int4* pos, uchar4* rgb_s,
                              float4* nrm_s) {
    chain();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    uint32_t i = perm[s];
    pos[s] = make_int4(xyz[3 * (int64_t)i], xyz[3 * (int64_t)i + 1], xyz[3 * (int64_t)i + 2],
                       (int)i);
    if (rgb_s) {
        rgb_s[s] = make_uchar4(rgb[3 * (int64_t)i], rgb[3 * (int64_t)i + 1],
                               rgb[3 * (int64_t)i + 2], 0);
    }
    if (nrm_s) {
        nrm_s[s] = make_float4(nrm[3 * (int64_t)i], nrm[3 * (int64_t)i + 1],
                               nrm[3 * (int64_t)i + 2], 0.f);
    }
}

cudaError_t launch_gather(const int32_t* xyz, const uint8_t* rgb, const float* nrm,
                          const uint32_t* perm, int64_t n, int4* pos, uchar4* rgb_s,
                          float4* nrm_s, cudaStream_t st) {
    launch_chained(gather_kernel, (unsigned)((n + 255) / 256), 256, 0, st, xyz,
                   rgb_s ? rgb : nullptr, nrm_s ? nrm : nullptr, perm, n, pos, rgb_s, nrm_s);
    note_launch();
    return cudaGetLastError();
}

__global__ void gather_nrm_kernel(const float* __restrict__ nrm, const int4* __restrict__ pos,
                                  int64_t n, float4* __restrict__ out) {
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int64_t i = pos[s].w;
    out[s] = make_float4(nrm[3 * i], nrm[3 * i + 1], nrm[3 * i + 2], 0.f);
}

cudaError_t launch_gather_nrm(const float* nrm, const int4* pos, int64_t n, float4* out,
                              cudaStream_t st) {
    gather_nrm_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(nrm, pos, n, out); note_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ leaf levels
// A level-L cell holding s has more than T points iff some window of T+1
// consecutive Morton positions around s shares the level-L prefix.  With
// Ls(j) = smallest level at which code[j] and code[j+T] share a cell, the
// leaf level of s is min over j in [s-T, s] of Ls(j), minus one.
__global__ void leaf_level_kernel(const u64* code, int64_t n, int T, int B, uint8_t* leaf) {
    chain();
    extern __shared__ uint8_t ls[];
    int64_t b0 = (int64_t)blockIdx.x * 256;
    for (int x = threadIdx.x; x < 256 + T; x += 256) {
        int64_t j = b0 - T + x;
        uint8_t v = 255;
        if (j >= 0 && j + T < n) {
            u64 d = code[j] ^ code[j + T];
            v = d == 0 ? 0 : (uint8_t)((63 - __clzll((long long)d)) / 3 + 1);
        }
        ls[x] = v;
    }
    __syncthreads();
    int64_t i = b0 + threadIdx.x;
    if (i >= n) return;
    int mn = 255;
    for (int x = 0; x <= T; x++) mn = min(mn, (int)ls[threadIdx.x + x]);
    int L = mn == 255 ? B : (mn > 0 ? mn - 1 : 0);
    if (L > B) L = B;
    leaf[i] = (uint8_t)L;
}

cudaError_t launch_leaf_levels(const u64* code, int64_t n, int T, int B, uint8_t* leaf,
                               cudaStream_t st) {
    launch_chained(leaf_level_kernel, (unsigned)((n + 255) / 256), 256, 256 + T, st, code, n, T,
                   B, leaf);
    note_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ cell table
// Highest level at which the level prefixes (code >> 3L) of a and b differ;
// -1 for equal codes.  Position i opens a level-L cell (a run head) iff
// i == 0 or L <= diff_level(code[i-1], code[i]); it closes one (a run tail)
// iff i == n-1 or L <= diff_level(code[i], code[i+1]).
__device__ inline int diff_level(u64 a, u64 b) {
    u64 d = a ^ b;
    return d ? (63 - __clzll((long long)d)) / 3 : -1;
}
__device__ inline int head_level(const u64* code, int64_t i, int B) {
    return i == 0 ? B : diff_level(code[i - 1], code[i]);
}
__device__ inline int tail_level(const u64* code, int64_t i, int64_t n, int B) {
    return i == n - 1 ? B : diff_level(code[i], code[i + 1]);
}

// Octree nodes: one per (level L >= the point's leaf level, run head).
__global__ void node_count_kernel(const u64* code, const uint8_t* leaf, int64_t n, int B,
                                  unsigned long long* count) {
    chain();
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned c = 0;
    if (i < n) {
        int hi = min(head_level(code, i, B), B);
        int lo = leaf[i];
        c = hi >= lo ? (unsigned)(hi - lo + 1) : 0u;
    }
    block_add(count, c);
}

cudaError_t launch_node_count(const u64* code, const uint8_t* leaf, int64_t n, int B,
                              unsigned long long* count, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), st);
    if (e) return e;
    launch_chained(node_count_kernel, (unsigned)((n + 255) / 256), 256, 0, st, code, leaf, n, B,
                   count);
    note_launch();
    return cudaGetLastError();
}

__device__ inline long long hash_insert(HashSlot* tab, u64 mask, u64 key) {
    u64 h = hash_slot(key, mask);
    for (u64 it = 0; it <= mask; it++) {
        u64 prev = atomicCAS(&tab[h].key, PD_EMPTY_KEY, key);
        if (prev == PD_EMPTY_KEY || prev == key) return (long long)h;
        h = (h + 1) & mask;
    }
    return -1;
}

__global__ void node_insert_kernel(const u64* code, const uint8_t* leaf, int64_t n, int B,
                                   HashSlot* tab, u64 mask) {
    chain();
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int hh = head_level(code, i, B), ht = tail_level(code, i, n, B);
    const int top = min(max(hh, ht), B);  // above it i neither opens nor closes a cell
    const u64 c = code[i];
    for (int L = leaf[i]; L <= top; L++) {
        bool h = L <= hh, t = L <= ht;
        u64 prefix = c >> (3 * L);
        long long slot = hash_insert(tab, mask, cell_key(prefix, L, B));
        if (slot < 0) continue;  // table sized at 2x the node count: cannot fill
        if (h) tab[slot].b = (uint32_t)i;
        if (t) tab[slot].e = (uint32_t)(i + 1);
    }
}

cudaError_t launch_node_insert(const u64* code, const uint8_t* leaf, int64_t n, int B,
                               HashSlot* tab, u64 mask, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(tab, 0, (mask + 1) * sizeof(HashSlot), st);
    if (e) return e;
    launch_chained(node_insert_kernel, (unsigned)((n + 255) / 256), 256, 0, st, code, leaf, n, B,
                   tab, mask);
    note_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ groups
// Range [b, e) of the leaf that holds Morton position s.
__device__ inline bool leaf_range(const GridView& g, int64_t s, uint32_t& b, uint32_t& e) {
    int L = g.leaf[s];
    return hash_find(g.hash, g.hmask, cell_key(g.code[s] >> (3 * L), L, g.B), b, e);
}

// Groups of <= 32 consecutive points of one leaf.  Position s starts a group
// when it opens its leaf, or when the leaf holds 32 or more points before s
// (leaves above 32 points only occur at level 0) and s - b is a multiple of
// 32, b the leaf's first position (from the cell table).
__global__ void leaf_groups_kernel(GridView g, int64_t n, int4* groups, int* ngroups) {
    chain();
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool start = false;
    int cnt = 0, L = 0;
    if (s < n) {
        L = g.leaf[s];
        const u64 p = g.code[s] >> (3 * L);
        if (s == 0 || (g.code[s - 1] >> (3 * L)) != p) {
            start = true;
        } else if (s >= 32 && (g.code[s - 32] >> (3 * L)) == p) {
            uint32_t b, e;
            start = leaf_range(g, s, b, e) && ((uint32_t)s - b) % 32 == 0;
        }
        if (start) {
            cnt = 1;
            while (cnt < 32 && s + cnt < n && (g.code[s + cnt] >> (3 * L)) == p) cnt++;
        }
    }
    const int slot = block_append(start, ngroups);
    if (start) groups[slot] = make_int4((int)s, cnt, L, 0);
}

cudaError_t launch_leaf_groups(const GridView& g, int64_t n, int4* groups, int* ngroups,
                               cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(ngroups, 0, sizeof(int), st);
    if (e) return e;
    launch_chained(leaf_groups_kernel, (unsigned)((n + 255) / 256), 256, 0, st, g, n, groups,
                   ngroups);
    note_launch();
    return cudaGetLastError();
}

// ------------------------------------------------------------------ compaction
__global__ void compact_count_kernel(const uint8_t* __restrict__ flag, int64_t n,
                                     uint32_t* counts) {
    __shared__ uint32_t ws[8];
    int64_t base = (int64_t)blockIdx.x * 1024;
    uint32_t c = 0;
    for (int j = 0; j < 4; j++) {
        int64_t i = base + j * 256 + threadIdx.x;
        c += (i < n && flag[i]) ? 1u : 0u;
    }
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int w = 0; w < 8; w++) s += ws[w];
        counts[blockIdx.x] = s;
    }
}

__global__ void compact_write_kernel(const uint8_t* __restrict__ flag, int64_t n,
                                     const uint32_t* __restrict__ offs, int nblk, int* out,
                                     int* count) {
    __shared__ uint32_t ws[8];
    __shared__ uint32_t run;
    int t = threadIdx.x, lane = t & 31, w = t >> 5;
    if (t == 0) run = offs[blockIdx.x];
    int64_t base = (int64_t)blockIdx.x * 1024;
    for (int j = 0; j < 4; j++) {
        __syncthreads();
        int64_t i = base + j * 256 + t;
        bool f = i < n && flag[i];
        unsigned bal = __ballot_sync(0xffffffffu, f);
        if (lane == 0) ws[w] = __popc(bal);
        __syncthreads();
        uint32_t off = run;
        for (int ww = 0; ww < w; ww++) off += ws[ww];
        if (f) out[off + __popc(bal & ((1u << lane) - 1u))] = (int)i;
        __syncthreads();
        if (t == 0) {
            uint32_t s = 0;
            for (int ww = 0; ww < 8; ww++) s += ws[ww];
            run += s;
        }
    }
    __syncthreads();
    if (blockIdx.x == nblk - 1 && t == 0) *count = (int)run;
}

cudaError_t stable_compact(const uint8_t* flag, int64_t n, int* out, int* count,
                           const Scratch& s, cudaStream_t st) {
    if (n <= 0) return cudaMemsetAsync(count, 0, sizeof(int), st);
    int nblk = (int)((n + 1023) / 1024);
    uint32_t* offs = (uint32_t*)s.get((size_t)nblk * sizeof(uint32_t));
    if (!offs) return cudaErrorMemoryAllocation;
    compact_count_kernel<<<nblk, 256, 0, st>>>(flag, n, offs); note_launch();
    cudaError_t e = cudaGetLastError();
    if (!e) e = exclusive_scan_u32(offs, nblk, s, st);
    if (!e) {
        compact_write_kernel<<<nblk, 256, 0, st>>>(flag, n, offs, nblk, out, count); note_launch();
        e = cudaGetLastError();
    }
    s.put(offs);
    return e;
}

}  // namespace pd
