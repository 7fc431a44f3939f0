// batch.cu -- packed batches: many independent scans decimated in one grid.
//
// The scans of a batch are moved into disjoint aligned tiles (scan i into
// the tile whose Morton index is i) and decimated as one cloud: one grid
// build, one first neighbour pass and one sequence of round launches for all
// of them.  Nothing on the neighbour path knows about scans: tiles are so far
// apart that every neighbour a search returns lies in the query's own scan.
// Only the removal threshold of a round (rule R2: a point may go only if its
// key is among the `need` largest of its cloud) is per scan, so it is
// selected per scan (select.cu) over work items of PD_SEG_CHUNK grid positions
// that never cross a scan boundary.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define BATCH_BLOCKS (device_sms() * 8)

__device__ __forceinline__ int pack_scan_of(const PackScan* sc, int nsc, int w) {
    int lo = 0, hi = nsc - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (sc[mid].chunk0 <= w) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// ------------------------------------------------------------------ packing
__global__ void pack_bbox_kernel(PackScan* sc, int nsc, int nchunks) {
    __shared__ int s_i;
    __shared__ long long s_lo, s_hi;
    __shared__ int red[6][32];
    for (int w = blockIdx.x; w < nchunks; w += gridDim.x) {
        if (threadIdx.x == 0) {
            int i = pack_scan_of(sc, nsc, w);
            long long lo = (long long)(w - sc[i].chunk0) * PD_SEG_CHUNK;
            long long hi = lo + PD_SEG_CHUNK < sc[i].n ? lo + PD_SEG_CHUNK : sc[i].n;
            s_i = i;
            s_lo = lo;
            s_hi = hi;
        }
        __syncthreads();
        const int i = s_i;
        const int32_t* x = sc[i].xyz;
        int v[6] = {0x7fffffff, 0x7fffffff, 0x7fffffff, (int)0x80000000, (int)0x80000000,
                    (int)0x80000000};
        for (long long j = s_lo + threadIdx.x; j < s_hi; j += blockDim.x) {
            for (int a = 0; a < 3; a++) {
                int c = x[3 * j + a];
                v[a] = c < v[a] ? c : v[a];
                v[3 + a] = c > v[3 + a] ? c : v[3 + a];
            }
        }
        for (int o = 16; o; o >>= 1)
            for (int a = 0; a < 6; a++) {
                int u = __shfl_xor_sync(0xffffffffu, v[a], o);
                v[a] = a < 3 ? (u < v[a] ? u : v[a]) : (u > v[a] ? u : v[a]);
            }
        const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane == 0)
            for (int a = 0; a < 6; a++) red[a][wp] = v[a];
        __syncthreads();
        if (threadIdx.x < 6) {
            const int a = threadIdx.x;
            int r = red[a][0];
            for (int q = 1; q < (int)(blockDim.x >> 5); q++)
                r = a < 3 ? (red[a][q] < r ? red[a][q] : r) : (red[a][q] > r ? red[a][q] : r);
            if (a < 3) atomicMin(&sc[i].bb[a], r);
            else atomicMax(&sc[i].bb[a], r);
        }
        __syncthreads();
    }
}

__global__ void pack_copy_kernel(const PackScan* sc, int nsc, int nchunks, int32_t* out_xyz,
                                 uint8_t* out_rgb, float* out_nrm) {
    for (int w = blockIdx.x; w < nchunks; w += gridDim.x) {
        const int i = pack_scan_of(sc, nsc, w);  // uniform over the block
        const PackScan& s = sc[i];
        const long long lo = (long long)(w - s.chunk0) * PD_SEG_CHUNK;
        const long long hi = lo + PD_SEG_CHUNK < s.n ? lo + PD_SEG_CHUNK : s.n;
        for (long long j = lo + threadIdx.x; j < hi; j += blockDim.x) {
            const long long o = s.off + j;
            out_xyz[3 * o + 0] = s.xyz[3 * j + 0] + s.ox;
            out_xyz[3 * o + 1] = s.xyz[3 * j + 1] + s.oy;
            out_xyz[3 * o + 2] = s.xyz[3 * j + 2] + s.oz;
            if (out_rgb) {
                out_rgb[3 * o + 0] = s.rgb[3 * j + 0];
                out_rgb[3 * o + 1] = s.rgb[3 * j + 1];
                out_rgb[3 * o + 2] = s.rgb[3 * j + 2];
            }
            if (out_nrm) {
                out_nrm[3 * o + 0] = s.nrm[3 * j + 0];
                out_nrm[3 * o + 1] = s.nrm[3 * j + 1];
                out_nrm[3 * o + 2] = s.nrm[3 * j + 2];
            }
        }
    }
}

__global__ void pack_unpack_kernel(const PackScan* sc, int nsc, int nchunks,
                                   const uint8_t* __restrict__ keep) {
    for (int w = blockIdx.x; w < nchunks; w += gridDim.x) {
        const int i = pack_scan_of(sc, nsc, w);
        const PackScan& s = sc[i];
        const long long lo = (long long)(w - s.chunk0) * PD_SEG_CHUNK;
        const long long hi = lo + PD_SEG_CHUNK < s.n ? lo + PD_SEG_CHUNK : s.n;
        for (long long j = lo + threadIdx.x; j < hi; j += blockDim.x) s.keep[j] = keep[s.off + j];
    }
}

// ------------------------------------------------------------------ scan ranges
// b of scan i = the first grid position whose tile index is >= i (tile
// indices never decrease along the Morton order).
__global__ void seg_ranges_kernel(const int4* __restrict__ pos, int64_t ng, SegDev* seg,
                                  int nseg, int shift) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > nseg) return;
    long long lo = 0, hi = ng;
    while (lo < hi) {
        long long mid = (lo + hi) >> 1;
        if (seg_of(pos[mid], shift) >= i) hi = mid;
        else lo = mid + 1;
    }
    if (i < nseg) seg[i].b = (int)lo;
    if (i > 0) seg[i - 1].e = (int)lo;
}

// chunk0[i] = work items of the scans before i, items[w] = the scan of work
// item w; one block of 1024 threads.
__global__ void seg_chunks_kernel(const SegDev* seg, int nseg, int* chunk0, int* items) {
    __shared__ int part[1024];
    const int t = threadIdx.x;
    const int per = (nseg + 1023) / 1024;
    int loc[PD_SEG_MAX / 1024];
    int sum = 0;
    for (int j = 0; j < per; j++) {
        const int i = t * per + j;
        int c = 0;
        if (i < nseg) c = (seg[i].e - seg[i].b + PD_SEG_CHUNK - 1) / PD_SEG_CHUNK;
        loc[j] = c;
        sum += c;
    }
    part[t] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        int v = t >= o ? part[t - o] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int acc = t ? part[t - 1] : 0;
    for (int j = 0; j < per; j++) {
        const int i = t * per + j;
        if (i < nseg) {
            chunk0[i] = acc;
            for (int w = 0; w < loc[j]; w++) items[acc + w] = i;
        }
        acc += loc[j];
    }
    if (t == 1023) chunk0[nseg] = part[1023];
}

// ------------------------------------------------------------------ per-scan counts
__global__ void seg_count_kernel(const uint8_t* __restrict__ flag, const int4* __restrict__ pos,
                                 int64_t ng, int shift, unsigned long long* cnt) {
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= ng || !flag[s]) return;
    atomicAdd(&cnt[seg_of(pos[s], shift)], 1ull);
}

__global__ void seg_accept_kernel(const u64* __restrict__ prim, const int4* __restrict__ pos,
                                  const uint8_t* __restrict__ alive, int64_t ng,
                                  const RoundDev* rd, uint8_t* inP, int* cand, int* ncand) {
    const int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= ng || !alive[s]) return;
    const int4 p = pos[s];
    u64 tp;
    int ti;
    round_tau(rd, p, tp, ti);
    if (key_gt(tp, ti, prim[s], p.w)) return;
    inP[s] = 1;
    cand[atomicAdd(ncand, 1)] = (int)s;
}

// ------------------------------------------------------------------ launchers
static int grid_for(long long items) {
    long long b = items < BATCH_BLOCKS ? items : BATCH_BLOCKS;
    return b < 1 ? 1 : (int)b;
}

cudaError_t pack_launch_bbox(PackScan* sc, int nsc, int nchunks, cudaStream_t st) {
    pack_bbox_kernel<<<grid_for(nchunks), 256, 0, st>>>(sc, nsc, nchunks); note_launch();
    return cudaGetLastError();
}
cudaError_t pack_launch_copy(const PackScan* sc, int nsc, int nchunks, int32_t* out_xyz,
                             uint8_t* out_rgb, float* out_nrm, cudaStream_t st) {
    pack_copy_kernel<<<grid_for(nchunks), 256, 0, st>>>(sc, nsc, nchunks, out_xyz, out_rgb,
                                                        out_nrm); note_launch();
    return cudaGetLastError();
}
cudaError_t pack_launch_unpack(const PackScan* sc, int nsc, int nchunks, const uint8_t* keep,
                               cudaStream_t st) {
    pack_unpack_kernel<<<grid_for(nchunks), 256, 0, st>>>(sc, nsc, nchunks, keep); note_launch();
    return cudaGetLastError();
}
cudaError_t seg_launch_ranges(const int4* pos, int64_t ng, SegDev* seg, int* chunk0, int* items,
                              int nseg, int shift, cudaStream_t st) {
    if (nseg < 1 || nseg > PD_SEG_MAX) return cudaErrorInvalidValue;
    seg_ranges_kernel<<<(nseg + 1 + 255) / 256, 256, 0, st>>>(pos, ng, seg, nseg, shift); note_launch();
    seg_chunks_kernel<<<1, 1024, 0, st>>>(seg, nseg, chunk0, items); note_launch();
    return cudaGetLastError();
}
cudaError_t seg_launch_count(const uint8_t* flag, const int4* pos, int64_t ng, int shift,
                             unsigned long long* cnt, cudaStream_t st) {
    if (ng < 1) return cudaSuccess;
    seg_count_kernel<<<(unsigned)((ng + 255) / 256), 256, 0, st>>>(flag, pos, ng, shift, cnt); note_launch();
    return cudaGetLastError();
}
cudaError_t seg_launch_accept(const u64* prim, const int4* pos, const uint8_t* alive, int64_t ng,
                              const RoundDev* rd, uint8_t* inP, int* cand, int* ncand,
                              cudaStream_t st) {
    if (ng < 1) return cudaSuccess;
    seg_accept_kernel<<<(unsigned)((ng + 255) / 256), 256, 0, st>>>(prim, pos, alive, ng, rd, inP,
                                                                    cand, ncand); note_launch();
    return cudaGetLastError();
}

}  // namespace pd
