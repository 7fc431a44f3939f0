// pd_kernels.h -- host-side launchers of the libpd kernels (internal).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "pd_internal.cuh"

namespace pd {

typedef unsigned long long u64;

// Scratch memory handed to launchers by the caller (the grid object).
struct Scratch {
    void* (*alloc)(void* self, size_t bytes);
    void (*free)(void* self, void* p);
    void* self;
    void* get(size_t bytes) const { return alloc(self, bytes); }
    void put(void* p) const { free(self, p); }
};

// ---------------------------------------------------------------- grid.cu
cudaError_t launch_bbox(const int32_t* xyz, int64_t n, int* out6, cudaStream_t st);
// Morton codes ((x - origin) >> shift, `bits` bits) in ascending order, equal ones
// in input order, in keys; their input indices in vals.
cudaError_t sort_points(const int32_t* xyz, int64_t n, int3 origin, int shift, int bits, u64* keys,
                        uint32_t* vals, const Scratch& s, cudaStream_t st);
cudaError_t exclusive_scan_u32(uint32_t* data, int64_t len, const Scratch& s, cudaStream_t st);
cudaError_t launch_gather(const int32_t* xyz, const uint8_t* rgb, const float* nrm,
                          const uint32_t* perm, int64_t n, int4* pos, uchar4* rgb_s,
                          float4* nrm_s, cudaStream_t st);
cudaError_t launch_gather_nrm(const float* nrm, const int4* pos, int64_t n, float4* out,
                              cudaStream_t st);
cudaError_t launch_leaf_levels(const u64* code, int64_t n, int T, int B, uint8_t* leaf,
                               cudaStream_t st);
cudaError_t launch_node_count(const u64* code, const uint8_t* leaf, int64_t n, int B,
                              unsigned long long* count, cudaStream_t st);
cudaError_t launch_node_insert(const u64* code, const uint8_t* leaf, int64_t n, int B,
                               HashSlot* tab, u64 mask, cudaStream_t st);
// Groups of <= 32 points of one leaf, for every point (full mode).
cudaError_t launch_leaf_groups(const GridView& g, int64_t n, int4* groups, int* ngroups,
                               cudaStream_t st);
// Stable compaction: out = ascending s with flag[s] != 0; *count on device.
cudaError_t stable_compact(const uint8_t* flag, int64_t n, int* out, int* count,
                           const Scratch& s, cudaStream_t st);

// ---------------------------------------------------------------- quality.cu
#define PD_QUALITY_MAXR 32
// Per retained point: neighbour counts within each radius (r2: ascending
// squared radii, nr <= PD_QUALITY_MAXR, rmax the largest radius) over the leaf
// groups of the grid, from the 3x3x3 cells of level L (cell edge >= the largest
// radius); per radius the sums of N and N^2 and a histogram of N with H bins
// (the top bin holds N >= H - 1).  next: one int of device scratch.
cudaError_t launch_radius_counts(const GridView& g, const int4* groups, int ngroups, int L,
                                 int rmax, const u64* r2, int nr, u64* sum_n, u64* sum_n2,
                                 uint32_t* hist, int H, int* next, cudaStream_t st);
// Per block of 256 points: least nearest squared distance and sum of sqrt.
cudaError_t launch_spacing(const u64* rk2, int64_t n, u64* bmin, double* bsum, cudaStream_t st);
// out[t] = xyz row list[t] for t < *count (cap >= *count rows are reserved).
cudaError_t launch_take_xyz(const int* list, const int* count, int64_t cap, const int32_t* xyz,
                            int32_t* out, cudaStream_t st);

// ---------------------------------------------------------------- round state
#define PD_FIX_ITERS 6     // fixpoint launches of a k = 1 round (the most), each of up to
#define PD_FIX_ITERS_KK 3  //   PD_FIX_INNER sweeps, and of a k >= 2 round (danger pairs)
#define PD_FIX_INNER 16

// ---------------------------------------------------------------- packed batches
// Many independent scans decimated in one grid (batch.cu).  Scan i is moved
// into the aligned cube ("tile") of edge 2^shift mm whose Morton index is i;
// tiles are far enough apart that no neighbour search reaches another scan,
// and every scan occupies one contiguous range of the Morton order.  The
// removal threshold of a round (R2) is selected per scan.
#define PD_SEG_MAX 4096      // scans of one packed batch (16 tiles per axis)
#define PD_SEG_CHUNK 4096    // grid positions per work item of the per-scan passes
struct SegDev {
    long long live, m, need, rank;
    unsigned long long tau_prim;  // this round's threshold (~0: nothing to remove)
    int tau_idx;
    int done;                     // selection finished for this round
    unsigned pre[8];
    int len;                      // selection list: [b, b + len) of the list buffers
    int b, e;                     // the scan's grid positions [b, e)
    unsigned ticket;              // blocks that finished a pass over the scan (0 between)
};

// Per-round control block in device memory (read by the host once per round).
struct RoundDev {
    long long live, m, need, rank;
    double band, band_max;
    unsigned long long removed, cap_over;
    unsigned long long tot_requery, tot_filtered, tot_sources, tot_lambda;
    unsigned long long tau_prim;
    int tau_idx;
    int done;
    unsigned pre[8];
    int len;                   // length of the selection list
    unsigned ticket;           // blocks that finished a launch (0 between launches)
    int finished;              // the round's counts are added up
    int ncand, nslow, nsrc, npairs, overflow;
    int nreq, nfq, nlq;  // this round's re-searches, filtered and lambda searches
    int take_src, take_filt, take_req;  // next item of those lists, past each warp's first
    int ndep;  // k = 1: candidates with a shell member of larger input index
    int changed[PD_FIX_ITERS];
    int fix_unconverged;
    int density_k1;
    int density;    // no colour or orientation weights: any band gives the same result
    int band_mode;  // 0: shrink on overflow only; 1: also on poor yield
    int fix_iters;  // device fixpoint sweeps per round (<= PD_FIX_ITERS)
    // packed batch (NULL seg: one scan).  Then tau_prim above is the least
    // threshold over the scans (a prefilter) and each point takes its own
    // scan's threshold.
    SegDev* seg;
    const int* seg_chunk0;  // nseg + 1 prefix counts of PD_SEG_CHUNK work items
    int nseg, seg_shift;
    int seg_rank_one;       // select each scan's largest key only (host settle)
};

#ifdef __CUDACC__
// The scan of a packed batch that holds grid point p (its tile's Morton index).
__device__ __forceinline__ int seg_of(int4 p, int shift) {
    return (int)morton3((uint32_t)p.x >> shift, (uint32_t)p.y >> shift, (uint32_t)p.z >> shift);
}
// The removal threshold of the round that applies to grid point p.
__device__ __forceinline__ void round_tau(const RoundDev* rd, int4 p, unsigned long long& tp,
                                          int& ti) {
    if (rd->seg) {
        const SegDev& s = rd->seg[seg_of(p, rd->seg_shift)];
        tp = s.tau_prim;
        ti = s.tau_idx;
    } else {
        tp = rd->tau_prim;
        ti = rd->tau_idx;
    }
}
#endif

struct SelBuffers {
    u64* p;  // the selection list: keys and input indices
    int* i;
    uint32_t* hist;  // 4096 words, zero between launches
};

// ---------------------------------------------------------------- knn.cu
enum { FILT_NONE = 0, FILT_BELOW_SELF = 1, FILT_BELOW_TAU = 2 };
#define PD_PAIR_SLOTS 64

struct KnnArgs {
    const int4* groups;
    int ngroups;
    const uint8_t* alive;     // NULL = every point live (launch_knn only)
    const u64* prim;          // keys (filtered searches)
    const RoundDev* rd;       // round state: the thresholds of the lambda searches
    const uint8_t* qflag;     // when set, only flagged points of each group are queried
    int k;
    int S;                    // stored neighbours (template width)
    int density_k1;           // integer-ordered k = 1 density cost
    int term;
    double weight;
    const uchar4* rgb;
    const float4* nrm;
    // outputs (full / re-query mode)
    int* nbr;                 // n x S Morton positions
    int* nbr0_out;            // optional: the first stored entry again, one int per point
    u64* prim_out;            // key primary
    u64* rk2_out;             // k-th squared distance
    uint8_t* flg_out;
    u64* hz_out;              // horizon: S-th stored squared distance (~0 if fewer)
    double* cost_out;         // cost in Morton order (optional)
    unsigned long long* pairs_out;  // optional: + (query, candidate) pairs scanned, spread
                                    //   over PD_PAIR_SLOTS counters (their sum is the count)
    int r_exact;              // full searches: nearest entries that must be exact
                              //   (0 = all S; the k = 1 density cost keeps the
                              //   rest below the horizon)
    // launch_knn_queries: the queries (Morton positions), counts on the device.
    // qlist2 NULL: full searches of qlist.  Otherwise filtered searches: the
    // points of qlist whose cost over smaller keys equals their own join the
    // candidates (inP, its bitmap inPb, cand, *ncand); lam_out of those of qlist2
    // takes the k-th squared distance over keys below the threshold.
    RoundDev* finish;         // full searches: the round to add up
    int ordered;              // equal distances in Morton order (term 0; with a term they are
                              //   always in input order)
    int* take;                // optional, zero: a short list's queries are taken one by one
    const int* qlist;
    const int* qcount;
    const int* qlist2;
    const int* qcount2;
    u64* lam_out;
    uint8_t* inP;
    uint32_t* inPb;
    int* cand;
    int* ncand;
    const u64* cmin;          // filtered searches: least live key primary of every aligned
                              //   32-position chunk (chunks above the threshold are skipped)
};
// Full searches of every point (a.qflag: of the flagged ones), a warp per leaf
// group, then a warp for each query that is left.  rest: n ints and nrest: one
// int, device scratch.
cudaError_t launch_knn(const GridView& g, const KnnArgs& a, int64_t n, int* rest, int* nrest,
                       cudaStream_t st);
// Searches of the listed queries, one warp each; at most cap of them.
cudaError_t launch_knn_queries(const GridView& g, const KnnArgs& a, int64_t cap, cudaStream_t st);
// Internal neighbour-weight term: unit weights with equal distances ordered by
// input index (the normals' 16-NN order).
#define PD_TERM_INDEX_TIE 3

// ---------------------------------------------------------------- rounds_dev.cu
// Sizes of launches that walk lists whose length the device knows: n / per
// blocks, at most `per_sm` per multiprocessor (an idle block costs about as
// much as a little work).
inline unsigned list_blocks(int64_t n, int64_t per, int per_sm) {
    int64_t b = n / per + 1;
    const int64_t lim = (int64_t)device_sms() * per_sm;
    return (unsigned)(b < lim ? b : lim);
}
// The candidate band of the next round (k >= 2 and weighted costs) from this
// round's counts; the same arithmetic runs on the device after a normal round
// and on the host after a round it settled.
//   density: any band gives the same result.  A poor yield then never narrows
// it below PD_BAND_LEAST keys: a round costs its passes over the cloud whatever
// it removes, and a dense spot without lower keys nearby yields few points of a
// wide band but fewer still of a narrow one.  Only candidate lists that
// overflow (cap_over, which make the danger test expensive) narrow it further.
// Without a floor, with 256, 1024, 4096 keys (k = 4 unless stated): 31M site points
// 831, 815, 781 ms; 2.4M outdoor, k = 2, 65.9, 63.3, 60.8; 12M site 150, 147, 148, 167;
// four outdoor scans of 9.8M 122 to 125, 120 to 124, 121 to 128, 166; room scans within
// 2 % of each other.
#define PD_BAND_LEAST 1024
__device__ __host__ inline double next_band(double band, double band_max, int band_mode,
                                            int density, long long live,
                                            unsigned long long cap_over, long long ncand,
                                            unsigned long long removed) {
    bool shrink = cap_over != 0;
    double grow = 1.5;
    if (band_mode == 1) {
        double yield = ncand > 0 ? (double)removed / ncand : 1.0;
        const bool least = density && band * (double)live <= PD_BAND_LEAST;
        shrink = shrink || (yield < 0.5 && !least);
        grow = yield > 0.8 ? (density ? 1.5 : 1.25) : 1.0;
        if (density && least && !shrink) grow = 1.5;
    }
    double b = shrink ? band * 0.5 : band * grow;
    if (b > band_max) b = band_max;
    if (b < 1e-7) b = 1e-7;
    return b;
}
#ifdef __CUDACC__
// Adds up a round once its removals and re-search list are complete; one
// thread of the re-search launch calls it.
__device__ inline void round_finish(RoundDev* rd) {
    if (rd->seg) rd->tau_prim = ~0ull;  // the next selection lowers it
    if (rd->finished) return;  // the second update of a round settled on the host
    rd->finished = 1;
    rd->live -= (long long)rd->removed;
    rd->tot_sources += (unsigned long long)rd->nsrc;
    rd->tot_filtered += (unsigned long long)rd->nfq;
    rd->tot_lambda += (unsigned long long)rd->nlq;
    rd->tot_requery += (unsigned long long)rd->nreq;
    // a held round (settled on the host) updates its band there, from the
    // points it finally removes: the band must not depend on whether the
    // device fixpoint happened to converge within its sweeps
    if (!rd->density_k1 && !(rd->overflow || rd->fix_unconverged)) {
        rd->band = next_band(rd->band, rd->band_max, rd->band_mode, rd->density, rd->live,
                             rd->cap_over, rd->ncand, rd->removed);
    }
}
#endif
// select.cu: the round's threshold (rank from the live count, target and
// band), and the round's counters opened.  long_list: the list of the keys that
// agree in their leading digits is walked by the whole grid, not by one cluster
// (the caller's guess from the round before, PD_SEL_LONG; either is correct).
// Selections of a gridded cloud's 3 rounds, cluster and whole grid: lists of 64k keys
// 0.120 and 0.134 ms, 166k 0.165 and 0.137, 343k 0.241 and 0.143, 2.0M 0.97 and 0.21.
// In a first round the list is not known: on a cloud whose keys differ the whole
// grid's five further launches cost 0.02 to 0.03 ms, on a gridded one the cluster
// 0.25 ms at 0.7M points and 5 of 16 ms at 8.0M (PD_SEL_FIRST).
#define PD_SEL_LONG 131072
#define PD_SEL_FIRST (1 << 20)
cudaError_t round_launch_select(const u64* prim, const int4* pos, const uint8_t* alive, int64_t n,
                                SelBuffers& b, bool long_list, RoundDev* rd, cudaStream_t st);
// dep: list of the candidates that have a shell member of larger input index
// (the only ones condition (B) can reject; the fixpoint sweeps walk it).
// nbr0: the first stored entries apart (may be NULL).
cudaError_t round_launch_k1(const GridView& g, const u64* prim, const uint8_t* alive,
                            const int* nbr, const int* nbr0, const uint8_t* flg, const u64* rk2,
                            int64_t n, int S, RoundDev* rd, uint8_t* inP, uint8_t* rej, int* cand,
                            int* slow, int* dep, int fix_iters, cudaStream_t st);
// inPb: bitmap of inP over the Morton positions.
cudaError_t round_launch_danger(const GridView& g, const int* src, const u64* prim,
                                const uint8_t* alive, const uint32_t* inPb, uint8_t* rej,
                                const u64* lam, const int* nbr, int S, int k, int2* pairs,
                                int pair_cap, int64_t n, RoundDev* rd, cudaStream_t st);
cudaError_t round_launch_pairs_fix(const int2* pairs, int pair_cap, const uint8_t* inP,
                                   uint8_t* rej, int64_t n, RoundDev* rd, cudaStream_t st);
cudaError_t round_launch_remove(const int* cand, uint8_t* inP, uint8_t* rej, uint8_t* alive,
                                int64_t n, RoundDev* rd, cudaStream_t st);
// Lists (list[0 .. rd->nreq)) the live points that lost one of their first
// kchk stored neighbours.
cudaError_t round_launch_dirty(const uint8_t* alive, const int* nbr, int64_t n, int S, int kchk,
                               int* list, RoundDev* rd, cudaStream_t st);
struct BufView {  // the k+b neighbour buffer of every point
    const int4* pos;
    u64* prim;
    int* nbr;
    int* nbr0;  // optional (k = 1 density): nbr[s * S] kept apart, read coalesced
    u64* rk2;
    uint8_t* flg;
    u64* hz;
    const uchar4* rgb;
    const float4* nrm;
    int term;
    double weight;
};
// k = 1 density cost: absorb removals in the stored nearest entries (the
// shell at the new nearest distance must lie below the search horizon);
// list[0 .. rd->nreq) takes the points that need a new search.
cudaError_t round_launch_k1_update(const BufView& b, const uint8_t* alive, int64_t n, int S,
                                   int* list, RoundDev* rd, cudaStream_t st);
cudaError_t round_launch_kk_update(const BufView& b, const uint8_t* alive, int64_t n, int S, int k,
                                   int* list, RoundDev* rd, cudaStream_t st);
// Candidates (inP, its bitmap, cand), danger sources (src, lam) and the lists
// of the searches that the stored neighbours do not settle (fq, lq); cmin as
// in KnnArgs.
cudaError_t round_launch_kk_cand2(const BufView& b, const uint8_t* alive, int64_t n, int S, int k,
                                  RoundDev* rd, uint8_t* inP, uint32_t* inPb, int* cand, int* fq,
                                  int* lq, u64* lam, int* src, u64* cmin, cudaStream_t st);
}  // namespace pd

// ---------------------------------------------------------------- normals.cu
struct pd_ctx;
struct pd_grid;
namespace pd {
struct GridNbrs {
    const int4* pos;
    const int* nbr;  // n x S Morton positions, nearest first, -1 past the found ones
    int S;
    int64_t n;
    pd_ctx* ctx;
};
// capi.cu: context allocator, error text, and the 16-NN pass over a grid
void* api_alloc(pd_ctx* c, size_t bytes, cudaStream_t st);
void api_free(pd_ctx* c, void* p, cudaStream_t st);
void api_error(pd_ctx* c, const char* what, long long v);
int grid_knn16(pd_grid* g, cudaStream_t st, GridNbrs* out);
cudaError_t launch_features(const int4* pos, const int* nbr, int S, int64_t n, uint16_t* feat,
                            float* pca, uint8_t* valid, cudaStream_t st);
cudaError_t launch_mlp_forward(const float* prm, const uint16_t* feat, int64_t n, float* outn,
                               float* onorm, cudaStream_t st);
// Partials: mlp_backward_part_floats() floats of scratch; the gradient is
// reduced over blocks in a fixed order (deterministic).
int64_t mlp_backward_part_floats();
// Mean loss and gradient over rows 0..n-1.
cudaError_t launch_mlp_gradient(const float* prm, const uint16_t* feat, const float* labels,
                                int64_t n, float* grad, float* loss, float* part,
                                cudaStream_t st);
// Step t (1-based) of Adam over b rows sampled from the pool.  overlap: the
// launch ahead in the stream is the step before (its tail may overlap).
cudaError_t launch_mlp_step(float* prm, float* m, float* v, const uint16_t* feat, const int* pool,
                            int64_t npool, u64 seed, int t, const float* labels, int64_t b,
                            float lr, float* loss, float* part, bool overlap, cudaStream_t st);
cudaError_t launch_mlp_init(float* prm, u64 seed, cudaStream_t st);
cudaError_t launch_normal_fallback(const float* mlp, const float* onorm, const float* pca,
                                   int64_t n, float min_norm, float* out, cudaStream_t st);
// ---------------------------------------------------------------- wup.cu
#define WUP_BATCH 4  // removal rounds between two host reads
struct WupDev {
    int count[2];     // candidates in either list
    unsigned ticket;
    unsigned long long removed[WUP_BATCH];
};
struct WupBuffers {
    uint8_t *cand, *beaten;  // per point: a candidate; one of smaller key than an adjacent one
    int* list[2];
    WupDev* wd;
    void* block_least;       // wup_least_bytes() of scratch
};
int64_t wup_blocks();
size_t wup_least_bytes();
cudaError_t wup_launch_list(const BufView& b, const uint8_t* alive, int64_t n, RoundDev* rd,
                            const WupBuffers& w, cudaStream_t st);
cudaError_t wup_launch_rounds(const BufView& b, uint8_t* alive, int64_t most, int S, int k,
                              const RoundDev* rd, const WupBuffers& w, cudaStream_t st);

// ---------------------------------------------------------------- batch.cu
// One scan of a packed batch (device array, host-built): its caller-owned
// buffers, its first packed position and work item, and the per-axis offset
// that moves it into its tile (packed = input + o).
struct PackScan {
    const int32_t* xyz;
    const uint8_t* rgb;
    const float* nrm;
    uint8_t* keep;
    long long n, off;
    int chunk0;
    int ox, oy, oz;
    int bb[6];  // bounding box (min x, y, z, max x, y, z), from pack_launch_bbox
};
// Bounding boxes of every scan (sc[i].bb, preset to empty boxes by the caller).
cudaError_t pack_launch_bbox(PackScan* sc, int nsc, int nchunks, cudaStream_t st);
// Packed coordinates (and colours, normals where out_rgb / out_nrm are set).
cudaError_t pack_launch_copy(const PackScan* sc, int nsc, int nchunks, int32_t* out_xyz,
                             uint8_t* out_rgb, float* out_nrm, cudaStream_t st);
// Every scan's keep mask from the packed one.
cudaError_t pack_launch_unpack(const PackScan* sc, int nsc, int nchunks, const uint8_t* keep,
                               cudaStream_t st);
// Grid ranges [b, e) of every scan, the prefix counts of their work items
// (chunk0[0..nseg]) and the scan of every work item (items: ng / PD_SEG_CHUNK
// + nseg entries at least), from the Morton-ordered positions.
cudaError_t seg_launch_ranges(const int4* pos, int64_t ng, SegDev* seg, int* chunk0, int* items,
                              int nseg, int shift, cudaStream_t st);
// Per-scan selection of the round's threshold (R2): every scan's rank-th
// largest live key, rank from its live count, target and the band.  hist:
// nseg x 4096 words, zero on entry and on return.
cudaError_t seg_launch_select(const u64* prim, const int4* pos, const uint8_t* alive, int64_t ng,
                              SelBuffers& b, uint32_t* hist, RoundDev* rd, SegDev* seg,
                              const int* items, int nseg, cudaStream_t st);
// cnt[scan] += flagged points of the scan.
cudaError_t seg_launch_count(const uint8_t* flag, const int4* pos, int64_t ng, int shift,
                             unsigned long long* cnt, cudaStream_t st);
// Candidates: every live point whose key reaches its scan's threshold.
cudaError_t seg_launch_accept(const u64* prim, const int4* pos, const uint8_t* alive, int64_t ng,
                              const RoundDev* rd, uint8_t* inP, int* cand, int* ncand,
                              cudaStream_t st);

}  // namespace pd
