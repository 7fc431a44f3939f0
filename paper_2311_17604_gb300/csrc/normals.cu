// normals.cu -- unit normals for the orientation term (Eq. 13): PCA of the 16
// nearest neighbours, and a small network that maps the 16 neighbour offsets
// to a normal, trained on the PCA normals by the kernels below.
//
// The paper takes oriented input as given (section "Additional cost terms")
// and names no estimator; these kernels supply the normals.
//
// Parameter layout (float32, PD_MLP_PARAMS values):
//   W1[64][48] b1[64] W2[64][64] b2[64] W3[3][64] b3[3]
// Forward: h1 = relu(x W1^T + b1), h2 = relu(h1 W2^T + b2), o = h2 W3^T + b3,
// normal = o / |o|.  x, W1..W3, h1 and h2 are bfloat16; products accumulate
// in float32 on the tensor cores (mma.sync m16n8k16, bf16 in, f32 out).
// Loss per row: 1 - (u . y)^2 with u = o / |o| (labels are unoriented).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pd.h"
#include "../../include/pd_normals.h"
#include "pd_internal.cuh"
#include "pd_kernels.h"

namespace pd {

#define NF PD_MLP_IN
#define NH PD_MLP_HIDDEN
#define O_W1 0
#define O_B1 (O_W1 + NH * NF)
#define O_W2 (O_B1 + NH)
#define O_B2 (O_W2 + NH * NH)
#define O_W3 (O_B2 + NH)
#define O_B3 (O_W3 + 3 * NH)
#define N_PARAMS (O_B3 + 3)
static_assert(N_PARAMS == PD_MLP_PARAMS, "parameter count");
static_assert(NF == 3 * PD_NORMAL_K, "feature width");

// ------------------------------------------------------------------ PCA + features
// Unit eigenvector of the smallest eigenvalue of the symmetric matrix
// (c00 c01 c02 / . c11 c12 / . . c22): the eigenvalue from the trigonometric
// closed form of O. K. Smith (CACM 4(4), 1961), the eigenvector as the longest
// cross product of two rows of (A - lambda I).  False when that product's
// length is <= 1e-6 trace(A)^2 (the smallest eigenvalue is not simple).
// *lmid receives the middle eigenvalue.
__device__ inline bool smallest_eigvec(double a00, double a01, double a02, double a11,
                                       double a12, double a22, double out[3], double* lmid) {
    double p1 = a01 * a01 + a02 * a02 + a12 * a12;
    double q = (a00 + a11 + a22) / 3.0;
    double lam;
    if (p1 == 0.0) {
        lam = fmin(a00, fmin(a11, a22));
        *lmid = a00 + a11 + a22 - lam - fmax(a00, fmax(a11, a22));
    } else {
        double e0 = a00 - q, e1 = a11 - q, e2 = a22 - q;
        double p = sqrt((e0 * e0 + e1 * e1 + e2 * e2 + 2.0 * p1) / 6.0);
        double b00 = e0 / p, b11 = e1 / p, b22 = e2 / p;
        double b01 = a01 / p, b02 = a02 / p, b12 = a12 / p;
        double det = b00 * (b11 * b22 - b12 * b12) - b01 * (b01 * b22 - b12 * b02) +
                     b02 * (b01 * b12 - b11 * b02);
        double r = fmin(1.0, fmax(-1.0, det / 2.0));
        // eigenvalues q + 2p cos(acos(r)/3 + 2 pi j / 3); j = 1 is the smallest
        double phi = acos(r) / 3.0;
        lam = q + 2.0 * p * cos(phi + 2.0943951023931957);
        *lmid = q + 2.0 * p * cos(phi + 4.1887902047863905);  // j = 2: the middle one
    }
    double r0x = a00 - lam, r0y = a01, r0z = a02;
    double r1x = a01, r1y = a11 - lam, r1z = a12;
    double r2x = a02, r2y = a12, r2z = a22 - lam;
    double c0x = r0y * r1z - r0z * r1y, c0y = r0z * r1x - r0x * r1z, c0z = r0x * r1y - r0y * r1x;
    double c1x = r0y * r2z - r0z * r2y, c1y = r0z * r2x - r0x * r2z, c1z = r0x * r2y - r0y * r2x;
    double c2x = r1y * r2z - r1z * r2y, c2y = r1z * r2x - r1x * r2z, c2z = r1x * r2y - r1y * r2x;
    double n0 = c0x * c0x + c0y * c0y + c0z * c0z;
    double n1 = c1x * c1x + c1y * c1y + c1z * c1z;
    double n2 = c2x * c2x + c2y * c2y + c2z * c2z;
    double best = n0, bx = c0x, by = c0y, bz = c0z;
    if (n1 > best) {
        best = n1;
        bx = c1x;
        by = c1y;
        bz = c1z;
    }
    if (n2 > best) {
        best = n2;
        bx = c2x;
        by = c2y;
        bz = c2z;
    }
    double tr = a00 + a11 + a22;
    if (!(best > 1e-12 * (tr * tr) * (tr * tr))) return false;
    double inv = 1.0 / sqrt(best);
    out[0] = bx * inv;
    out[1] = by * inv;
    out[2] = bz * inv;
    return true;
}

// The bfloat16 nearest to v / rms.  binary64 division is a long sequence on a
// pipe this GPU has little of (48 of them were most of the kernel), so the
// quotient is taken in binary32 from the reciprocal first: it is within 2^-21 of
// the exact one, and only where that leaves the rounding open (within 16 units
// in the last place of the midpoint of two bfloat16 values, one case in 2000)
// does the division run (2.0M points: 4.16 -> 1.15 ms).
__device__ __noinline__ uint32_t ratio_bf16_exact(int v, double rms) {
    return (uint32_t)__bfloat16_as_ushort(__double2bfloat16((double)v / rms));
}
__device__ __forceinline__ uint32_t ratio_bf16(int v, float inv, double rms) {
    const float f = (float)v * inv;
    const uint32_t u = __float_as_uint(f), low = u & 0xffffu;
    if (low - 0x7ff0u <= 0x20u || (v >= 1 << 24) || (v <= -(1 << 24))) return ratio_bf16_exact(v, rms);
    return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(f));
}

// One thread per point (Morton position s).  Offsets are exact int32; the
// moment sums are exact int64, so the covariance scaled by m^2 is the exact
// integer m * sum(u v) - sum(u) sum(v) before its conversion to binary64.
__global__ void __launch_bounds__(128)
    features_kernel(const int4* pos, const int* nbr, int S, int64_t n, uint4* feat, float* pca,
                    uint8_t* valid) {
    chain();
    int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (s >= n) return;
    int4 p = pos[s];
    int64_t out = p.w;
    int ox[PD_NORMAL_K], oy[PD_NORMAL_K], oz[PD_NORMAL_K];
    int m = 0;
    long long sx = 0, sy = 0, sz = 0, sxx = 0, sxy = 0, sxz = 0, syy = 0, syz = 0, szz = 0;
#pragma unroll
    for (int i = 0; i < PD_NORMAL_K; i++) {
        int x = i < S ? nbr[s * S + i] : -1;
        int4 q = x >= 0 ? pos[x] : p;
        int dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
        ox[i] = dx;
        oy[i] = dy;
        oz[i] = dz;
        m += x >= 0;
        sx += dx;
        sy += dy;
        sz += dz;
        sxx += (long long)dx * dx;
        sxy += (long long)dx * dy;
        sxz += (long long)dx * dz;
        syy += (long long)dy * dy;
        syz += (long long)dy * dz;
        szz += (long long)dz * dz;
    }
    // neighbours are stored nearest first, so the missing ones are the last
    // (their offsets are 0 and add nothing to the sums)
    long long ss = sxx + syy + szz;
    double rms = m ? sqrt((double)ss / (double)m) : 0.0;
    const float inv = rms > 0.0 ? (float)(1.0 / rms) : 0.f;
    uint32_t w[NF / 2];
#pragma unroll
    for (int c = 0; c < NF; c += 2) {
        int i0 = c / 3, c0 = c % 3, i1 = (c + 1) / 3, c1 = (c + 1) % 3;
        int v0 = c0 == 0 ? ox[i0] : (c0 == 1 ? oy[i0] : oz[i0]);
        int v1 = c1 == 0 ? ox[i1] : (c1 == 1 ? oy[i1] : oz[i1]);
        const uint32_t f0 = rms > 0.0 ? ratio_bf16(v0, inv, rms) : 0u;
        const uint32_t f1 = rms > 0.0 ? ratio_bf16(v1, inv, rms) : 0u;
        w[c / 2] = f0 | (f1 << 16);
    }
    uint4* fr = feat + out * (NF / 8);
#pragma unroll
    for (int j = 0; j < NF / 8; j++)
        fr[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    long long mm = m;
    double nv[3] = {0.0, 0.0, 0.0};
    double a00 = (double)(mm * sxx - sx * sx), a11 = (double)(mm * syy - sy * sy),
           a22 = (double)(mm * szz - sz * sz);
    double lmid = 0.0;
    bool ok = m >= 3 && smallest_eigvec(a00, (double)(mm * sxy - sx * sy),
                                        (double)(mm * sxz - sx * sz), a11,
                                        (double)(mm * syz - sy * sz), a22, nv, &lmid);
    // planar: the smallest eigenvalue (A n . n) at most PD_PLANAR_RATIO of the middle one
    bool planar = false;
    if (ok) {
        double c01 = (double)(mm * sxy - sx * sy), c02 = (double)(mm * sxz - sx * sz),
               c12 = (double)(mm * syz - sy * sz);
        double an0 = a00 * nv[0] + c01 * nv[1] + c02 * nv[2];
        double an1 = c01 * nv[0] + a11 * nv[1] + c12 * nv[2];
        double an2 = c02 * nv[0] + c12 * nv[1] + a22 * nv[2];
        double l0 = an0 * nv[0] + an1 * nv[1] + an2 * nv[2];
        planar = lmid > 0.0 && l0 <= PD_PLANAR_RATIO * lmid;
    }
    pca[out * 3 + 0] = ok ? (float)nv[0] : 0.f;
    pca[out * 3 + 1] = ok ? (float)nv[1] : 0.f;
    pca[out * 3 + 2] = ok ? (float)nv[2] : 0.f;
    if (valid) valid[out] = (uint8_t)((ok ? PD_NORMAL_DEFINED : 0) | (planar ? PD_NORMAL_PLANAR : 0));
}

// ------------------------------------------------------------------ forward (tensor cores)
__device__ inline uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ inline float2 unpack_bf16(uint32_t u) {
    __nv_bfloat162 v = *reinterpret_cast<__nv_bfloat162*>(&u);
    return make_float2(__bfloat162float(v.x), __bfloat162float(v.y));
}

// D = A B + D for one m16n8k16 tile (A row-major 16x16, B column-major 16x8).
__device__ inline void mma16816(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Accumulators of two adjacent n-tiles (one 16-column k-slice) -> the next
// layer's A fragment, after ReLU and rounding to bfloat16.
__device__ inline uint32_t relu_bf16(float lo, float hi) {
    // rounding and ReLU commute; NaN gives 0, as fmaxf would
    __nv_bfloat162 v = __hmax2(__floats2bfloat162_rn(lo, hi), __floats2bfloat162_rn(0.f, 0.f));
    return *reinterpret_cast<uint32_t*>(&v);
}
__device__ inline void relu_pack(const float lo[4], const float hi[4], uint32_t a[4]) {
    a[0] = relu_bf16(lo[0], lo[1]);
    a[1] = relu_bf16(lo[2], lo[3]);
    a[2] = relu_bf16(hi[0], hi[1]);
    a[3] = relu_bf16(hi[2], hi[3]);
}

__device__ inline uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ inline void ldsm4(uint32_t r[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}
__device__ inline void ldsm4t(uint32_t r[4], const void* p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}
// rows x cols floats (row-major, cols a multiple of 4) to bf16 rows of stride ld.
__device__ __forceinline__ void load_weights(__nv_bfloat16* dst, int ld, const float* src,
                                             int rows, int cols, bool vec) {
#pragma unroll 4
    for (int i = threadIdx.x; i < rows * cols / 4; i += blockDim.x) {
        const int r = 4 * i / cols, c = 4 * i % cols;
        float4 v;
        if (vec) {
            v = *reinterpret_cast<const float4*>(src + 4 * i);
        } else {
            v = make_float4(src[4 * i], src[4 * i + 1], src[4 * i + 2], src[4 * i + 3]);
        }
        uint32_t* o = reinterpret_cast<uint32_t*>(dst + r * ld + c);
        o[0] = pack_bf16(v.x, v.y);
        o[1] = pack_bf16(v.z, v.w);
    }
}


// 4 warps and 46 KB a block: within what a launch takes without an attribute call
// on the host (a call of 1500 rows: 16.2 us with the host side, 17.8 with 16-row tiles
// and 8 warps, 3 to 5 more with the attribute call)
#define MLP_WARPS 4
#define MLP_BLOCKS_PER_SM 4
#define MT 2                  // 16-row tiles of a warp's step: they share the weight fragments
#define MLP_ROWS (16 * MT)

// Rows of an odd number of 16-byte words: no bank conflicts under ldmatrix.
#define W1_LD 56
#define W2_LD 72
struct MlpSmem {
    __nv_bfloat16 w1[NH][W1_LD];
    __nv_bfloat16 w2[NH][W2_LD];
    __nv_bfloat16 w3[8][W2_LD];  // rows 3..7 zero
    float b1[NH], b2[NH], b3[8];
    __nv_bfloat16 x[MLP_WARPS][2][MLP_ROWS][W1_LD];  // feature rows, this step's and the next's
};

// One layer of MT 16-row tiles: c[tile][n-tile] = bias + A W^T over KK k-slices.
template <int KK, int LD>
__device__ __forceinline__ void mlp_layer(float (&c)[MT][8][4], const uint32_t (&a)[MT][KK][4],
                                          const __nv_bfloat16 (*w)[LD], const float* bias,
                                          int lane) {
    const int t = lane & 3, lr = lane & 7, lm = lane >> 3;
#pragma unroll
    for (int j = 0; j < 8; j++) {
        const float b0 = bias[8 * j + 2 * t], b1 = bias[8 * j + 2 * t + 1];
#pragma unroll
        for (int m = 0; m < MT; m++) {
            c[m][j][0] = b0;
            c[m][j][1] = b1;
            c[m][j][2] = b0;
            c[m][j][3] = b1;
        }
    }
#pragma unroll
    for (int kk = 0; kk < KK; kk++) {
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            uint32_t bb[4];
            ldsm4(bb, &w[8 * (j + (lm >> 1)) + lr][16 * kk + 8 * (lm & 1)]);
#pragma unroll
            for (int m = 0; m < MT; m++) {
                mma16816(c[m][j], a[m][kk], bb[0], bb[1]);
                mma16816(c[m][j + 1], a[m][kk], bb[2], bb[3]);
            }
        }
    }
}

// Persistent: a warp takes 32 rows at a time, the weights rounded into shared
// memory once per block; the next rows arrive by 16-byte asynchronous copies
// while these are computed.  Outputs per row: unit normal and |o|.
// Bound: latency.  4.0M rows take 201 us with the tensor pipe 53 % and the schedulers
// 46 % busy (128 registers, 14 warps in flight per SM); a warp's stalls per issue are
// 2.7 cycles of fixed latency, 1.2 for the tensor pipe and 1.1 for the rows.  One or two
// tiles a step and 8 to 32 warps per SM all took 192 us or more; blocks of 8 warps 192,
// but a small call pays the attribute call above.
// Fragments and features by 4-byte loads, as before, took 231 us.
__global__ void __launch_bounds__(MLP_WARPS * 32, MLP_BLOCKS_PER_SM)
    mlp_forward_kernel(const float* __restrict__ prm, const uint16_t* __restrict__ feat,
                       int64_t n, float* outn, float* onorm, bool vec_prm, bool vec_feat) {
    __shared__ __align__(16) MlpSmem sm;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int lr = lane & 7, lm = lane >> 3;
    const int64_t nsteps = (n + MLP_ROWS - 1) / MLP_ROWS;
    const int64_t wstride = (int64_t)gridDim.x * MLP_WARPS;
    int64_t step = (int64_t)blockIdx.x * MLP_WARPS + w;
    auto fetch = [&](int64_t st, int buf) {
        if (st < nsteps) {
#pragma unroll
            for (int i = 0; i < MLP_ROWS * (NF / 8) / 32; i++) {
                const int e = i * 32 + lane, r = e / (NF / 8), c = 8 * (e % (NF / 8));
                const int64_t row = st * MLP_ROWS + r;
                __nv_bfloat16* dst = &sm.x[w][buf][r][c];
                const uint16_t* src = feat + row * NF + c;
                if (row >= n) {
                    *reinterpret_cast<uint4*>(dst) = make_uint4(0, 0, 0, 0);
                } else if (vec_feat) {
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                                     smem_addr(dst)),
                                 "l"(src));
                } else {
                    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(src);
                    *reinterpret_cast<uint4*>(dst) = make_uint4(s32[0], s32[1], s32[2], s32[3]);
                }
            }
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    fetch(step, 0);
    load_weights(&sm.w1[0][0], W1_LD, prm + O_W1, NH, NF, vec_prm);
    load_weights(&sm.w2[0][0], W2_LD, prm + O_W2, NH, NH, vec_prm);
    load_weights(&sm.w3[0][0], W2_LD, prm + O_W3, 3, NH, vec_prm);
    for (int i = threadIdx.x; i < 5 * NH; i += blockDim.x)
        sm.w3[3 + i / NH][i % NH] = __float2bfloat16_rn(0.f);
    for (int i = threadIdx.x; i < NH; i += blockDim.x) {
        sm.b1[i] = prm[O_B1 + i];
        sm.b2[i] = prm[O_B2 + i];
    }
    if (threadIdx.x < 8) sm.b3[threadIdx.x] = threadIdx.x < 3 ? prm[O_B3 + threadIdx.x] : 0.f;
    __syncthreads();
    for (int buf = 0; step < nsteps; step += wstride, buf ^= 1) {
        fetch(step + wstride, buf ^ 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncwarp();
        uint32_t a1[MT][3][4];
#pragma unroll
        for (int m = 0; m < MT; m++)
#pragma unroll
            for (int kk = 0; kk < 3; kk++)
                ldsm4(a1[m][kk],
                      &sm.x[w][buf][16 * m + lr + 8 * (lm & 1)][16 * kk + 8 * (lm >> 1)]);
        __syncwarp();  // read before the next fetch overwrites the other buffer's peer
        float c[MT][8][4];
        mlp_layer<3, W1_LD>(c, a1, sm.w1, sm.b1, lane);
        uint32_t a2[MT][4][4];
#pragma unroll
        for (int m = 0; m < MT; m++)
#pragma unroll
            for (int kk = 0; kk < 4; kk++) relu_pack(c[m][2 * kk], c[m][2 * kk + 1], a2[m][kk]);
        mlp_layer<4, W2_LD>(c, a2, sm.w2, sm.b2, lane);
#pragma unroll
        for (int m = 0; m < MT; m++)
#pragma unroll
            for (int kk = 0; kk < 4; kk++) relu_pack(c[m][2 * kk], c[m][2 * kk + 1], a2[m][kk]);
        // layer 3: K = 64, N = 8 (3 used)
        float c3[MT][4];
#pragma unroll
        for (int m = 0; m < MT; m++) {
            c3[m][0] = c3[m][2] = sm.b3[2 * t];
            c3[m][1] = c3[m][3] = sm.b3[2 * t + 1];
        }
#pragma unroll
        for (int kk = 0; kk < 4; kk += 2) {
            uint32_t bb[4];  // two k-slices of the one n-tile
            ldsm4(bb, &sm.w3[lr][16 * kk + 8 * lm]);
#pragma unroll
            for (int m = 0; m < MT; m++) {
                mma16816(c3[m], a2[m][kk], bb[0], bb[1]);
                mma16816(c3[m], a2[m][kk + 1], bb[2], bb[3]);
            }
        }
#pragma unroll
        for (int m = 0; m < MT; m++) {
            // columns 0,1 sit on lane t = 0 and column 2 on t = 1 of each row
            const float o2a = __shfl_down_sync(0xffffffffu, c3[m][0], 1);
            const float o2b = __shfl_down_sync(0xffffffffu, c3[m][2], 1);
            if (t == 0) {
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int64_t row = step * MLP_ROWS + 16 * m + 8 * h + g;
                    if (row >= n) continue;
                    float o0 = h ? c3[m][2] : c3[m][0], o1 = h ? c3[m][3] : c3[m][1],
                          o2 = h ? o2b : o2a;
                    float nr = sqrtf(o0 * o0 + o1 * o1 + o2 * o2);
                    if (onorm) onorm[row] = nr;
                    if (outn) {
                        float inv = nr > 0.f ? 1.f / nr : 0.f;
                        outn[row * 3 + 0] = o0 * inv;
                        outn[row * 3 + 1] = o1 * inv;
                        outn[row * 3 + 2] = o2 * inv;
                    }
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// ------------------------------------------------------------------ gradient (tensor cores)
// Forward and backward of a batch in one launch, persistent over tiles of
// BT_ROWS = 64 rows; 4 warps per block, warp w owning rows 16w..16w+15 of a tile
// for the row-wise products and the 16-row slice w of the weight gradients.
// All matrix products run as mma.sync m16n8k16 (bf16 in, fp32 accumulate):
//   h1, h2, o                            as mlp_forward_kernel
//   dh1 = (dh2 W2) relu'(h1)             A = dh2 [row][j], B = W2 [j][c]
//   dW2 = dh2^T h1                       A = dh2^T [j][row], B = h1 [row][c]
//   dW1 = dh1^T x                        A = dh1^T [a][row], B = x [row][f]
// Every matrix is kept once in shared memory, row-major; the operands that
// enter transposed are read with ldmatrix.trans.
// x, h1 and the weights are bfloat16 values already (what the forward used).
// The gradients dh1 and dh2 are float32: each enters as the sum of two
// bfloat16 parts hi + lo (hi = bf16(v), lo = bf16(v - hi)), two products per
// tile, so the result keeps about 16 bits of the float32 value.  The small
// pieces (dh2 = do W3 masked, dW3, the biases, the loss) run on the CUDA
// cores.  Weights enter as the bfloat16 values the forward used; rounding is
// treated as the identity (a straight-through gradient).
//
// A step of 4096 rows is 64 blocks of one tile each: what it costs is the chain
// of loads and barriers of one block, so everything it reads comes as 16-byte
// loads issued together, the forward's activations never leave shared memory,
// and a training step's launches overlap (the rows are sampled and read before
// the wait for the step before).  Separate sampling, forward and backward
// launches with the activations in global memory took 28.5 us of a step, all
// of it: a training step of 4096 rows takes 14.6 us where it took 44.
#define BT_ROWS 64
#define BT_THREADS 128
#define BT_LD 72   // row stride (bf16) of the 64-wide tiles: 144 bytes, an odd number
#define BT_LDX 56  //   of 16-byte words (no bank conflicts); of the 48-wide: 112 bytes
#define BT_BLOCKS_PER_SM 2

// a0 b0 + a1 b1 + a2 b2 with the order of its roundings fixed (the middle
// product is rounded, the others fused), so that a gradient does not depend on
// how the compiler contracts the sum in one kernel or another.
__device__ __forceinline__ float dot3(float a0, float b0, float a1, float b1, float a2, float b2) {
    return __fmaf_rn(a2, b2, __fmaf_rn(a0, b0, __fmul_rn(a1, b1)));
}

struct StepSmem {
    __nv_bfloat16 w1[NH][BT_LDX];         // W1 [a][f]
    __nv_bfloat16 w2[NH][BT_LD];          // W2 [j][c]
    __nv_bfloat16 w3[8][BT_LD];           // W3, rows 3..7 zero
    __nv_bfloat16 x[BT_ROWS][BT_LDX];     // rows beyond the batch are zero in all of these
    __nv_bfloat16 h1[BT_ROWS][BT_LD];
    __nv_bfloat16 h2[BT_ROWS][BT_LD];
    __nv_bfloat16 d2[2][BT_ROWS][BT_LD];  // dh2, hi and lo
    __nv_bfloat16 d1[2][BT_ROWS][BT_LD];  // dh1, hi and lo
    float b1[NH], b2[NH], b3[8];
    float raw[BT_ROWS][4];
    float dout[BT_ROWS][4];               // d loss / d o (divided by n)
    float red[BT_THREADS][4];             // end-of-kernel reductions
    float db1w[4][NH];                    // per-warp column sums of dh1
    int64_t row[BT_ROWS];                 // feature row of each tile row
};

// Programmatic dependent launch: a launch that carries the attribute may start
// before the one ahead of it in the stream has finished; what depends on that
// one comes after the wait.
__device__ inline void wait_prior_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ inline void allow_next_launch() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// splitmix64 output function (Steele, Lea and Flood, OOPSLA 2014) of state x
__device__ inline u64 splitmix64(u64 x) {
    u64 z = x + 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// Rows of a batch: row i is feature row pool[splitmix64(seed ^ (t << 32) ^ i) %
// npool]; pool NULL: row i.
struct BatchRows {
    const int* pool;
    int64_t npool;
    u64 seed;
    long long t;
    __device__ __forceinline__ int64_t at(int64_t i) const {
        if (!pool) return i;
        const u64 h = splitmix64(seed ^ ((u64)t << 32) ^ (u64)i);
        return pool[h % (u64)npool];
    }
};

__global__ void __launch_bounds__(BT_THREADS, BT_BLOCKS_PER_SM)
    mlp_gradient_kernel(const float* prm, const uint16_t* __restrict__ feat, BatchRows rows,
                        const float* __restrict__ labels, int64_t n, float* part, bool vec_prm,
                        bool vec_feat) {
    extern __shared__ __align__(16) unsigned char smraw[];
    StepSmem& sm = *reinterpret_cast<StepSmem*>(smraw);
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const float inv_n = 1.0f / (float)n;
    allow_next_launch();
    // accumulators: dW1 rows a = 16w.. (6 n-tiles of f), dW2 rows j = 16w.. (8 n-tiles of c)
    float g1[6][4], g2[8][4];
#pragma unroll
    for (int i = 0; i < 6; i++) g1[i][0] = g1[i][1] = g1[i][2] = g1[i][3] = 0.f;
#pragma unroll
    for (int i = 0; i < 8; i++) g2[i][0] = g2[i][1] = g2[i][2] = g2[i][3] = 0.f;
    float db1[16];  // columns 8 nt + 2 t (+1) of dh1, this lane's rows
#pragma unroll
    for (int i = 0; i < 16; i++) db1[i] = 0.f;
    float db2 = 0.f, dw3[3] = {0.f, 0.f, 0.f}, db3[3] = {0.f, 0.f, 0.f}, lsum = 0.f;
    const int jcol = tid & 63;  // the dh2 column this thread computes
    const int64_t ntiles = (n + BT_ROWS - 1) / BT_ROWS;
    // ldmatrix lane addresses: matrix lane / 8, row lane % 8 of it
    const int lr = lane & 7, lm = lane >> 3;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t r0 = tile * BT_ROWS;
        const int nr = (int)min((int64_t)BT_ROWS, n - r0);
        const bool first = tile == blockIdx.x;
        __syncthreads();  // the previous tile's readers are done
        if (tid < BT_ROWS) sm.row[tid] = tid < nr ? rows.at(r0 + tid) : -1;
        __syncthreads();
        for (int i = tid; i < BT_ROWS * (NF / 8); i += BT_THREADS) {
            const int r = i / (NF / 8), c = 8 * (i % (NF / 8));
            uint4 v = make_uint4(0, 0, 0, 0);
            if (r < nr) {
                const uint16_t* src = feat + sm.row[r] * NF + c;
                if (vec_feat) {
                    v = *reinterpret_cast<const uint4*>(src);
                } else {
                    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(src);
                    v = make_uint4(s32[0], s32[1], s32[2], s32[3]);
                }
            }
            *reinterpret_cast<uint4*>(&sm.x[r][c]) = v;
        }
        float y0 = 0.f, y1 = 0.f, y2 = 0.f;
        if (tid < nr) {
            const int64_t x = sm.row[tid];
            y0 = labels[x * 3];
            y1 = labels[x * 3 + 1];
            y2 = labels[x * 3 + 2];
        }
        if (first) {  // the weights of the step before are complete from here
            wait_prior_launch();
            load_weights(&sm.w1[0][0], BT_LDX, prm + O_W1, NH, NF, vec_prm);
            load_weights(&sm.w2[0][0], BT_LD, prm + O_W2, NH, NH, vec_prm);
            load_weights(&sm.w3[0][0], BT_LD, prm + O_W3, 3, NH, vec_prm);
            for (int i = tid; i < 5 * NH; i += BT_THREADS)
                sm.w3[3 + i / NH][i % NH] = __float2bfloat16_rn(0.f);
            for (int i = tid; i < NH; i += BT_THREADS) {
                sm.b1[i] = prm[O_B1 + i];
                sm.b2[i] = prm[O_B2 + i];
            }
            if (tid < 8) sm.b3[tid] = tid < 3 ? prm[O_B3 + tid] : 0.f;
        }
        __syncthreads();
        const int ra = 16 * w + g, rb = ra + 8;
        const bool va = ra < nr, vb = rb < nr;
        // ---- forward of rows 16w..16w+15
        {
            float c1[8][4];
#pragma unroll
            for (int j = 0; j < 8; j++) {
                float b0 = sm.b1[8 * j + 2 * t], b1v = sm.b1[8 * j + 2 * t + 1];
                c1[j][0] = b0;
                c1[j][1] = b1v;
                c1[j][2] = b0;
                c1[j][3] = b1v;
            }
#pragma unroll
            for (int kk = 0; kk < 3; kk++) {
                uint32_t a[4];
                ldsm4(a, &sm.x[16 * w + lr + 8 * (lm & 1)][16 * kk + 8 * (lm >> 1)]);
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    uint32_t bb[4];
                    ldsm4(bb, &sm.w1[8 * (j + (lm >> 1)) + lr][16 * kk + 8 * (lm & 1)]);
                    mma16816(c1[j], a, bb[0], bb[1]);
                    mma16816(c1[j + 1], a, bb[2], bb[3]);
                }
            }
            uint32_t a2[4][4];
#pragma unroll
            for (int kk = 0; kk < 4; kk++) {
                relu_pack(c1[2 * kk], c1[2 * kk + 1], a2[kk]);
                *reinterpret_cast<uint32_t*>(&sm.h1[ra][16 * kk + 2 * t]) = va ? a2[kk][0] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h1[rb][16 * kk + 2 * t]) = vb ? a2[kk][1] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h1[ra][16 * kk + 8 + 2 * t]) =
                    va ? a2[kk][2] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h1[rb][16 * kk + 8 + 2 * t]) =
                    vb ? a2[kk][3] : 0u;
            }
            float c2[8][4];
#pragma unroll
            for (int j = 0; j < 8; j++) {
                float b0 = sm.b2[8 * j + 2 * t], b1v = sm.b2[8 * j + 2 * t + 1];
                c2[j][0] = b0;
                c2[j][1] = b1v;
                c2[j][2] = b0;
                c2[j][3] = b1v;
            }
#pragma unroll
            for (int kk = 0; kk < 4; kk++) {
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    uint32_t bb[4];
                    ldsm4(bb, &sm.w2[8 * (j + (lm >> 1)) + lr][16 * kk + 8 * (lm & 1)]);
                    mma16816(c2[j], a2[kk], bb[0], bb[1]);
                    mma16816(c2[j + 1], a2[kk], bb[2], bb[3]);
                }
            }
            uint32_t a3[4][4];
#pragma unroll
            for (int kk = 0; kk < 4; kk++) {
                relu_pack(c2[2 * kk], c2[2 * kk + 1], a3[kk]);
                *reinterpret_cast<uint32_t*>(&sm.h2[ra][16 * kk + 2 * t]) = va ? a3[kk][0] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h2[rb][16 * kk + 2 * t]) = vb ? a3[kk][1] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h2[ra][16 * kk + 8 + 2 * t]) =
                    va ? a3[kk][2] : 0u;
                *reinterpret_cast<uint32_t*>(&sm.h2[rb][16 * kk + 8 + 2 * t]) =
                    vb ? a3[kk][3] : 0u;
            }
            float c3[4] = {sm.b3[2 * t], sm.b3[2 * t + 1], sm.b3[2 * t], sm.b3[2 * t + 1]};
#pragma unroll
            for (int kk = 0; kk < 4; kk += 2) {
                uint32_t bb[4];  // two k-slices of the one n-tile
                ldsm4(bb, &sm.w3[lr][16 * kk + 8 * lm]);
                mma16816(c3, a3[kk], bb[0], bb[1]);
                mma16816(c3, a3[kk + 1], bb[2], bb[3]);
            }
            // columns 0,1 sit on lane t = 0 and column 2 on t = 1 of each row
            if (t == 0) {
                sm.raw[ra][0] = c3[0];
                sm.raw[ra][1] = c3[1];
                sm.raw[rb][0] = c3[2];
                sm.raw[rb][1] = c3[3];
            } else if (t == 1) {
                sm.raw[ra][2] = c3[0];
                sm.raw[rb][2] = c3[2];
            }
        }
        __syncthreads();
        if (tid < BT_ROWS) {  // d loss / d o for row tid, already divided by n
            int r = tid;
            float d0 = 0.f, d1 = 0.f, d2 = 0.f;
            if (r < nr) {
                float o0 = sm.raw[r][0], o1 = sm.raw[r][1], o2 = sm.raw[r][2];
                float nrm = sqrtf(dot3(o0, o0, o1, o1, o2, o2));
                if (nrm > 0.f) {
                    float u0 = o0 / nrm, u1 = o1 / nrm, u2 = o2 / nrm;
                    float dot = dot3(u1, y1, u0, y0, u2, y2);
                    lsum += 1.f - dot * dot;
                    // dL/du = -2 dot y; dL/do = (dL/du - (dL/du . u) u) / |o|
                    float q0 = -2.f * dot * y0, q1 = -2.f * dot * y1, q2 = -2.f * dot * y2;
                    float gu = dot3(q0, u0, q1, u1, q2, u2);
                    float sc = inv_n / nrm;
                    d0 = (q0 - gu * u0) * sc;
                    d1 = (q1 - gu * u1) * sc;
                    d2 = (q2 - gu * u2) * sc;
                }
            }
            sm.dout[r][0] = d0;
            sm.dout[r][1] = d1;
            sm.dout[r][2] = d2;
            db3[0] += d0;
            db3[1] += d1;
            db3[2] += d2;
        }
        __syncthreads();
        // dh2 = (do W3) relu'(h2): thread (jcol, rows tid/64 + 2i); dW3 and db2 on the side
        {
            const float w30 = __bfloat162float(sm.w3[0][jcol]);
            const float w31 = __bfloat162float(sm.w3[1][jcol]);
            const float w32 = __bfloat162float(sm.w3[2][jcol]);
#pragma unroll 4
            for (int r = tid >> 6; r < BT_ROWS; r += BT_THREADS / 64) {
                float v = 0.f;
                if (r < nr) {
                    float h2 = __bfloat162float(sm.h2[r][jcol]);
                    float d0 = sm.dout[r][0], d1 = sm.dout[r][1], d2 = sm.dout[r][2];
                    dw3[0] += d0 * h2;
                    dw3[1] += d1 * h2;
                    dw3[2] += d2 * h2;
                    v = dot3(d0, w30, d1, w31, d2, w32);
                    if (!(h2 > 0.f)) v = 0.f;
                }
                db2 += v;
                __nv_bfloat16 hi = __float2bfloat16_rn(v);
                sm.d2[0][r][jcol] = hi;
                sm.d2[1][r][jcol] = __float2bfloat16_rn(v - __bfloat162float(hi));
            }
        }
        __syncthreads();
        // dh1 = (dh2 W2) relu'(h1) for rows 16w.. of the tile (tensor cores)
        {
            float acc[8][4];
#pragma unroll
            for (int nt = 0; nt < 8; nt++) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
            for (int kk = 0; kk < 4; kk++) {
                uint32_t a[2][4];
#pragma unroll
                for (int q = 0; q < 2; q++)
                    ldsm4(a[q], &sm.d2[q][16 * w + lr + 8 * (lm & 1)][16 * kk + 8 * (lm >> 1)]);
#pragma unroll
                for (int nt = 0; nt < 8; nt += 2) {
                    uint32_t bb[4];
                    ldsm4t(bb, &sm.w2[16 * kk + lr + 8 * (lm & 1)][8 * (nt + (lm >> 1))]);
#pragma unroll
                    for (int q = 0; q < 2; q++) {
                        mma16816(acc[nt], a[q], bb[0], bb[1]);
                        mma16816(acc[nt + 1], a[q], bb[2], bb[3]);
                    }
                }
            }
#pragma unroll
            for (int nt = 0; nt < 8; nt++) {
                const int c = 8 * nt + 2 * t;
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                    const int r = e ? rb : ra;
                    const float2 h = unpack_bf16(*reinterpret_cast<uint32_t*>(&sm.h1[r][c]));
                    float v0 = acc[nt][e], v1 = acc[nt][e + 1];
                    if (!(h.x > 0.f)) v0 = 0.f;
                    if (!(h.y > 0.f)) v1 = 0.f;
                    db1[2 * nt] += v0;
                    db1[2 * nt + 1] += v1;
                    const uint32_t hi = pack_bf16(v0, v1);
                    const float2 hf = unpack_bf16(hi);
                    *reinterpret_cast<uint32_t*>(&sm.d1[0][r][c]) = hi;
                    *reinterpret_cast<uint32_t*>(&sm.d1[1][r][c]) =
                        pack_bf16(v0 - hf.x, v1 - hf.y);
                }
            }
        }
        __syncthreads();
        // weight gradients over the tile's rows (K = 64): slice w of dW1 and dW2
#pragma unroll
        for (int kk = 0; kk < 4; kk++) {
            const int kr = 16 * kk + lr;
            uint32_t a1[2][4], a2[2][4];
#pragma unroll
            for (int q = 0; q < 2; q++) {
                ldsm4t(a1[q], &sm.d1[q][kr + 8 * (lm >> 1)][16 * w + 8 * (lm & 1)]);
                ldsm4t(a2[q], &sm.d2[q][kr + 8 * (lm >> 1)][16 * w + 8 * (lm & 1)]);
            }
#pragma unroll
            for (int nt = 0; nt < 6; nt += 2) {
                uint32_t bb[4];
                ldsm4t(bb, &sm.x[kr + 8 * (lm & 1)][8 * (nt + (lm >> 1))]);
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    mma16816(g1[nt], a1[q], bb[0], bb[1]);
                    mma16816(g1[nt + 1], a1[q], bb[2], bb[3]);
                }
            }
#pragma unroll
            for (int nt = 0; nt < 8; nt += 2) {
                uint32_t bb[4];
                ldsm4t(bb, &sm.h1[kr + 8 * (lm & 1)][8 * (nt + (lm >> 1))]);
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    mma16816(g2[nt], a2[q], bb[0], bb[1]);
                    mma16816(g2[nt + 1], a2[q], bb[2], bb[3]);
                }
            }
        }
    }
    // this block's partial sums; the reduction adds the blocks in a fixed
    // order, so the gradient is the same bit for bit on every run
    float* mine = part + (int64_t)blockIdx.x * (N_PARAMS + 1);
    {
        const int ma = 16 * w + g, mb = ma + 8;
#pragma unroll
        for (int nt = 0; nt < 6; nt++) {
            int f = 8 * nt + 2 * t;
            mine[O_W1 + ma * NF + f] = g1[nt][0];
            mine[O_W1 + ma * NF + f + 1] = g1[nt][1];
            mine[O_W1 + mb * NF + f] = g1[nt][2];
            mine[O_W1 + mb * NF + f + 1] = g1[nt][3];
        }
#pragma unroll
        for (int nt = 0; nt < 8; nt++) {
            int c = 8 * nt + 2 * t;
            mine[O_W2 + ma * NH + c] = g2[nt][0];
            mine[O_W2 + ma * NH + c + 1] = g2[nt][1];
            mine[O_W2 + mb * NH + c] = g2[nt][2];
            mine[O_W2 + mb * NH + c + 1] = g2[nt][3];
        }
    }
    // db1: sum this lane's rows over the 8 lanes of equal t, then the 4 warps
#pragma unroll
    for (int i = 0; i < 16; i++) {
        float v = db1[i];
        v += __shfl_xor_sync(0xffffffffu, v, 4);
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        db1[i] = v;
    }
    if (g == 0) {
#pragma unroll
        for (int nt = 0; nt < 8; nt++) {
            sm.db1w[w][8 * nt + 2 * t] = db1[2 * nt];
            sm.db1w[w][8 * nt + 2 * t + 1] = db1[2 * nt + 1];
        }
    }
    // db2, dW3: two threads per column (tid and tid + 64)
    sm.red[tid][0] = db2;
    sm.red[tid][1] = dw3[0];
    sm.red[tid][2] = dw3[1];
    sm.red[tid][3] = dw3[2];
    __syncthreads();
    if (tid < NH) {
        float v = 0.f;
        for (int ww = 0; ww < 4; ww++) v += sm.db1w[ww][tid];
        mine[O_B1 + tid] = v;
        mine[O_B2 + tid] = sm.red[tid][0] + sm.red[tid + 64][0];
        for (int c = 0; c < 3; c++) mine[O_W3 + c * NH + tid] = sm.red[tid][1 + c] + sm.red[tid + 64][1 + c];
    }
    __syncthreads();
    // db3 and the loss: rows tid < 64
    sm.red[tid][0] = db3[0];
    sm.red[tid][1] = db3[1];
    sm.red[tid][2] = db3[2];
    sm.red[tid][3] = lsum;
    __syncthreads();
    if (tid < 4) {
        float v = 0.f;
#pragma unroll 16
        for (int r = 0; r < BT_ROWS; r++) v += sm.red[r][tid];
        if (tid < 3) mine[O_B3 + tid] = v;
        else mine[N_PARAMS] = v * inv_n;
    }
}

// Sum of entry i of the blocks' partials, in block order; 32 loads in flight.
__device__ __forceinline__ float sum_partials(const float* __restrict__ part, int nblocks, int i) {
    float v = 0.f;
    int b = 0;
    for (; b + 32 <= nblocks; b += 32) {
        float x[32];
#pragma unroll
        for (int j = 0; j < 32; j++) x[j] = part[(int64_t)(b + j) * (N_PARAMS + 1) + i];
#pragma unroll
        for (int j = 0; j < 32; j++) v += x[j];
    }
    for (; b < nblocks; b++) v += part[(int64_t)b * (N_PARAMS + 1) + i];
    return v;
}

// grad[i] (and the loss, entry N_PARAMS) = sum of the blocks' partials.
__global__ void grad_reduce_kernel(const float* __restrict__ part, int nblocks, float* grad,
                                   float* loss) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i > N_PARAMS) return;
    const float v = sum_partials(part, nblocks, i);
    if (i < N_PARAMS) grad[i] = v;
    else *loss = v;
}

// ------------------------------------------------------------------ Adam, init, sampling
// The step's gradient (sum of the blocks' partials) and loss, then Adam (Kingma
// & Ba, ICLR 2015) with bias correction; t = step number (1-based).
__global__ void __launch_bounds__(64)
    adam_kernel(const float* part, int nblocks, float* prm, float* m, float* v, float* loss, int t,
                float lr, float b1, float b2, float eps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    allow_next_launch();
    wait_prior_launch();  // the partials
    if (i > N_PARAMS) return;
    const float g = sum_partials(part, nblocks, i);
    if (i == N_PARAMS) {
        *loss = g;
        return;
    }
    float mi = b1 * m[i] + (1.f - b1) * g;
    float vi = b2 * v[i] + (1.f - b2) * g * g;
    m[i] = mi;
    v[i] = vi;
    float mh = mi / (1.f - powf(b1, (float)t));
    float vh = vi / (1.f - powf(b2, (float)t));
    prm[i] -= lr * mh / (sqrtf(vh) + eps);
}

__global__ void mlp_init_kernel(float* prm, u64 seed) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N_PARAMS) return;
    u64 h = splitmix64(seed * 0x100000001b3ull + (u64)i);
    float u = (float)(h >> 40) * (1.0f / 16777216.0f) * 2.0f - 1.0f;  // exact, in [-1, 1)
    float v = 0.f;
    if (i < O_B1) v = u * sqrtf(6.0f / NF);
    else if (i >= O_W2 && i < O_B2) v = u * sqrtf(6.0f / NH);
    else if (i >= O_W3 && i < O_B3) v = u * sqrtf(3.0f / NH);
    prm[i] = v;
}

__global__ void fallback_kernel(const float* __restrict__ mlp, const float* __restrict__ onorm,
                                const float* __restrict__ pca, int64_t n, float min_norm,
                                float* out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    bool use = mlp && onorm[i] >= min_norm;
    const float* src = use ? mlp : pca;
    out[i * 3] = src[i * 3];
    out[i * 3 + 1] = src[i * 3 + 1];
    out[i * 3 + 2] = src[i * 3 + 2];
}

__global__ void iota_kernel(int* out, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = (int)i;
}

// ------------------------------------------------------------------ launchers
cudaError_t launch_iota(int* out, int64_t n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    iota_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(out, n);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_features(const int4* pos, const int* nbr, int S, int64_t n, uint16_t* feat,
                            float* pca, uint8_t* valid, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    launch_chained(features_kernel, (unsigned)((n + 127) / 128), 128, 0, st, pos, nbr, S, n,
                   (uint4*)feat, pca, valid);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const float* prm, const uint16_t* feat, int64_t n, float* outn,
                               float* onorm, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    static_assert(sizeof(MlpSmem) <= 48 * 1024, "shared memory");
    int64_t steps = (n + MLP_ROWS - 1) / MLP_ROWS;
    int64_t blocks = (steps + MLP_WARPS - 1) / MLP_WARPS;
    int64_t cap = (int64_t)device_sms() * MLP_BLOCKS_PER_SM;
    if (blocks > cap) blocks = cap;
    // wider loads where the caller's arrays are aligned for them
    mlp_forward_kernel<<<(unsigned)blocks, MLP_WARPS * 32, 0, st>>>(
        prm, feat, n, outn, onorm, ((uintptr_t)prm & 15) == 0, ((uintptr_t)feat & 15) == 0);
    note_launch();
    return cudaGetLastError();
}

static int64_t bt_blocks() { return (int64_t)device_sms() * BT_BLOCKS_PER_SM; }

int64_t mlp_backward_part_floats() { return bt_blocks() * (N_PARAMS + 1); }

// Partials of the batch's gradient; *blocks_out of them.
static cudaError_t launch_gradient(const float* prm, const uint16_t* feat, const BatchRows& rows,
                                   const float* labels, int64_t n, float* part, int* blocks_out,
                                   bool overlap, cudaStream_t st) {
    static_assert(sizeof(StepSmem) <= 227 * 1024 / BT_BLOCKS_PER_SM - 1024, "shared memory");
    cudaError_t e = cudaFuncSetAttribute(mlp_gradient_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(StepSmem));
    if (e) return e;
    int64_t tiles = (n + BT_ROWS - 1) / BT_ROWS;
    int64_t cap = bt_blocks();
    *blocks_out = (int)(tiles < cap ? tiles : cap);
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((unsigned)*blocks_out);
    c.blockDim = dim3(BT_THREADS);
    c.dynamicSmemBytes = sizeof(StepSmem);
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = overlap ? 1 : 0;
    note_launch();
    // wider loads where the caller's arrays are aligned for them
    return cudaLaunchKernelEx(&c, mlp_gradient_kernel, prm, feat, rows, labels, n, part,
                              ((uintptr_t)prm & 15) == 0, ((uintptr_t)feat & 15) == 0);
}

cudaError_t launch_mlp_gradient(const float* prm, const uint16_t* feat, const float* labels,
                                int64_t n, float* grad, float* loss, float* part,
                                cudaStream_t st) {
    if (n <= 0) {
        cudaError_t e = cudaMemsetAsync(grad, 0, N_PARAMS * sizeof(float), st);
        if (!e) e = cudaMemsetAsync(loss, 0, sizeof(float), st);
        return e;
    }
    int blocks = 0;
    const BatchRows rows = {nullptr, 0, 0, 0};
    cudaError_t e = launch_gradient(prm, feat, rows, labels, n, part, &blocks, false, st);
    if (e) return e;
    grad_reduce_kernel<<<(N_PARAMS + 1 + 255) / 256, 256, 0, st>>>(part, blocks, grad, loss);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_mlp_step(float* prm, float* m, float* v, const uint16_t* feat, const int* pool,
                            int64_t npool, u64 seed, int t, const float* labels, int64_t b,
                            float lr, float* loss, float* part, bool overlap, cudaStream_t st) {
    int blocks = 0;
    const BatchRows rows = {pool, npool, seed, t};
    cudaError_t e = launch_gradient(prm, feat, rows, labels, b, part, &blocks, overlap, st);
    if (e) return e;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3((N_PARAMS + 1 + 63) / 64);
    c.blockDim = dim3(64);
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&c, adam_kernel, (const float*)part, blocks, prm, m, v, loss, t, lr,
                              0.9f, 0.999f, 1e-8f);
}

cudaError_t launch_mlp_init(float* prm, u64 seed, cudaStream_t st) {
    mlp_init_kernel<<<(N_PARAMS + 255) / 256, 256, 0, st>>>(prm, seed);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_normal_fallback(const float* mlp, const float* onorm, const float* pca,
                                   int64_t n, float min_norm, float* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    fallback_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(mlp, onorm, pca, n, min_norm,
                                                                out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace pd

// ============================================================ C ABI (pd_normals.h)
using namespace pd;

#define NCK(x)                                                        \
    do {                                                              \
        cudaError_t e_ = (x);                                         \
        if (e_ != cudaSuccess) {                                      \
            if (ctx) api_error(ctx, "CUDA error at " #x, (long long)e_); \
            rc = e_ == cudaErrorMemoryAllocation ? PD_ENOMEM : PD_ECUDA; \
            goto done;                                                \
        }                                                             \
    } while (0)
#define NALLOC(ptr, type, count)                                                   \
    do {                                                                           \
        ptr = (type*)api_alloc(ctx, sizeof(type) * (size_t)(count), st);           \
        if (!ptr) {                                                                \
            api_error(ctx, "allocation failed: " #ptr, (long long)(count));       \
            rc = PD_ENOMEM;                                                        \
            goto done;                                                             \
        }                                                                          \
    } while (0)

extern "C" int pd_normals_pca(pd_grid* g, uint16_t* feat_dev, float* pca_dev, uint8_t* valid_dev,
                              void* stream) {
    if (!g || !feat_dev || !pca_dev) return PD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    GridNbrs nb;
    int rc = grid_knn16(g, st, &nb);
    if (rc) return rc;
    pd_ctx* ctx = nb.ctx;
    NCK(launch_features(nb.pos, nb.nbr, nb.S, nb.n, feat_dev, pca_dev, valid_dev, st));
    NCK(cudaStreamSynchronize(st));
done:
    return rc;
}

extern "C" int pd_mlp_init(float* params_dev, uint64_t seed, void* stream) {
    if (!params_dev) return PD_EINVAL;
    if (launch_mlp_init(params_dev, seed, (cudaStream_t)stream) != cudaSuccess) return PD_ECUDA;
    return PD_OK;
}

extern "C" int pd_mlp_forward(const float* params_dev, const uint16_t* feat_dev, int64_t n,
                              float* normals_dev, float* norm_dev, void* stream) {
    if (!params_dev || !feat_dev || n < 0 || (!normals_dev && !norm_dev)) return PD_EINVAL;
    cudaError_t e = launch_mlp_forward(params_dev, feat_dev, n, normals_dev, norm_dev,
                                       (cudaStream_t)stream);
    return e == cudaSuccess ? PD_OK : PD_ECUDA;
}

extern "C" int pd_mlp_grad(pd_ctx* ctx, const float* params_dev, const uint16_t* feat_dev,
                           const float* labels_dev, int64_t n, float* grad_dev, float* loss_dev,
                           void* stream) {
    if (!ctx || !params_dev || !feat_dev || !labels_dev || !grad_dev || !loss_dev || n < 1)
        return PD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = PD_OK;
    float* part = nullptr;
    NALLOC(part, float, mlp_backward_part_floats());
    NCK(launch_mlp_gradient(params_dev, feat_dev, labels_dev, n, grad_dev, loss_dev, part, st));
    NCK(cudaStreamSynchronize(st));
done:
    api_free(ctx, part, st);
    return rc;
}

extern "C" int pd_mlp_train(pd_ctx* ctx, float* params_dev, float* adam_dev, int step0,
                            const uint16_t* feat_dev, const float* labels_dev,
                            const uint8_t* valid_dev, int64_t n, const pd_train_params* tp,
                            float* loss_dev, void* stream) {
    if (!ctx || !params_dev || !adam_dev || !feat_dev || !labels_dev || !tp || n < 1 ||
        n >= (1ll << 31) || tp->steps < 0 || tp->batch < 1 || step0 < 0 || !(tp->lr > 0.f))
        return PD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = PD_OK;
    int b = tp->batch;
    int *pool = nullptr, *cnt = nullptr;
    float *lossbuf = nullptr, *part = nullptr;
    int npool = 0;
    NALLOC(pool, int, n);
    NALLOC(cnt, int, 1);
    NALLOC(lossbuf, float, 1);
    NALLOC(part, float, mlp_backward_part_floats());
    if (valid_dev) {
        Scratch s;
        struct Ctx {
            pd_ctx* c;
            cudaStream_t st;
        } cs = {ctx, st};
        s.alloc = [](void* self, size_t bytes) -> void* {
            Ctx* c = (Ctx*)self;
            return api_alloc(c->c, bytes, c->st);
        };
        s.free = [](void* self, void* p) {
            Ctx* c = (Ctx*)self;
            api_free(c->c, p, c->st);
        };
        s.self = &cs;
        NCK(stable_compact(valid_dev, n, pool, cnt, s, st));
        NCK(cudaMemcpyAsync(&npool, cnt, sizeof(int), cudaMemcpyDeviceToHost, st));
        NCK(cudaStreamSynchronize(st));
    } else {
        NCK(launch_iota(pool, n, st));
        npool = (int)n;
    }
    if (npool < 1) {
        api_error(ctx, "pd_mlp_train: no valid rows", 0);
        rc = PD_EINVAL;
        goto done;
    }
    for (int i = 0; i < tp->steps; i++) {
        int t = step0 + i + 1;
        float* lp = loss_dev ? loss_dev + i : lossbuf;
        // from the second step on the launch ahead is this loop's own
        NCK(launch_mlp_step(params_dev, adam_dev, adam_dev + N_PARAMS, feat_dev, pool, npool,
                            tp->seed, t, labels_dev, b, tp->lr, lp, part, i > 0, st));
    }
    NCK(cudaStreamSynchronize(st));
done:
    void* bufs[] = {pool, cnt, lossbuf, part};
    for (void* p : bufs) api_free(ctx, p, st);
    return rc;
}

extern "C" int pd_normals_mlp(pd_ctx* ctx, const float* params_dev, const uint16_t* feat_dev,
                              const float* pca_dev, int64_t n, float min_norm, float* normals_dev,
                              void* stream) {
    if (!ctx || !pca_dev || !normals_dev || n < 0 || (params_dev && !feat_dev)) return PD_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int rc = PD_OK;
    float *mlp = nullptr, *onorm = nullptr;
    if (min_norm <= 0.f) min_norm = 1e-3f;
    if (params_dev && n > 0) {
        NALLOC(mlp, float, n * 3);
        NALLOC(onorm, float, n);
        NCK(launch_mlp_forward(params_dev, feat_dev, n, mlp, onorm, st));
    }
    NCK(launch_normal_fallback(mlp, onorm, pca_dev, n, min_norm, normals_dev, st));
done:
    api_free(ctx, mlp, st);
    api_free(ctx, onorm, st);
    return rc;
}
