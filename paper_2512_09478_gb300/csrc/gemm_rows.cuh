// Gathered row products: out[t] (=|+=) Op in[src(t)], one operator per
// class of rows (M2M over the children's octants, L2L, the factors of the leaf
// pseudo-inverses and their adjoints), one FMA per product in input order.
//
// Operators are stored [block][nkp][ldp], the inputs padded with zeros to a
// multiple of 16 and the outputs to a multiple of the kernels' column block
// (gemm_ldp), so that they come by 16-byte asynchronous copies without bounds
// tests.  Two tiles:
//  k_rows_big    (FP32; k_rows_f64 in fmm.cu) 64 rows by 32 NC outputs per 128 threads, a thread 8 rows by
//                NC pairs of outputs on packed f32x2 FMAs.  FMA-bound: with
//                operands from shared memory the loop alone reaches 95 FMA
//                lanes per clock and SM (the inputs unduplicated, their pairs
//                formed in registers: 95 against 86), a scalar three-operand
//                FMA 82.
//  k_rows_small  (FP32 and FP64) 16 or 4 rows by 32 outputs, the whole input staged by four groups
//                of asynchronous copies at once: a coarse level's time is the
//                latency of its loads, which the big tile's chunks (and the
//                16-input chunks of its predecessor) take one after the other.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace kifmm {
namespace {

constexpr int kRK = 16;         // inputs per staged chunk of the big tile
constexpr int kRThreads = 128;

// Ranges of up to 8 classes (blockIdx.y = class) in one launch.
struct ClassRanges {
    int64_t b[9];
};

// Source row and operator of a target row: parent[t] with parent, else t;
// operator block `class` with by_class, else block 0.
template <typename T>
struct RowMap {
    const int32_t *parent;
    const T *ops;
    int64_t blk;  // elements per operator block
    bool by_class;
    __device__ int src(int t) const { return parent ? parent[t] : t; }
    __device__ const T *op(int cls) const { return ops + (by_class ? cls * blk : 0); }
    // the child inherits the parent's mean
    __device__ double mean_base(int t, const double *dbar) const { return parent ? dbar[parent[t]] : 0.0; }
};

__device__ __forceinline__ void row_cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void row_cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// With dbar: output column n (the operators' mean row) goes to dbar[t] (FP64,
// plus the map's mean_base) instead of out.
template <typename T>
__device__ __forceinline__ void row_store(T v, int t, int j, int n, T *out, int accumulate, double *dbar,
                                          const RowMap<T> &g) {
    if (j < n) {
        T *o = out + (size_t)t * n + j;
        *o = accumulate ? *o + v : v;
    } else if (j == n && dbar) {
        dbar[t] = (accumulate ? dbar[t] : 0.0) + (double)v + g.mean_base(t, dbar);
    }
}

// VEC: the input rows are 16-byte aligned (n a multiple of 4).
template <int NC, bool VEC>
__global__ void __launch_bounds__(kRThreads, 3)
    k_rows_big(RowMap<float> g, const int32_t *__restrict__ targets, ClassRanges cr, int n, int nkp, int ldp,
               const float *__restrict__ in, float *out, int accumulate, double *dbar) {
    constexpr int RT = 8, TT = 8 * RT, TJ = 32 * NC;
    __shared__ __align__(16) float Us[2][kRK][TT];
    __shared__ __align__(16) float Ms[2][kRK][TJ];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int cls = blockIdx.y, j0 = blockIdx.z * TJ;
    int64_t t_begin = 0, t_end = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c == cls) t_begin = cr.b[c], t_end = cr.b[c + 1];
    const int64_t t0 = t_begin + (int64_t)blockIdx.x * TT;
    if (t0 >= t_end) return;  // uniform for the block
    // staging: input quad r of a thread is row tid % 64, inputs 4 (tid / 64 + 2 r)
    const int64_t tr = t0 + tid % TT;
    const int row = tr < t_end ? g.src(targets[tr]) : -1;
    const float *src = in + (size_t)(row >= 0 ? row : 0) * n;
    constexpr int kMQ = kRK * TJ / 4 / kRThreads;
    const float *M = g.op(cls) + j0;
    float4 ru[2];
    auto load = [&](int kc, int b) {
        const float *Mk = M + (size_t)kc * kRK * ldp;
#pragma unroll
        for (int r = 0; r < kMQ; ++r) {
            const int e = tid + kRThreads * r, k = e / (TJ / 4);
            row_cp16(&Ms[b][0][0] + 4 * e, Mk + (size_t)k * ldp + 4 * (e - k * (TJ / 4)));
        }
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = kc * kRK + 4 * (tid / TT + 2 * r);
            ru[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (row >= 0) {
                if (VEC) {
                    if (k < n) ru[r] = *reinterpret_cast<const float4 *>(src + k);
                } else {
                    if (k < n) ru[r].x = src[k];
                    if (k + 1 < n) ru[r].y = src[k + 1];
                    if (k + 2 < n) ru[r].z = src[k + 2];
                    if (k + 3 < n) ru[r].w = src[k + 3];
                }
            }
        }
    };
    auto store = [&](int b) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int t = tid % TT, k = 4 * (tid / TT + 2 * r);
            Us[b][k][t] = ru[r].x;
            Us[b][k + 1][t] = ru[r].y;
            Us[b][k + 2][t] = ru[r].z;
            Us[b][k + 3][t] = ru[r].w;
        }
        row_cp_wait_all();
    };
    float2 acc[RT][NC];
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[a][c] = make_float2(0.f, 0.f);
    const int nk = nkp / kRK;
    load(0, 0);
    store(0);
    __syncthreads();
    for (int kc = 0; kc < nk; ++kc) {
        const int b = kc & 1;
        if (kc + 1 < nk) load(kc + 1, b ^ 1);  // last read before the previous barrier
#pragma unroll 4
        for (int k = 0; k < kRK; ++k) {
            const float4 w0 = *reinterpret_cast<const float4 *>(&Us[b][k][RT * ty]);
            const float4 w1 = *reinterpret_cast<const float4 *>(&Us[b][k][RT * ty + 4]);
            const float uv[RT] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
            float2 mv[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) mv[c] = *reinterpret_cast<const float2 *>(&Ms[b][k][2 * tx + 32 * c]);
#pragma unroll
            for (int a = 0; a < RT; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[a][c] = __ffma2_rn(make_float2(uv[a], uv[a]), mv[c], acc[a][c]);
        }
        if (kc + 1 < nk) {
            store(b ^ 1);
            __syncthreads();
        }
    }
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        const int64_t ti = t0 + RT * ty + a;
        if (ti >= t_end) continue;
        const int32_t t = targets[ti];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int j = j0 + 2 * tx + 32 * c;
            row_store<float>(acc[a][c].x, t, j, n, out, accumulate, dbar, g);
            row_store<float>(acc[a][c].y, t, j + 1, n, out, accumulate, dbar, g);
        }
    }
}

// 4 RW rows by 32 outputs: warp w rows RW w .. RW w + RW - 1, a lane per
// output.  RW = 4, or 1 for levels of so few rows that their blocks leave SMs
// idle (a tile's sums take 2 us in FP32, 7 on one SM's FP64 lanes at n_s = 56).
// VEC: the input rows are 16-byte aligned (FP32: n a multiple of 4; FP64: n
// even, as every n_s is).
constexpr int kSmallCols = 32;
template <typename T>
inline size_t rows_small_smem(int nkp, int rw = 4) {
    return sizeof(T) * ((size_t)nkp * kSmallCols + (size_t)(4 * rw) * (nkp + 4));
}
template <typename T, bool VEC, int RW>
__global__ void __launch_bounds__(kRThreads)
    k_rows_small(RowMap<T> g, const int32_t *__restrict__ targets, ClassRanges cr, int n, int nkp, int ldp,
                 const T *__restrict__ in, T *out, int accumulate, double *dbar) {
    constexpr int kV = 16 / sizeof(T);                   // values per 16-byte copy
    constexpr int kRows = 4 * RW, kPer = kRThreads / kRows;  // rows, staging threads per row
    extern __shared__ __align__(16) unsigned char rows_sm[];
    T *Ms = reinterpret_cast<T *>(rows_sm);              // [nkp][32]
    const int ldu = nkp + 4;                             // rows on other banks, 16-byte aligned
    T *Us = Ms + (size_t)nkp * kSmallCols;               // [kRows][ldu]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cls = blockIdx.y, j0 = blockIdx.z * kSmallCols;
    int64_t t_begin = 0, t_end = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c == cls) t_begin = cr.b[c], t_end = cr.b[c + 1];
    const int64_t t0 = t_begin + (int64_t)blockIdx.x * kRows;
    if (t0 >= t_end) return;  // uniform for the block
    const T *M = g.op(cls) + j0;
    // rows: thread t stages row t / kPer, 16-byte pieces t % kPer, + kPer, ...
    const int64_t tr = t0 + tid / kPer;
    const int row = tr < t_end ? g.src(targets[tr]) : -1;
    const T *src = in + (size_t)(row >= 0 ? row : 0) * n;
    T *du = Us + (tid / kPer) * ldu;
    const int step = (nkp / 4 + 15) / 16 * 16;           // inputs per group of copies (four groups)
    for (int q = 0; q < 4; ++q) {
        const int k0 = min(nkp, q * step), k1 = min(nkp, k0 + step);
        constexpr int kPieces = kSmallCols / kV;
        for (int e = tid; e < (k1 - k0) * kPieces; e += kRThreads) {
            const int k = k0 + e / kPieces, c = kV * (e % kPieces);
            row_cp16(Ms + (size_t)k * kSmallCols + c, M + (size_t)k * ldp + c);
        }
        for (int k = k0 + kV * (tid % kPer); k < k1; k += kPer * kV) {
            if (VEC && row >= 0 && k < n) {
                row_cp16(du + k, src + k);
            } else {
#pragma unroll
                for (int i = 0; i < kV; ++i) du[k + i] = (!VEC && row >= 0 && k + i < n) ? src[k + i] : T(0);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    T acc[RW];
#pragma unroll
    for (int a = 0; a < RW; ++a) acc[a] = T(0);
    const T *u0 = Us + RW * warp * ldu, *m0 = Ms + lane;
    auto sum = [&](int q) {
        __syncthreads();
        const int k0 = min(nkp, q * step), k1 = min(nkp, k0 + step);
#pragma unroll 2
        for (int k = k0; k < k1; k += 4) {
            T u[RW][4], m[4];
#pragma unroll
            for (int a = 0; a < RW; ++a) {
                if constexpr (sizeof(T) == 4) {
                    const float4 w = *reinterpret_cast<const float4 *>(u0 + a * ldu + k);
                    u[a][0] = w.x, u[a][1] = w.y, u[a][2] = w.z, u[a][3] = w.w;
                } else {
                    const double2 w = *reinterpret_cast<const double2 *>(u0 + a * ldu + k);
                    const double2 x = *reinterpret_cast<const double2 *>(u0 + a * ldu + k + 2);
                    u[a][0] = w.x, u[a][1] = w.y, u[a][2] = x.x, u[a][3] = x.y;
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) m[i] = m0[(k + i) * kSmallCols];
#pragma unroll
            for (int a = 0; a < RW; ++a)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[a] = fma(u[a][i], m[i], acc[a]);
        }
    };
    asm volatile("cp.async.wait_group 3;" ::: "memory");
    sum(0);
    asm volatile("cp.async.wait_group 2;" ::: "memory");
    sum(1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    sum(2);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    sum(3);
#pragma unroll
    for (int a = 0; a < RW; ++a) {
        const int64_t ti = t0 + RW * warp + a;
        if (ti < t_end) row_store<T>(acc[a], targets[ti], j0 + lane, n, out, accumulate, dbar, g);
    }
}

}  // namespace

// Column pairs per 16 threads (NC) of the big tile for ld outputs, and the
// operators' padded row length: the least padding, the wider tile on a tie.
inline int gemm_nc(int ld) {
    int best = 5, least = 1 << 30;
    for (int nc = 5; nc >= 1; --nc) {
        const int l = (ld + 32 * nc - 1) / (32 * nc) * 32 * nc;
        if (l < least) least = l, best = nc;
    }
    return best;
}
inline int gemm_ldp(int ld) {
    const int w = 32 * gemm_nc(ld);
    return (ld + w - 1) / w * w;
}
inline int gemm_nkp(int n) { return (n + 15) / 16 * 16; }

}  // namespace kifmm
