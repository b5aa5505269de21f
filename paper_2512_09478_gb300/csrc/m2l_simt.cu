// M2L in FP32 arithmetic on the SIMT cores, for the plans whose outputs hang
// on the rounding of this stage: the Stokeslet in FP32 (its regularised
// operators keep a near-null density that amplifies any FP32 rounding of the
// translations to 6e-5 of the velocities at p = 6; the exact-split products of
// m2l_exact.cu are closer to the exact translations but move the velocities by
// that much) and FP32 periodic cells (whose energy comes back in FP64).
//
//     d(t) = sum_{s < 189} M_{off(c,s)} u(src(t, s))
//
// Every slot sums its products in input order, one FMA each, into a fresh
// partial that is added to the running total in slot order.
//
// FMA-bound: 2 n^2 flops per V entry.  A block of 128 threads owns 8 RT
// targets of one octant class by 160 outputs, a thread RT targets by five
// pairs of outputs, on packed f32x2 FMAs (each half rounds as a scalar FMA;
// packed they reach 111 lanes per clock and SM, three-operand scalar ones 82):
// at RT = 8, 40 of them per input for seven shared-memory reads.  The inputs
// are staged once and paired (u, u) in registers (the loop alone: 95 lanes per
// clock and SM, 86 with staged pairs); the operators, padded to whole blocks of 16 inputs x 160 outputs at
// plan time, come by 16-byte asynchronous copies without bounds tests.  One
// barrier per 16 inputs (two buffers).  Stokeslet, 60k points, p = 6 (4672
// targets, n = 456): 27.1 ms with 16 x 32 tiles of scalar FMAs, 11.7 here,
// where 240 blocks on 152 SMs leave 6.7 at the FMA rate.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace kifmm {

namespace {

constexpr int kSK = 16;         // inputs per staged chunk
constexpr int kSCols = 160;     // outputs per block
constexpr int kSThreads = 128;  // 16 threads across the outputs, 8 across the targets

template <int RT>
struct SimtSmem {
    float u[2][kSK][8 * RT];
    float m[2][kSK][kSCols];
};

struct ClassStarts {
    int64_t b[9];  // target range of each octant class
};

__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ops: [316][nkp][ldp], nkp and ldp the inputs and outputs padded with zeros
// to multiples of kSK and kSCols.  VEC: the input rows are 16-byte aligned (n
// a multiple of 4).
template <int RT, bool VEC>
__global__ void __launch_bounds__(kSThreads, RT == 8 ? 2 : (RT == 4 ? 3 : 4))
    k_m2l_simt(const int32_t *__restrict__ targets, ClassStarts cs, const int32_t *__restrict__ vdense,
               const int *__restrict__ slot_off, const float *__restrict__ ops, int n, int nkp, int ldp,
               const float *__restrict__ in, float *__restrict__ out, double *__restrict__ dbar) {
    constexpr int TT = 8 * RT;
    extern __shared__ __align__(16) unsigned char simt_sm[];
    SimtSmem<RT> &S = *reinterpret_cast<SimtSmem<RT> *>(simt_sm);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int cls = blockIdx.y, j0 = blockIdx.z * kSCols;
    const int64_t t_end = cs.b[cls + 1], t0 = cs.b[cls] + (int64_t)blockIdx.x * TT;
    if (t0 >= t_end) return;  // uniform for the block
    float2 acc[RT][5], run[RT][5];
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
        for (int c = 0; c < 5; ++c) acc[a][c] = run[a][c] = make_float2(0.f, 0.f);
    const int nk = nkp / kSK;
    // staging: input quad (target e % TT, inputs 4 (e / TT)); operator quads
    // (input, outputs 4 q) in order, five per thread
    constexpr int kQ = (TT * (kSK / 4) + kSThreads - 1) / kSThreads;
    constexpr bool kAll = TT * (kSK / 4) >= kSThreads;  // every thread has a quad
    constexpr int kMQ = kSK * kSCols / 4 / kSThreads;
    static_assert(kMQ * 4 * kSThreads == kSK * kSCols, "whole operator quads per thread");
    int32_t row[kQ], tgt[kQ];
#pragma unroll
    for (int r = 0; r < kQ; ++r) {
        const int e = tid + kSThreads * r;
        const int64_t t = t0 + e % TT;
        tgt[r] = ((kAll || e < TT * (kSK / 4)) && t < t_end) ? targets[t] : -1;
    }
    // operator quad r of this thread: input mk[r], outputs mj[r] .. + 3
    int moff[kMQ];
#pragma unroll
    for (int r = 0; r < kMQ; ++r) {
        const int e = tid + kSThreads * r, k = e / (kSCols / 4);
        moff[r] = k * ldp + 4 * (e - k * (kSCols / 4));
    }
    float4 ru[kQ];
    for (int s = 0; s < kVSlots; ++s) {
        bool any = false;
#pragma unroll
        for (int r = 0; r < kQ; ++r) {
            row[r] = tgt[r] >= 0 ? vdense[(size_t)tgt[r] * kVSlots + s] : -1;
            any = any || row[r] >= 0;
        }
        // (a slot without a source in this tile adds zero to every total);
        // the barrier also frees both buffers of the previous slot
        if (!__syncthreads_or(any)) continue;
        const float *M = ops + (size_t)slot_off[cls * kVSlots + s] * nkp * ldp + j0;
        auto load = [&](int kc, int b) {
            const float *Mk = M + (size_t)kc * kSK * ldp;
#pragma unroll
            for (int r = 0; r < kMQ; ++r) cp16(&S.m[b][0][0] + 4 * (tid + kSThreads * r), Mk + moff[r]);
#pragma unroll
            for (int r = 0; r < kQ; ++r) {
                const int k = kc * kSK + 4 * ((tid + kSThreads * r) / TT);
                ru[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (row[r] >= 0) {
                    const float *p = in + (size_t)row[r] * n + k;
                    if (VEC) {
                        if (k < n) ru[r] = *reinterpret_cast<const float4 *>(p);
                    } else {
                        if (k < n) ru[r].x = p[0];
                        if (k + 1 < n) ru[r].y = p[1];
                        if (k + 2 < n) ru[r].z = p[2];
                        if (k + 3 < n) ru[r].w = p[3];
                    }
                }
            }
        };
        auto store = [&](int b) {
#pragma unroll
            for (int r = 0; r < kQ; ++r) {
                const int e = tid + kSThreads * r, t = e % TT, k = 4 * (e / TT);
                if (!kAll && e >= TT * (kSK / 4)) continue;
                S.u[b][k][t] = ru[r].x;
                S.u[b][k + 1][t] = ru[r].y;
                S.u[b][k + 2][t] = ru[r].z;
                S.u[b][k + 3][t] = ru[r].w;
            }
            cp_wait_all();
        };
        load(0, 0);
        store(0);
        __syncthreads();
        for (int kc = 0; kc < nk; ++kc) {
            const int b = kc & 1;
            if (kc + 1 < nk) load(kc + 1, b ^ 1);  // last read before the previous barrier
            const float *su = &S.u[b][0][RT * ty];
            const float *sm = &S.m[b][0][2 * tx];
#pragma unroll 4
            for (int k = 0; k < kSK; ++k) {
                float uv[RT];
                float2 mv[5];
#pragma unroll
                for (int a = 0; a < RT; a += 4) {
                    if constexpr (RT >= 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(su + k * TT + a);
                        uv[a] = w.x, uv[a + 1] = w.y, uv[a + 2] = w.z, uv[a + 3] = w.w;
                    } else {
                        const float2 w = *reinterpret_cast<const float2 *>(su + k * TT);
                        uv[0] = w.x, uv[1] = w.y;
                    }
                }
#pragma unroll
                for (int c = 0; c < 5; ++c) mv[c] = *reinterpret_cast<const float2 *>(sm + k * kSCols + 32 * c);
#pragma unroll
                for (int a = 0; a < RT; ++a)
#pragma unroll
                    for (int c = 0; c < 5; ++c) acc[a][c] = __ffma2_rn(make_float2(uv[a], uv[a]), mv[c], acc[a][c]);
            }
            if (kc + 1 < nk) {
                store(b ^ 1);
                __syncthreads();
            }
        }
#pragma unroll
        for (int a = 0; a < RT; ++a)
#pragma unroll
            for (int c = 0; c < 5; ++c) {
                run[a][c] = __fadd2_rn(run[a][c], acc[a][c]);
                acc[a][c] = make_float2(0.f, 0.f);
            }
    }
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        const int64_t ti = t0 + RT * ty + a;
        if (ti >= t_end) continue;
        const int32_t t = targets[ti];
#pragma unroll
        for (int c = 0; c < 5; ++c)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int j = j0 + 2 * tx + 32 * c + e;
                const float v = e ? run[a][c].y : run[a][c].x;
                if (j < n) out[(size_t)t * n + j] = v;
                else if (j == n && dbar) dbar[t] = (double)v;
            }
    }
}

// [316][n][ld] operators to [316][nkp][ldp], zero padded.
__global__ void k_pad_ops(int64_t total, int n, int ld, int nkp, int ldp, const float *__restrict__ in,
                          float *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int64_t row = i / ldp;
    const int j = (int)(i - row * ldp), k = (int)(row % nkp);
    out[i] = (k < n && j < ld) ? in[((row / nkp) * n + k) * ld + j] : 0.f;
}

int pad_to(int x, int m) { return (x + m - 1) / m * m; }

template <int RT>
cudaError_t simt_launch(Plan &P, int64_t most, const float *u, float *d, double *dbar, cudaStream_t s) {
    const dim3 grid((unsigned)((most + 8 * RT - 1) / (8 * RT)), 8, (unsigned)((P.op_ld + kSCols - 1) / kSCols));
    const size_t smem = sizeof(SimtSmem<RT>);
    ClassStarts cs;
    for (int c = 0; c <= 8; ++c) cs.b[c] = P.m2l_class_start[c];
    const int nkp = pad_to(P.ns, kSK), ldp = pad_to(P.op_ld, kSCols);
    if (P.ns % 4 == 0)
        ++g_launches, k_m2l_simt<RT, true><<<grid, kSThreads, smem, s>>>(P.m2l_targets, cs, P.vdense, P.slot_off,
                                                                        (const float *)P.m2l_t, P.ns, nkp, ldp, u, d,
                                                                        dbar);
    else
        ++g_launches, k_m2l_simt<RT, false><<<grid, kSThreads, smem, s>>>(P.m2l_targets, cs, P.vdense, P.slot_off,
                                                                         (const float *)P.m2l_t, P.ns, nkp, ldp, u, d,
                                                                         dbar);
    return cudaGetLastError();
}

}  // namespace

// Plan time: the operators in their padded form (in place of m2l_t).
cudaError_t m2l_simt_setup(Plan &P) {
    const int nkp = pad_to(P.ns, kSK), ldp = pad_to(P.op_ld, kSCols);
    const int64_t total = (int64_t)kNumM2L * nkp * ldp;
    void *padded = nullptr;
    KIFMM_CUDA_TRY(plan_alloc(P, &padded, sizeof(float) * total));
    ++g_launches, k_pad_ops<<<(unsigned)((total + 255) / 256), 256>>>(total, P.ns, P.op_ld, nkp, ldp,
                                                                     (const float *)P.m2l_t, (float *)padded);
    KIFMM_CUDA_TRY(cudaDeviceSynchronize());
    plan_free(P, &P.m2l_t);
    P.m2l_t = padded;
    const auto dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_m2l_simt<8, true>, dyn, (int)sizeof(SimtSmem<8>)));
    return cudaFuncSetAttribute(k_m2l_simt<8, false>, dyn, (int)sizeof(SimtSmem<8>));
}

// 64, 32 or 16 targets per block, whichever is estimated to finish first: the
// fullest SM's blocks times their targets, over the FMA rate of the tile (95,
// 82 and 60 lanes per clock and SM: smaller tiles read shared memory more per
// FMA, but share out more evenly; 4672 targets of n = 456 are 240 blocks of 64
// on 152 SMs, or three of 32 on each).
cudaError_t m2l_simt(Plan &P, const float *u, float *d, double *dbar, cudaStream_t s) {
    int64_t most = 0;
    int64_t blocks[3] = {0, 0, 0};
    for (int c = 0; c < 8; ++c) {
        const int64_t t = P.m2l_class_start[c + 1] - P.m2l_class_start[c];
        most = std::max(most, t);
        for (int k = 0; k < 3; ++k) blocks[k] += (t + (64 >> k) - 1) / (64 >> k);
    }
    if (most == 0) return cudaSuccess;  // no V-list targets
    const int64_t ncb = (P.op_ld + kSCols - 1) / kSCols;
    const double rate[3] = {95.0, 82.0, 60.0};
    int pick = 0;
    double least = 1e30;
    for (int k = 0; k < 3; ++k) {
        const double t = (double)((blocks[k] * ncb + P.num_sms - 1) / P.num_sms) * (64 >> k) / rate[k];
        if (t < 0.97 * least) least = t, pick = k;
    }
    if (pick == 0) return simt_launch<8>(P, most, u, d, dbar, s);
    return pick == 1 ? simt_launch<4>(P, most, u, d, dbar, s) : simt_launch<2>(P, most, u, d, dbar, s);
}

}  // namespace kifmm
