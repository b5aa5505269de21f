// M2L in FP32 arithmetic on the SIMT cores, for the FP32 Stokeslet and FP32
// periodic cells, whose outputs keep the bits of a sum of FMAs (the
// Stokeslet's regularised operators keep a near-null density that amplifies
// any FP32 rounding of the translations to 6e-5 of the velocities at p = 6, so
// that the exact-split products of m2l_exact.cu, closer to the exact
// translations, move the velocities by that much).
//
//     d(t) = sum_{s < 189} M_{off(c,s)} u(src(t, s))
//
// Every slot sums its products in input order, one FMA each, into a fresh
// partial that is added to the running total in slot order.
//
// FMA-bound: 2 n^2 flops per V entry.  A block of 128 threads owns 8 RT
// targets of one octant class by 32 NC outputs, a thread RT targets by NC
// pairs of outputs, on packed f32x2 FMAs (each half rounds as a scalar FMA;
// packed they reach 111 lanes per clock and SM, three-operand scalar ones 82).
// The inputs are staged once and paired (u, u) in registers; the operators,
// padded to whole blocks of 16 inputs x 32 NC outputs at plan time, come by
// 16-byte asynchronous copies without bounds tests.  One barrier per 16 inputs
// (two buffers).
//
// SPLIT: a small tree has too few blocks for the SMs and its time is 189 slots
// in a row, whatever its size.  blockIdx.z then takes a range of the slots,
// every slot's partial is stored and k_simt_sum adds them in slot order:
// the additions, and so the bits, of the unsplit form.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace kifmm {

namespace {

constexpr int kSK = 16;         // inputs per staged chunk
constexpr int kSThreads = 128;  // 16 threads across the outputs, 8 across the targets

template <int RT, int NC>
struct SimtSmem {
    float u[2][kSK][8 * RT];
    float m[2][kSK][32 * NC];
};

struct ClassStarts {
    int64_t b[9];  // target range of each octant class
};

__device__ __forceinline__ void cp16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

struct SimtArgs {
    const int32_t *targets;  // class-major target boxes
    ClassStarts cs;
    const int32_t *vdense;   // [nb][189]
    const int *slot_off;     // [8][189]
    const float *ops;        // [316][nkp][ldp], zero padded
    const float *in;         // [nb][n]
    float *out;              // [nb][n]
    double *dbar;            // [nb]: output column n (the mean row), or nullptr
    float *part;             // SPLIT: [slot of the round][target][ldp]
    int n, nkp, ldp, ncb;    // column blocks of 32 NC
    int slot0, nslots;       // SPLIT: the slots of this launch
};

constexpr int simt_blocks(int rt, int nc, bool split) {  // blocks per SM the registers are held to
    return rt * nc >= 32 ? (split ? 3 : 2) : (rt * nc >= 20 ? (split ? 4 : 3) : 4);
}

// VEC: the input rows are 16-byte aligned (n a multiple of 4).
template <int RT, int NC, bool VEC, bool SPLIT>
__global__ void __launch_bounds__(kSThreads, simt_blocks(RT, NC, SPLIT)) k_m2l_simt(SimtArgs a) {
    constexpr int TT = 8 * RT, TJ = 32 * NC;
    extern __shared__ __align__(16) unsigned char simt_sm[];
    SimtSmem<RT, NC> &S = *reinterpret_cast<SimtSmem<RT, NC> *>(simt_sm);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int cls = blockIdx.y, zr = SPLIT ? (int)blockIdx.z / a.ncb : 0;
    const int j0 = (SPLIT ? (int)blockIdx.z - zr * a.ncb : (int)blockIdx.z) * TJ;
    const int n = a.n, ldp = a.ldp;
    const int64_t t_end = a.cs.b[cls + 1], t0 = a.cs.b[cls] + (int64_t)blockIdx.x * TT;
    if (t0 >= t_end) return;  // uniform for the block
    const int nz = SPLIT ? (int)gridDim.z / a.ncb : 1;
    const int s_lo = SPLIT ? a.slot0 + a.nslots * zr / nz : 0;
    const int s_hi = SPLIT ? a.slot0 + a.nslots * (zr + 1) / nz : kVSlots;
    float2 acc[RT][NC], run[RT][NC];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[r][c] = run[r][c] = make_float2(0.f, 0.f);
    const int nk = a.nkp / kSK;
    // staging: input quad (target e % TT, inputs 4 (e / TT)); operator quads
    // (input, outputs 4 q) in order, NC per thread
    constexpr int kQ = (TT * (kSK / 4) + kSThreads - 1) / kSThreads;
    constexpr bool kAll = TT * (kSK / 4) >= kSThreads;  // every thread has a quad
    int32_t row[kQ], tgt[kQ];
#pragma unroll
    for (int r = 0; r < kQ; ++r) {
        const int e = tid + kSThreads * r;
        const int64_t t = t0 + e % TT;
        tgt[r] = ((kAll || e < TT * (kSK / 4)) && t < t_end) ? a.targets[t] : -1;
    }
    int moff[NC];
#pragma unroll
    for (int r = 0; r < NC; ++r) {
        const int e = tid + kSThreads * r, k = e / (TJ / 4);
        moff[r] = k * ldp + 4 * (e - k * (TJ / 4));
    }
    float4 ru[kQ];
    for (int s = s_lo; s < s_hi; ++s) {
        bool any = false;
#pragma unroll
        for (int r = 0; r < kQ; ++r) {
            row[r] = tgt[r] >= 0 ? a.vdense[(size_t)tgt[r] * kVSlots + s] : -1;
            any = any || row[r] >= 0;
        }
        // (a slot without a source in this tile adds zero to every total);
        // the barrier also frees both buffers of the previous slot
        const bool some = __syncthreads_or(any);
        if (!SPLIT && !some) continue;
        if (some) {
            const float *M = a.ops + (size_t)a.slot_off[cls * kVSlots + s] * a.nkp * ldp + j0;
            auto load = [&](int kc, int b) {
                const float *Mk = M + (size_t)kc * kSK * ldp;
#pragma unroll
                for (int r = 0; r < NC; ++r) cp16(&S.m[b][0][0] + 4 * (tid + kSThreads * r), Mk + moff[r]);
#pragma unroll
                for (int r = 0; r < kQ; ++r) {
                    const int k = kc * kSK + 4 * ((tid + kSThreads * r) / TT);
                    ru[r] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (row[r] >= 0) {
                        const float *p = a.in + (size_t)row[r] * n + k;
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
                    float2 mv[NC];
#pragma unroll
                    for (int r = 0; r < RT; r += 4) {
                        const float4 w = *reinterpret_cast<const float4 *>(su + k * TT + r);
                        uv[r] = w.x, uv[r + 1] = w.y, uv[r + 2] = w.z, uv[r + 3] = w.w;
                    }
#pragma unroll
                    for (int c = 0; c < NC; ++c) mv[c] = *reinterpret_cast<const float2 *>(sm + k * TJ + 32 * c);
#pragma unroll
                    for (int r = 0; r < RT; ++r)
#pragma unroll
                        for (int c = 0; c < NC; ++c) acc[r][c] = __ffma2_rn(make_float2(uv[r], uv[r]), mv[c], acc[r][c]);
                }
                if (kc + 1 < nk) {
                    store(b ^ 1);
                    __syncthreads();
                }
            }
        }
        if constexpr (SPLIT) {
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const int64_t ti = t0 + RT * ty + r;
                float *o = a.part + ((size_t)(s - a.slot0) * a.cs.b[8] + ti) * ldp + j0 + 2 * tx;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (ti < t_end) *reinterpret_cast<float2 *>(o + 32 * c) = acc[r][c];
                    acc[r][c] = make_float2(0.f, 0.f);
                }
            }
        } else {
#pragma unroll
            for (int r = 0; r < RT; ++r)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    run[r][c] = __fadd2_rn(run[r][c], acc[r][c]);
                    acc[r][c] = make_float2(0.f, 0.f);
                }
        }
    }
    if constexpr (!SPLIT) {
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const int64_t ti = t0 + RT * ty + r;
            if (ti >= t_end) continue;
            const int32_t t = a.targets[ti];
#pragma unroll
            for (int c = 0; c < NC; ++c)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int j = j0 + 2 * tx + 32 * c + e;
                    const float v = e ? run[r][c].y : run[r][c].x;
                    if (j < n) a.out[(size_t)t * n + j] = v;
                    else if (j == n && a.dbar) a.dbar[t] = (double)v;
                }
        }
    }
}

// The round's partials added to the running sums, in slot order (carry: the
// sums between rounds, [target][ldp]).
constexpr int kSumSlots = 21;  // loads in flight per thread; a round is a multiple of it
__global__ void __launch_bounds__(256) k_simt_sum(const int32_t *__restrict__ targets, int64_t n_t, int n, int ld,
                                                  int ldp, int nslots, const float *__restrict__ part, float *carry,
                                                  int first, int last, float *__restrict__ out,
                                                  double *__restrict__ dbar) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_t * ld) return;
    const int64_t i = idx / ld;
    const int j = (int)(idx - i * ld);
    const size_t at = (size_t)i * ldp + j, step = (size_t)n_t * ldp;
    float v = first ? 0.f : carry[at];
    for (int s0 = 0; s0 < nslots; s0 += kSumSlots) {
        float p[kSumSlots];
#pragma unroll
        for (int k = 0; k < kSumSlots; ++k) p[k] = part[(s0 + k) * step + at];
#pragma unroll
        for (int k = 0; k < kSumSlots; ++k) v += p[k];
    }
    if (!last) {
        carry[at] = v;
        return;
    }
    const int32_t t = targets[i];
    if (j < n) out[(size_t)t * n + j] = v;
    else if (dbar) dbar[t] = (double)v;
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

// Column pairs per 16 threads (NC) of a plan with ld outputs: the least padded
// width over the FMA rate its tile reaches (measured at 20 k targets, RT = 8,
// padding counted: 88, 82, 85, 70 and 50 lanes per clock and SM for 160 ... 32
// columns).  n = 56 + 1 (p = 4) on 64 columns instead of 160: 441 -> 60 us at
// 576 targets, with the slots split.
int simt_nc(int ld) {
    const double rate[6] = {0.0, 50.0, 70.0, 85.0, 82.0, 88.0};
    int best = 5;
    double least = 1e30;
    for (int nc = 5; nc >= 1; --nc) {
        const double t = pad_to(ld, 32 * nc) / rate[nc];
        if (t < least) least = t, best = nc;
    }
    return best;
}

template <int RT, int NC, bool VEC, bool SPLIT>
cudaError_t simt_launch(const SimtArgs &a, int64_t most, int z, cudaStream_t s) {
    const dim3 grid((unsigned)((most + 8 * RT - 1) / (8 * RT)), 8, (unsigned)(a.ncb * z));
    ++g_launches, k_m2l_simt<RT, NC, VEC, SPLIT><<<grid, kSThreads, sizeof(SimtSmem<RT, NC>), s>>>(a);
    return cudaGetLastError();
}
template <int NC, bool VEC>
cudaError_t simt_launch_nc(const SimtArgs &a, int rt, bool split, int64_t most, int z, cudaStream_t s) {
    if (split) return rt == 8 ? simt_launch<8, NC, VEC, true>(a, most, z, s) : simt_launch<4, NC, VEC, true>(a, most, z, s);
    return rt == 8 ? simt_launch<8, NC, VEC, false>(a, most, 1, s) : simt_launch<4, NC, VEC, false>(a, most, 1, s);
}
template <bool VEC>
cudaError_t simt_launch_vec(const SimtArgs &a, int nc, int rt, bool split, int64_t most, int z, cudaStream_t s) {
    switch (nc) {
        case 1: return simt_launch_nc<1, VEC>(a, rt, split, most, z, s);
        case 2: return simt_launch_nc<2, VEC>(a, rt, split, most, z, s);
        case 3: return simt_launch_nc<3, VEC>(a, rt, split, most, z, s);
        case 4: return simt_launch_nc<4, VEC>(a, rt, split, most, z, s);
        default: return simt_launch_nc<5, VEC>(a, rt, split, most, z, s);
    }
}

struct SimtTree {
    int64_t most = 0;               // targets of the largest class
    int64_t blocks[2] = {0, 0};     // blocks of 64 and of 32 targets, all column blocks
    int ldp = 0, ncb = 0;
};
SimtTree simt_tree(const Plan &P) {
    SimtTree t;
    const int nc = simt_nc(P.op_ld);
    t.ldp = pad_to(P.op_ld, 32 * nc);
    t.ncb = t.ldp / (32 * nc);
    for (int c = 0; c < 8; ++c) {
        const int64_t n = P.m2l_class_start[c + 1] - P.m2l_class_start[c];
        t.most = std::max(t.most, n);
        for (int k = 0; k < 2; ++k) t.blocks[k] += (n + (64 >> k) - 1) / (64 >> k) * t.ncb;
    }
    return t;
}

// Slots per round of a split whose partial products and carried sums fit
// `room`; 0: none.  At most three rounds: the partial products of a larger
// tree cost more than its fuller SMs give.
int simt_round(const Plan &P, const SimtTree &t, size_t room) {
    const size_t slot = sizeof(float) * (size_t)P.m2l_class_start[8] * t.ldp;
    if (slot == 0) return 0;
    for (const int g : {9, 5, 3})  // groups of kSumSlots slots: 1, 2 or 3 rounds
        if (slot * (g * kSumSlots + (g < kVSlots / kSumSlots ? 1 : 0)) <= room) return g * kSumSlots;
    return 0;
}

}  // namespace

// Plan time: the operators in their padded form (in place of m2l_t).
cudaError_t m2l_simt_setup(Plan &P) {
    const int nkp = pad_to(P.ns, kSK), ldp = pad_to(P.op_ld, 32 * simt_nc(P.op_ld));
    const int64_t total = (int64_t)kNumM2L * nkp * ldp;
    void *padded = nullptr;
    KIFMM_CUDA_TRY(plan_alloc(P, &padded, sizeof(float) * total));
    ++g_launches, k_pad_ops<<<(unsigned)((total + 255) / 256), 256>>>(total, P.ns, P.op_ld, nkp, ldp,
                                                                     (const float *)P.m2l_t, (float *)padded);
    KIFMM_CUDA_TRY(cudaDeviceSynchronize());
    plan_free(P, &P.m2l_t);
    P.m2l_t = padded;
    return cudaSuccess;
}

size_t m2l_simt_part_bytes(const Plan &P, size_t room) {
    const SimtTree t = simt_tree(P);
    const int round = simt_round(P, t, room);
    return sizeof(float) * (size_t)P.m2l_class_start[8] * t.ldp * (round + (round && round < kVSlots ? 1 : 0));
}

// The slots are split whenever their partial products have room: a block then
// keeps no running sums, so an SM holds one or two more of them, and the CTAs'
// lengths even out.  Measured (FP32 periodic, p = 4 / 6; whole slots against
// split ones): 576 targets 441 -> 60 / 1060 -> 204 us, 4672 targets 442 -> 249 /
// 1469 -> 950, 20 k targets 1078 -> 919 / 4.9 ms, unsplit.  64 targets per block
// from half an SM's worth of blocks on (4672 targets, p = 4: 249 us, 269 with 32;
// 576 targets: 65 against 60), and ranges of three slots or more, up to 32 of
// them, so that the last wave is short.  Whole steps, against whole slots on 160
// columns: a periodic cell of 8k charges, p = 4, 940 -> 473 us, p = 6, 1827 -> 667;
// 150k, p = 6, 2247 -> 1720; Stokeslet, 2k points, p = 6, 4226 -> 833.  Unsplit, the height is the one whose
// fullest SM is estimated to finish first, at 95 and 82 lanes (4672 targets of n
// = 456 are 240 blocks of 64 on 152 SMs, or three of 32 on each).
cudaError_t m2l_simt(Plan &P, const float *u, float *d, double *dbar, cudaStream_t s) {
    const SimtTree t = simt_tree(P);
    if (t.most == 0) return cudaSuccess;  // no V-list targets
    const int nc = simt_nc(P.op_ld), round = simt_round(P, t, P.m2l_part_bytes);
    SimtArgs a;
    a.targets = P.m2l_targets;
    for (int c = 0; c <= 8; ++c) a.cs.b[c] = P.m2l_class_start[c];
    a.vdense = P.vdense;
    a.slot_off = P.slot_off;
    a.ops = (const float *)P.m2l_t;
    a.in = u;
    a.out = d;
    a.dbar = dbar;
    a.part = (float *)P.m2l_part;
    a.n = P.ns;
    a.nkp = pad_to(P.ns, kSK);
    a.ldp = t.ldp;
    a.ncb = t.ncb;
    a.slot0 = 0;
    a.nslots = kVSlots;
    auto launch = [&](int rt, bool split, int z) {
        return P.ns % 4 == 0 ? simt_launch_vec<true>(a, nc, rt, split, t.most, z, s)
                             : simt_launch_vec<false>(a, nc, rt, split, t.most, z, s);
    };
    if (round == 0) {
        const double rate[2] = {95.0, 82.0};
        double time[2];
        for (int k = 0; k < 2; ++k)
            time[k] = (double)((t.blocks[k] + P.num_sms - 1) / P.num_sms) * (64 >> k) / rate[k];
        return launch(time[1] < 0.97 * time[0] ? 4 : 8, false, 1);
    }
    const int64_t n_t = P.m2l_class_start[8];
    const int rt = 2 * t.blocks[0] >= P.num_sms ? 8 : 4;
    float *carry = a.part + (size_t)round * n_t * t.ldp;
    for (; a.slot0 < kVSlots; a.slot0 += round) {
        a.nslots = std::min(round, kVSlots - a.slot0);
        KIFMM_CUDA_TRY(launch(rt, true, std::min(32, a.nslots / 3)));
        ++g_launches, k_simt_sum<<<(unsigned)((n_t * P.op_ld + 255) / 256), 256, 0, s>>>(
                          P.m2l_targets, n_t, P.ns, P.op_ld, t.ldp, a.nslots, a.part, carry, a.slot0 == 0,
                          a.slot0 + a.nslots == kVSlots, d, dbar);
    }
    return cudaGetLastError();
}

}  // namespace kifmm
