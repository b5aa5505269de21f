// M2L at full FP32 or FP64 accuracy on the Blackwell tensor cores (tcgen05 /
// TMEM): the V-list translations of the FP64 mode, of the FP32 mode in free
// space with the Laplace kernel (the other FP32 plans: m2l_simt.cu) and of every
// adjoint,
//     d(t) = sum_{s < 189} M_{off(c,s)} u(src(t, s)),
// as sums of 16-bit products that the tensor core adds without rounding.
//
// Every gathered row u(b) and every operator M_o is scaled by a power of two
// of its own so that its largest entry is at most 1, and cut into slices:
//
//   FP32 (three FP16 slices): x = 2^-8 (h + l + l2), h an integer (|h| <= 256),
//     l and l2 the FP16 roundings of what is left (31 bits in all).  h h is
//     summed in one accumulator, where at most 256 products of at most 2^16
//     stay below 2^24 and every sum is an exact integer; the five products
//     h l, l h, l l, h l2, l2 h, 2^-9 and less of it, in a second one.
//   FP64 (eight BF16 slices): x = 2^-6 sum_i 2^-8i d_i, balanced base-256
//     digits (|d_0| <= 64, |d_i| <= 128).  The products d_i d_j with i + j = g
//     <= 7 go to the accumulator of g, where (up to g = 6) at most 160 (g + 1)
//     of them sum to an integer below 2^24 (times 2^-8g), exactly; at g = 7,
//     2^-56 of the first, a rounding would be below 2^-79.
//     The accumulators of g and the slices of the operator lie side by side,
//     so one MMA of up to 256 columns multiplies slice i of the rows with four
//     slices j of the operator: 24 MMAs per stage for the 72 products, whose
//     issue one by one took longer than the tensor core does.
//     The split scheme is Ozaki, Ogita, Oishi & Rump (Numer. Algorithms 59,
//     2012) for error-free matrix products, with the digits of a fixed-point
//     expansion.
//
// The drain warps add the accumulators of one slot (FP32: one IEEE sum; FP64:
// one 64-bit integer, one conversion), times the two scales, to running sums
// in the compute type.  Measured against 80-bit sums on the Laplace operators
// (p = 4 ... 10, random sources): a translation's error is 0.06-0.2 of that
// of a sequential FP32 dot product, 0.07-0.2 of a sequential FP64 one.
//
// What bounds it: the FP64 unit runs 2 lanes per clock and SM (conversions
// included), so a SIMT product takes 128 x 152 x 152 / 2 = 1.5 M clocks per
// slot of a 128-target tile; here the tensor core takes 36 (FP64) or 6 (FP32)
// products of 128 x 160 x 160, 28 k and 5 k clocks, and two FP64 operations per
// output and slot are left.  FP32 waits for its stages' bytes, like the mixed
// kernel.  FP64 has one set of accumulators (eight groups of 64 columns are all
// of tensor memory), so a slot's products wait for the drain of the slot before:
// its stages, 96 KB each, arrive at some 13 bytes per clock and SM where the
// mixed kernel's reach 33.  Measured, M2L alone: FP64, 60k Plummer, p = 6: 30.7
// -> 1.95 ms; FP32, 200k packing, p = 6: 3.30 -> 0.29 ms (the gathered SIMT
// product before).
//
// Pipeline and bounded waits as in m2l_tc.cu: producer warps (cp.async
// of the gathered rows, one bulk copy of the operator block per stage), one
// MMA warp, eight drain warps; one CTA per SM.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace kifmm {

namespace {

constexpr int kKB = 32;             // 16-bit elements per stage row (64 bytes)
constexpr int kRowB = 64;
constexpr int kDrain = 8;           // drain warps

template <typename T>
struct Slicing;
template <>
struct Slicing<float> {
    static constexpr int kSlices = 3, kGroups = 2, kCols = 160, kChunkBlocks = 8;  // 8 x 32 x 2^16 = 2^24
    static constexpr int kProd = 4;                                                // producer warps
    static constexpr uint32_t kFmt = 0;                                            // FP16
};
template <>
struct Slicing<double> {
    static constexpr int kSlices = 8, kGroups = 8, kCols = 64, kChunkBlocks = 5;  // K <= 160 per accumulation
    static constexpr int kProd = 2;  // producer warps: 11 warps leave the drain 168 registers (64 bytes spill)
    static constexpr uint32_t kFmt = 1;                                           // BF16
};

template <typename T>
constexpr int ex_threads() {
    return 32 * (Slicing<T>::kProd + 1 + kDrain);
}

// Scale exponent: the least e with m <= 2^e (m > 0).
__device__ __forceinline__ int ceil_exp(float m) {
    int e;
    const float f = frexpf(m, &e);
    return f == 0.5f ? e - 1 : e;
}
__device__ __forceinline__ int ceil_exp(double m) {
    int e;
    const double f = frexp(m, &e);
    return f == 0.5 ? e - 1 : e;
}

// The slices of x, |x| <= 2^e, as 16-bit words.
__device__ __forceinline__ void slice_of(float x, int e, uint16_t (&w)[3]) {
    const float v = ldexpf(x, 8 - e), h = rintf(v), r = v - h;  // exact: r holds the trailing bits of v
    const __half hh = __float2half_rn(h), l = __float2half_rn(r);
    const __half l2 = __float2half_rn(r - __half2float(l));
    w[0] = __half_as_ushort(hh);
    w[1] = __half_as_ushort(l);
    w[2] = __half_as_ushort(l2);
}
__device__ __forceinline__ void slice_of(double x, int e, uint16_t (&w)[8]) {
    // 2^62 x 2^-e as an integer, cut into balanced base-256 digits from the low end
    long long S = __double2ll_rn(ldexp(x, 62 - e));
#pragma unroll
    for (int i = 7; i >= 1; --i) {
        const int d = (int)(signed char)(S & 255);
        S = (S - d) >> 8;
        w[i] = __bfloat16_as_ushort(__float2bfloat16_rn((float)d * __int_as_float((127 - 8 * i) << 23)));
    }
    w[0] = __bfloat16_as_ushort(__float2bfloat16_rn((float)(int)S));  // |S| <= 64
}

// Slices of the expansions, [box][K block][slice][32], and each box's scale
// 2^(e - 8) (FP32) or 2^(e - 6) (FP64); one warp per box.  A row with a
// non-finite entry gets the scale NaN, which its translations carry on.
template <typename T>
__global__ void k_slice_u(int64_t nb, int ns, int kblocks, const T *__restrict__ u, uint16_t *__restrict__ us,
                          T *__restrict__ rscale) {
    constexpr int NS = Slicing<T>::kSlices;
    const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (b >= nb) return;
    const int lane = threadIdx.x & 31;
    const T *row = u + (size_t)b * ns;
    T m = T(0);
    bool fin = true;
    for (int k = lane; k < ns; k += 32) {
        const T x = row[k] < T(0) ? -row[k] : row[k];
        fin = fin && isfinite(x);
        m = x > m ? x : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const T y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    fin = __all_sync(0xffffffffu, fin);
    const int e = (fin && m > T(0)) ? ceil_exp(m) : 0;
    uint16_t *out = us + (size_t)b * kblocks * NS * kKB;
    for (int kb = 0; kb < kblocks; ++kb) {
        const int k = kb * kKB + lane;
        uint16_t w[NS];
        slice_of((fin && k < ns) ? row[k] : T(0), e, w);
#pragma unroll
        for (int i = 0; i < NS; ++i) out[((size_t)kb * NS + i) * kKB + lane] = w[i];
    }
    if (lane == 0) rscale[b] = fin ? (T)ldexp(1.0, e - (sizeof(T) == 4 ? 8 : 6)) : (T)NAN;
}

// Per operator: the scale exponent; the scale handed to the kernel carries
// the unit of the drained sums (FP64: 2^-42 of the first accumulator's).
template <typename T>
__global__ void k_op_scale(int64_t elems, const T *__restrict__ ops, int *__restrict__ oexp, T *__restrict__ oscale) {
    __shared__ T red[32];
    const T *M = ops + (size_t)blockIdx.x * elems;
    T m = T(0);
    for (int64_t i = threadIdx.x; i < elems; i += blockDim.x) {
        const T x = M[i] < T(0) ? -M[i] : M[i];
        m = x > m ? x : m;
    }
    for (int o = 16; o > 0; o >>= 1) {
        const T y = __shfl_xor_sync(0xffffffffu, m, o);
        m = y > m ? y : m;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = red[w] > m ? red[w] : m;
        const int e = m > T(0) ? ceil_exp(m) : 0;
        oexp[blockIdx.x] = e;
        oscale[blockIdx.x] = (T)ldexp(1.0, e - (sizeof(T) == 4 ? 8 : 6 + 42));
    }
}

// Operator slices: ops [o][k][ld] (input k, output j), stored per (o, K block,
// column block) as the slices of the block's rows j, 32 elements each, in the
// 64-byte swizzled K-major form (16-byte chunk c of row j at chunk position
// c ^ ((j >> 1) & 3)): one linear copy lands ready for the tensor core.
// Column blocks of nt outputs, the last one shorter.
template <typename T>
__global__ void k_slice_ops(int64_t total, int ns, int ld, int np, int nt, int kblocks, const T *__restrict__ ops,
                            const int *__restrict__ oexp, uint16_t *__restrict__ bs) {
    constexpr int NS = Slicing<T>::kSlices;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int64_t blk = idx / ((int64_t)np * kKB);  // o * kblocks + kb
    const int rem = (int)(idx - blk * np * kKB);
    const int o = (int)(blk / kblocks), kb = (int)(blk - (int64_t)o * kblocks);
    const int j = rem / kKB, pos = rem % kKB;       // pos: swizzled position in the row
    const int k = kb * kKB + (((pos >> 3) ^ ((j >> 1) & 3)) << 3) + (pos & 7);
    uint16_t w[NS];
    slice_of((j < ld && k < ns) ? ops[((size_t)o * ns + k) * ld + j] : T(0), oexp[o], w);
    const int cb = j / nt, jj = j - cb * nt, rows = min(nt, np - cb * nt);
    uint16_t *out = bs + ((size_t)blk * np + (size_t)cb * nt) * NS * kKB + (size_t)jj * kKB + pos;
#pragma unroll
    for (int i = 0; i < NS; ++i) out[(size_t)i * rows * kKB] = w[i];
}

template <typename T>
struct ExArgs {
    const int32_t *targets;  // class-major target boxes
    const int4 *tiles;       // (class, begin, end, unused), 128 targets at most
    const int32_t *vdense;   // [nb][189]
    const int *slot_off;     // [8][189]
    const uint16_t *us;      // [nb][K blocks][slices][32]
    const T *rscale;         // [nb]
    const uint16_t *bs;      // operator slices
    const T *oscale;         // [316]
    T *d;                    // [nb][ns]
    double *dbar;            // [nb]: output column ns (the mean row), or nullptr
    T *part;                 // [slot split][target][ld] partial sums, or nullptr (one split)
    int z0, zn, part_add;    // this launch: slot ranges z0 .. z0 + gridDim.z - 1 of zn; 1: added to part
    int64_t n_targets;
    int ns, ld, np, nt, kblocks, chunk_blocks, nchunks, nstages, nbuf, accumulate;
    long long wait_polls;
    int *status;
};

// An accumulator value as an integer of units 2^-E.
template <int E>
__device__ __forceinline__ int unit_int(uint32_t bits) {
    return __float2int_rn(__uint_as_float(bits) * __int_as_float((127 + E) << 23));
}

// Byte offset of 16-byte chunk c of row r inside a 64-byte-swizzled tile.
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * kRowB + ((c ^ ((r >> 1) & 3)) << 4)); }

template <typename T>
__global__ void __launch_bounds__(ex_threads<T>(), 1) k_m2l_exact(ExArgs<T> a) {
    using SL = Slicing<T>;
    constexpr int NS = SL::kSlices, NG = SL::kGroups, kProd = SL::kProd;
    constexpr uint32_t kTileB = kTcRows * kRowB;  // one slice of the gathered rows
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int cb = blockIdx.y, c_first = cb * a.nt;
    const int nt = min(a.nt, a.np - c_first);  // output columns of this CTA (MMA N, a multiple of 16)
    const uint32_t stage_bytes = NS * (kTileB + (uint32_t)a.nt * kRowB);
    const uint32_t b_slice = (uint32_t)nt * kRowB;
    __shared__ __align__(8) uint64_t full_bar[8], empty_bar[8], done_bar, accfull_bar[2], accfree_bar[2];
    __shared__ uint32_t tmem_base_s;
    __shared__ int32_t tgt_s[kTcRows];
    __shared__ volatile int abort_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int4 tile = a.tiles[blockIdx.x];
    const int cls = tile.x;
    // this CTA's slots
    const int s_lo = kVSlots * (a.z0 + (int)blockIdx.z) / a.zn;
    const int s_hi = kVSlots * (a.z0 + (int)blockIdx.z + 1) / a.zn;
    const int NST = a.nstages, kblocks = a.kblocks;
    if (threadIdx.x < kTcRows) {
        const int i = tile.y + threadIdx.x;
        tgt_s[threadIdx.x] = (i < tile.z) ? a.targets[i] : -1;
    }
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < NST; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 32 * kProd + 1);  // producer cp.async arrivals + the bulk-copy leader
            mbar_init(smem_u32(&empty_bar[s]), 1);
        }
        mbar_init(smem_u32(&done_bar), 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&accfull_bar[b]), 1);
            mbar_init(smem_u32(&accfree_bar[b]), kDrain);  // lane 0 of each drain warp
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const uint32_t buf_cols = (uint32_t)(NG * nt);
    const uint32_t want_cols = buf_cols * a.nbuf;
    const uint32_t tmem_cols = want_cols <= 128 ? 128u : (want_cols <= 256 ? 256u : 512u);
    if (warp == kProd) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_s)),
                     "r"(tmem_cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        tc_fence_before();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;

    if (warp < kProd) {
        // ---------------- producers ----------------
        // Thread t copies 16-byte chunk (t & 3) of every slice of rows
        // (t >> 2) + 32 i; a row's slices of one K block are adjacent.
        constexpr int kRows = kTcRows / (8 * kProd);
        const int ch = threadIdx.x & 3, r0 = threadIdx.x >> 2;
        int32_t src[kRows], src_next[kRows];
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int32_t tg = tgt_s[r0 + 8 * kProd * i];
            src[i] = -1;
            src_next[i] = (tg >= 0) ? a.vdense[(size_t)tg * kVSlots + s_lo] : -1;
        }
        const bool leader = threadIdx.x == 0;
        int o_cur = 0, o_next = leader ? a.slot_off[cls * kVSlots + s_lo] : 0;
        int it = 0, last_it = -1;
        bool ok = true;
        for (int s = s_lo; s < s_hi && ok; ++s) {
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                src[i] = src_next[i];
                const int32_t tg = tgt_s[r0 + 8 * kProd * i];
                if (s + 1 < s_hi) src_next[i] = (tg >= 0) ? a.vdense[(size_t)tg * kVSlots + s + 1] : -1;
            }
            if (leader) {
                o_cur = o_next;
                if (s + 1 < s_hi) o_next = a.slot_off[cls * kVSlots + s + 1];
            }
            for (int kb = 0; kb < kblocks; ++kb, ++it) {
                const int stage = it % NST;
                if (!mbar_wait(smem_u32(&empty_bar[stage]), ((it / NST) & 1) ^ 1, &abort_s, a.wait_polls)) {
                    set_status(a.status, KIFMM_ERR_TIMEOUT);
                    abort_s = 1;
                    ok = false;
                    break;
                }
                const uint32_t sA = smem_u32(smem + (size_t)stage * stage_bytes), sB = sA + NS * kTileB;
                const uint32_t fb = smem_u32(&full_bar[stage]);
                if (leader) {
                    const size_t boff = (((size_t)o_cur * kblocks + kb) * a.np + c_first) * (size_t)(NS * kKB);
                    mbar_arrive_expect_tx(fb, NS * b_slice);
                    bulk_g2s(sB, a.bs + boff, NS * b_slice, fb);
                    last_it = it;
                }
#pragma unroll
                for (int i = 0; i < kRows; ++i) {
                    const int r = r0 + 8 * kProd * i;
                    const uint16_t *row =
                        a.us + ((size_t)(src[i] >= 0 ? src[i] : 0) * kblocks + kb) * (size_t)(NS * kKB) + 8 * ch;
                    const uint32_t nbytes = (src[i] >= 0) ? 16u : 0u, dst = sA + swz(r, ch);
#pragma unroll
                    for (int q = 0; q < NS; ++q) cp_async16(dst + q * kTileB, row + q * kKB, nbytes);
                }
                cp_async_arrive_noinc(fb);
            }
        }
        cp_async_wait_all();
        if (leader) wait_bulk_copies(full_bar, NST, last_it);
    } else if (warp == kProd) {
        // ---------------- MMA issuer ----------------
        // One accumulation per (slot, K chunk), in accumulator set w % nbuf.
        if (lane == 0) {
            const uint32_t id = idesc_f16(nt, SL::kFmt);  // (FP32)
            const int wide = min(NS, 256 / nt);             // (FP64) operator slices per MMA, 256 columns at most
            int it = 0, w = 0;
            for (int s = s_lo; s < s_hi && !abort_s; ++s) {
                for (int c = 0; c < a.nchunks && !abort_s; ++c, ++w) {
                    const int buf = w % a.nbuf;
                    if (w >= a.nbuf &&
                        !mbar_wait(smem_u32(&accfree_bar[buf]), ((w / a.nbuf) - 1) & 1, &abort_s, a.wait_polls)) {
                        set_status(a.status, KIFMM_ERR_TIMEOUT);
                        abort_s = 1;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t acc0 = tmem + buf * buf_cols;
                    const int kb1 = min(kblocks, (c + 1) * a.chunk_blocks);
                    for (int kb = c * a.chunk_blocks; kb < kb1; ++kb, ++it) {
                        const int stage = it % NST;
                        if (!mbar_wait(smem_u32(&full_bar[stage]), (it / NST) & 1, &abort_s, a.wait_polls)) {
                            set_status(a.status, KIFMM_ERR_TIMEOUT);
                            abort_s = 1;
                            break;
                        }
                        fence_proxy_async();
                        tc_fence_after();
                        const uint32_t sA = smem_u32(smem + (size_t)stage * stage_bytes);
                        // descriptors differ in the address field only
                        const uint64_t dA0 = sdesc_sw64(sA), dB0 = sdesc_sw64(sA + NS * kTileB);
                        if constexpr (sizeof(T) == 8) {
                            // rows' slice i with operator slices j .. j + m - 1,
                            // into the accumulators i + j .. i + j + m - 1
                            for (int kk = 0; kk < 2; ++kk) {
                                const uint32_t on = (kb > c * a.chunk_blocks || kk > 0) ? 1u : 0u;
                                for (int i = 0; i < NS; ++i) {
                                    const uint64_t dA = dA0 + (uint64_t)((i * kTileB + 32 * kk) >> 4);
                                    for (int j = 0; j < NS - i; j += wide) {
                                        const int m = min(wide, NS - i - j);
                                        const uint64_t dB = dB0 + (uint64_t)((j * b_slice + 32 * kk) >> 4);
                                        mma_f16(acc0 + (uint32_t)((i + j) * nt), dA, dB, idesc_f16(m * nt, SL::kFmt),
                                                i == 0 ? on : 1u);  // d_0 meets every accumulator first
                                    }
                                }
                            }
                        } else {
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk) {
                                const uint32_t on = (kb > c * a.chunk_blocks || kk > 0) ? 1u : 0u;
                                const uint64_t dA = dA0 + (uint64_t)(2 * kk), dB = dB0 + (uint64_t)(2 * kk);
                                const uint32_t a_step = kTileB >> 4, b_step = b_slice >> 4;
                                const uint32_t acc1 = acc0 + (uint32_t)nt;
                                mma_f16_fill(acc0, dA, dB, id, on);                           // h h
                                mma_f16_use(acc1, dA, dB + b_step, id, on);                   // h l
                                mma_f16_lastuse(acc1, dA, dB + 2 * b_step, id, 1u);           // h l2
                                mma_f16_fill(acc1, dA + a_step, dB, id, 1u);                  // l h
                                mma_f16_lastuse(acc1, dA + a_step, dB + b_step, id, 1u);      // l l
                                mma_f16(acc1, dA + 2 * a_step, dB, id, 1u);                   // l2 h
                            }
                        }
                        mma_commit(smem_u32(&empty_bar[stage]));
                    }
                    if (abort_s) break;
                    mma_commit(smem_u32(&accfull_bar[buf]));
                }
            }
            mma_commit(smem_u32(&done_bar));
        }
        __syncwarp();
    } else {
        // ---------------- drain warps ----------------
        // Warp w may read TMEM lanes 32 (w % 4) .. + 31; two warps share each
        // quadrant, taking the 16-column groups h, h + 2, h + 4, ...
        const int dw = warp - kProd - 1;
        const int q = warp & 3, h = dw >> 2;
        const uint32_t lane_off = (uint32_t)(q * 32) << 16;
        constexpr int kMine = SL::kCols / 32;  // 16-column groups per warp, at most
        const int row = q * 32 + lane;
        const int32_t tb = tgt_s[row];
        T acc[kMine][16];
#pragma unroll
        for (int c = 0; c < kMine; ++c)
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[c][j] = T(0);
        // the row's source two slots ahead, its scale one slot ahead
        auto source = [&](int s) -> int32_t {
            return (tb >= 0 && s < s_hi) ? a.vdense[(size_t)tb * kVSlots + s] : -1;
        };
        auto scale = [&](int32_t src, int s) -> T {
            return src >= 0 ? a.rscale[src] * a.oscale[a.slot_off[cls * kVSlots + s]] : T(0);
        };
        int32_t src1 = source(s_lo);
        T sc_next = scale(src1, s_lo);
        src1 = source(s_lo + 1);
        bool ok = true;
        int w = 0;
        for (int s = s_lo; s < s_hi && ok; ++s) {
            const T sc = sc_next;
            sc_next = scale(src1, s + 1);
            src1 = source(s + 2);
            for (int c = 0; c < a.nchunks; ++c, ++w) {
                const int buf = w % a.nbuf;
                ok = mbar_wait(smem_u32(&accfull_bar[buf]), (w / a.nbuf) & 1, &abort_s, a.wait_polls);
                ok = __all_sync(0xffffffffu, ok);  // warp-uniform: tcgen05.ld is .sync.aligned
                if (!ok) {
                    set_status(a.status, KIFMM_ERR_TIMEOUT);
                    abort_s = 1;
                    break;
                }
                tc_fence_after();
                const uint32_t base = tmem + lane_off + buf * buf_cols;
#pragma unroll
                for (int g = 0; g < kMine; ++g) {
                    const int col = 16 * (h + 2 * g);
                    if (col >= nt) continue;  // uniform
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        const uint32_t at = base + (uint32_t)(col + 8 * half);
                        if constexpr (sizeof(T) == 4) {
                            uint32_t v[16];
#pragma unroll
                            for (int e = 0; e < 2; ++e) tmem_ld8_nowait(at + (uint32_t)(e * nt), v + 8 * e);
                            tmem_wait_ld(v);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                const float p = __uint_as_float(v[j]) + __uint_as_float(v[8 + j]);
                                acc[g][8 * half + j] = fmaf(p, sc, acc[g][8 * half + j]);
                            }
                        } else {
                            // group e is an integer times 2^-8e: the sum in units
                            // of 2^-42, three batches of groups
                            long long sum[8];
                            {
                                uint32_t v[24];
#pragma unroll
                                for (int e = 0; e < 3; ++e) tmem_ld8_nowait(at + (uint32_t)(e * nt), v + 8 * e);
                                tmem_wait_ld(v);
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    sum[j] = ((long long)unit_int<0>(v[j]) * 65536 +
                                              (unit_int<8>(v[8 + j]) * 256LL + unit_int<16>(v[16 + j])))
                                             * (1LL << 26);
                            }
                            {
                                uint32_t v[24];
#pragma unroll
                                for (int e = 0; e < 3; ++e) tmem_ld8_nowait(at + (uint32_t)((e + 3) * nt), v + 8 * e);
                                tmem_wait_ld(v);
#pragma unroll
                                for (int j = 0; j < 8; ++j)
                                    sum[j] += (long long)unit_int<24>(v[j]) * (1 << 18) +
                                              (long long)unit_int<32>(v[8 + j]) * 1024 +
                                              (long long)unit_int<40>(v[16 + j]) * 4;
                            }
                            uint32_t v[16];
#pragma unroll
                            for (int e = 0; e < 2; ++e) tmem_ld8_nowait(at + (uint32_t)((e + 6) * nt), v + 8 * e);
                            tmem_wait_ld(v);
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                sum[j] += unit_int<42>(
                                    __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(v[8 + j])));
                                acc[g][8 * half + j] = fma((double)sum[j], sc, acc[g][8 * half + j]);
                            }
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&accfree_bar[buf]));
            }
        }
        if (tb >= 0) {  // (timed out: NaN, so that no caller takes the row for a result)
            const bool valid = ok && !abort_s;
            T *out = a.part ? a.part + ((size_t)blockIdx.z * a.n_targets + tile.y + row) * a.ld
                            : a.d + (size_t)tb * a.ns;
#pragma unroll
            for (int g = 0; g < kMine; ++g) {
                const int col = 16 * (h + 2 * g);
                if (col >= nt) continue;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const int jc = c_first + col + j;
                    const T v = valid ? acc[g][j] : (T)NAN;
                    if (a.part) {
                        if (jc < a.ld) out[jc] = a.part_add ? out[jc] + v : v;
                    } else if (jc < a.ns) {
                        out[jc] = a.accumulate ? out[jc] + v : v;
                    } else if (jc == a.ns && a.dbar) {
                        a.dbar[tb] = (a.accumulate ? a.dbar[tb] : 0.0) + (double)v;
                    }
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kProd) {
        if (abort_s) wait_mmas(smem_u32(&done_bar));  // none may touch the memory given back below
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
    }
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }

}  // namespace

// out = the in-order sum of the slot splits' partial products.
template <typename T>
__global__ void k_m2l_part_sum(const int32_t *__restrict__ targets, int64_t n_t, int nsplit, int ns, int ld,
                               const T *__restrict__ part, T *__restrict__ out, int accumulate,
                               double *__restrict__ dbar) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_t * ld) return;
    const int64_t i = idx / ld;
    const int j = (int)(idx - i * ld);
    T v = T(0);
    for (int z = 0; z < nsplit; ++z) v += part[(size_t)z * n_t * ld + idx];
    const int32_t t = targets[i];
    if (j < ns) {
        T *o = out + (size_t)t * ns + j;
        *o = accumulate ? *o + v : v;
    } else if (dbar) {
        dbar[t] = (accumulate ? dbar[t] : 0.0) + (double)v;
    }
}
template <typename T>
static void part_sum(const Plan &P, int64_t n_t, int nsplit, int ns, int ld, const T *part, T *out, int accumulate,
                     double *dbar, cudaStream_t s) {
    ++g_launches, k_m2l_part_sum<T><<<(unsigned)((n_t * ld + 255) / 256), 256, 0, s>>>(
                      P.m2l_targets, n_t, nsplit, ns, ld, part, out, accumulate, dbar);
}

// A rule for how many CTAs share a tile's 189 slots when `units` (tiles x
// column blocks) CTAs would run at one per SM: the split z that minimises the
// waves' length ceil(units z / SMs) (189 / z + 4), a CTA's set-up, pipeline
// fill and partial store costing about four slots (three without the partial
// store, z = 1).  Few tiles (small trees)
// would otherwise leave most SMs idle for 189 slots in a row.
int m2l_slot_split(int64_t units, int num_sms) {
    if (units <= 0) return 1;
    int best = 1;
    double least = 1e30;
    for (int z = 1; z <= 63 && (z == 1 || units * z <= 8 * (int64_t)num_sms); ++z) {
        const double waves = (double)((units * z + num_sms - 1) / num_sms);
        const double t = waves * ((kVSlots + z - 1) / z + (z == 1 ? 3.0 : 4.0));
        if (t < 0.98 * least) {
            least = t;
            best = z;
        }
    }
    return best;
}

// Operator slices of one direction (forward or adjoint).
struct ExOps {
    uint16_t *bs = nullptr;
    void *oscale = nullptr;
};
struct ExState {
    int ns = 0, ld[2] = {0, 0}, np[2] = {0, 0}, nt[2] = {0, 0}, ncb[2] = {0, 0};
    int kblocks = 0, nchunks = 0, chunk_blocks = 0;
    ExOps ops[2];  // forward, adjoint
    uint16_t *us = nullptr;
    void *rscale = nullptr;
    int64_t u_cap = 0;
};

static ExState &ex_state(Plan &P) {
    if (!P.m2l_ex) P.m2l_ex = new ExState();
    return *(ExState *)P.m2l_ex;
}

void m2l_exact_release(Plan &P) {
    delete (ExState *)P.m2l_ex;
    P.m2l_ex = nullptr;
}

template <typename T>
static int ex_stages(int nt) {
    const size_t stage = (size_t)Slicing<T>::kSlices * (kTcRows * kRowB + (size_t)nt * kRowB);
    return (int)std::min<size_t>(8, (227 * 1024 - 4096) / stage);
}

// Plan time: slices of `ops` ([316][n_s][ld], device, compute type) for one
// direction (0: forward, 1: adjoint).
template <typename T>
static cudaError_t ex_setup(Plan &P, int dir, const T *ops, int ld) {
    using SL = Slicing<T>;
    ExState &S = ex_state(P);
    S.ns = P.ns;
    S.kblocks = (P.ns + kKB - 1) / kKB;
    S.nchunks = (S.kblocks + SL::kChunkBlocks - 1) / SL::kChunkBlocks;
    S.chunk_blocks = (S.kblocks + S.nchunks - 1) / S.nchunks;
    S.ld[dir] = ld;
    S.np[dir] = round_up(ld, 16);
    S.ncb[dir] = (S.np[dir] + SL::kCols - 1) / SL::kCols;
    S.nt[dir] = round_up((S.np[dir] + S.ncb[dir] - 1) / S.ncb[dir], 16);
    const size_t total = (size_t)kNumM2L * S.np[dir] * S.kblocks * kKB;
    int *oexp = nullptr;
    KIFMM_CUDA_TRY(cudaMalloc(&oexp, sizeof(int) * kNumM2L));
    KIFMM_CUDA_TRY(plan_alloc(P, (void **)&S.ops[dir].bs, sizeof(uint16_t) * SL::kSlices * total));
    KIFMM_CUDA_TRY(plan_alloc(P, &S.ops[dir].oscale, sizeof(T) * kNumM2L));
    ++g_launches, k_op_scale<T><<<kNumM2L, 256>>>((int64_t)P.ns * ld, ops, oexp, (T *)S.ops[dir].oscale);
    ++g_launches, k_slice_ops<T><<<(unsigned)((total + 255) / 256), 256>>>((int64_t)total, P.ns, ld, S.np[dir],
                                                                          S.nt[dir], S.kblocks, ops, oexp,
                                                                          S.ops[dir].bs);
    // the largest any column-block width takes
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_m2l_exact<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 2048));
    KIFMM_CUDA_TRY(cudaDeviceSynchronize());
    return cudaFree(oexp);
}

cudaError_t m2l_exact_setup(Plan &P, int dir, const void *ops, int ld) {
    return P.f64 ? ex_setup<double>(P, dir, (const double *)ops, ld) : ex_setup<float>(P, dir, (const float *)ops, ld);
}

// Slot ranges of one direction; they fix the order of the additions, so they
// depend on the tree alone, not on the memory there is.
static int ex_split(const Plan &P, const ExState &S, int dir) {
    return m2l_slot_split((int64_t)m2l_tiles_128(P) * S.ncb[dir], P.num_sms);
}
static size_t ex_part_bytes(const Plan &P, const ExState &S, int dir, int z) {
    return (P.f64 ? sizeof(double) : sizeof(float)) * z * (size_t)P.m2l_class_start[8] * S.ld[dir];
}

// After set_sources: room for the sliced expansions.
cudaError_t m2l_exact_prepare(Plan &P) {
    if (!P.m2l_ex) return cudaSuccess;
    ExState &S = ex_state(P);
    const size_t esz = P.f64 ? sizeof(double) : sizeof(float);
    const int NS = P.f64 ? Slicing<double>::kSlices : Slicing<float>::kSlices;
    if (P.nb > S.u_cap) {
        const int64_t cap = P.list_cap;
        KIFMM_CUDA_TRY(plan_replace(P, &S.u_cap, cap,
                                    {{(void **)&S.us, sizeof(uint16_t) * cap * S.kblocks * NS * kKB},
                                     {&S.rscale, esz * cap}}));
    }
    return cudaSuccess;
}

// The slot splits' partial sums: at most 8 x 152 CTAs' accumulators (some
// 100 MB), the adjoint's and the forward's never live at once.
size_t m2l_exact_part_bytes(Plan &P) {
    if (!P.m2l_ex) return 0;
    const ExState &S = ex_state(P);
    size_t need = 0;
    for (int dir = 0; dir < 2; ++dir) {
        const int z = S.ops[dir].bs ? ex_split(P, S, dir) : 1;
        if (z > 1) need = std::max(need, ex_part_bytes(P, S, dir, z));
    }
    return need;
}

template <typename T>
static cudaError_t ex_run(Plan &P, int dir, const T *u, T *d, int accumulate, double *dbar, cudaStream_t s) {
    using SL = Slicing<T>;
    ExState &S = ex_state(P);
    const int ntiles = m2l_tiles_128(P);
    if (ntiles == 0) return cudaSuccess;  // no V-list targets
    ++g_launches, k_slice_u<T><<<(unsigned)((P.nb + 7) / 8), 256, 0, s>>>(P.nb, P.ns, S.kblocks, u, S.us,
                                                                         (T *)S.rscale);
    ExArgs<T> a;
    a.targets = P.m2l_targets;
    a.tiles = m2l_tiles_dev(P);
    a.vdense = P.vdense;
    a.slot_off = P.slot_off;
    a.us = S.us;
    a.rscale = (const T *)S.rscale;
    a.bs = S.ops[dir].bs;
    a.oscale = (const T *)S.ops[dir].oscale;
    a.d = d;
    a.dbar = dbar;
    a.n_targets = P.m2l_class_start[8];
    a.ns = P.ns;
    a.ld = S.ld[dir];
    a.np = S.np[dir];
    a.nt = S.nt[dir];
    a.kblocks = S.kblocks;
    a.chunk_blocks = S.chunk_blocks;
    a.nchunks = S.nchunks;
    a.nstages = ex_stages<T>(a.nt);
    a.nbuf = (2 * SL::kGroups * a.nt <= 512) ? 2 : 1;
    a.accumulate = accumulate;
    a.wait_polls = P.m2l_wait_polls > 0 ? P.m2l_wait_polls : kWaitIters;
    a.status = P.status;
    const int z = ex_split(P, S, dir);
    const size_t smem = (size_t)a.nstages * SL::kSlices * (kTcRows + a.nt) * kRowB + 1024;
    auto launch = [&](int z0, int nz) {
        a.z0 = z0;
        a.part_add = nz == 1 && z0 > 0;
        ++g_launches, k_m2l_exact<T><<<dim3((unsigned)ntiles, (unsigned)S.ncb[dir], (unsigned)nz), ex_threads<T>(),
                                     smem, s>>>(a);
    };
    a.zn = z;
    if (z == 1 || ex_part_bytes(P, S, dir, z) <= P.m2l_part_bytes) {
        a.part = z > 1 ? (T *)P.m2l_part : nullptr;
        launch(0, z);
        if (z > 1) part_sum<T>(P, a.n_targets, z, a.ns, a.ld, a.part, d, accumulate, dbar, s);
    } else {  // no room: the ranges one after the other into one set of rows, the same additions
        a.part = (T *)P.tmp_chk;
        for (int k = 0; k < z; ++k) launch(k, 1);
        part_sum<T>(P, a.n_targets, 1, a.ns, a.ld, a.part, d, accumulate, dbar, s);
    }
    return cudaGetLastError();
}

// dir 0: d (=|+=) M2L u over the V lists (with dbar, the mean rows); dir 1:
// the transposed operators (V lists are symmetric).
cudaError_t m2l_exact(Plan &P, int dir, const void *u, void *d, int accumulate, double *dbar, cudaStream_t s) {
    return P.f64 ? ex_run<double>(P, dir, (const double *)u, (double *)d, accumulate, dbar, s)
                 : ex_run<float>(P, dir, (const float *)u, (float *)d, accumulate, dbar, s);
}

}  // namespace kifmm
