// KIFMM evaluation passes (Sec. 2.2): upward pass (P2M, M2M), M2L over the
// V lists, P2L over the X lists, downward pass (L2L), leaf evaluation (L2P,
// M2P over the W lists) and the near field (P2P over the U lists).
//
// Units: positions are root-normalised (root cube side 1) and every box
// stores potentials of the kernel 1/r on its check surfaces:
//   u(b) on UC = c_b + 2.95 h_b S  (upward), d(b) on DC = c_b + 1.05 h_b S.
// The 1/(4 pi), the coefficient and the 1/side, 1/side^2 of physical units
// are applied once in the final scatter.
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "gemm_rows.cuh"
#include "internal.h"

namespace kifmm {

cudaError_t m2l_tensor(Plan &P, cudaStream_t s);  // m2l_tc.cu

namespace {

constexpr int kLeafThreads = 128;
constexpr int kMaxNs = 6 * 9 * 9 + 2;  // n_s at the largest surface order, p = 10

template <typename T>
__device__ __forceinline__ T box_half(int level) {
    return (T)ldexp(1.0, -(level + 1));
}
template <typename T>
__device__ __forceinline__ T box_center(int c, int level) {
    return (T)(ldexp((double)(2 * c + 1), -(level + 1)));
}

// Offset of image s (13: the cell itself) in root units: the periodic cell is
// the root box, of side 1.
template <typename T>
__device__ __forceinline__ void image_offset(int s, T &x, T &y, T &z) {
    x = (T)(s / 9 - 1);
    y = (T)((s / 3) % 3 - 1);
    z = (T)(s % 3 - 1);
}


template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T &s, T &e) {
    s = a + b;
    const T bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// P2M: u(b)_j = (1/h) sum_i q_i / |2.95 S_j - (x_i - c_b)/h|.  One block
// per leaf with a thread per check point (blockDim = n_s rounded up to a
// warp); particles staged through shared memory in chunks of blockDim.  The
// check surface lies outside the leaf, so no distance is zero.
template <typename T>
__global__ void k_p2m(const int32_t *__restrict__ leaves, const int32_t *__restrict__ lvl,
                      const int32_t *__restrict__ first, const int32_t *__restrict__ cnt,
                      const typename Vec4<T>::type *__restrict__ pts, const T *__restrict__ surf, int ns,
                      T *__restrict__ u, const T *__restrict__ wts = nullptr, int adj = 0,
                      const T *__restrict__ dip = nullptr) {
    // Adjoint with dip ([N][3] sorted, root units): each particle also carries
    // the dipole dL/dgrad, whose field at the surface point y is
    // g . (y - x) / |y - x|^3 (the transpose of the gradient evaluation).
    extern __shared__ __align__(16) unsigned char p2m_sm[];
    T *sx = (T *)p2m_sm, *sy = sx + blockDim.x, *sz = sy + blockDim.x, *sq = sz + blockDim.x;
    T *gx = sq + blockDim.x, *gy = gx + blockDim.x, *gz = gy + blockDim.x;
    const int b = leaves[blockIdx.x];
    const T h = box_half<T>(lvl[b]), hinv = T(1) / h;
    const int n = cnt[b], f = first[b];
    const T a = (T)kAlphaOuter;
    for (int j0 = 0; j0 < ns; j0 += blockDim.x) {
        const int j = j0 + threadIdx.x;
        T px = 0, py = 0, pz = 0;
        if (j < ns) {
            px = a * surf[3 * j];
            py = a * surf[3 * j + 1];
            pz = a * surf[3 * j + 2];
        }
        T acc = 0;
        for (int c0 = 0; c0 < n; c0 += blockDim.x) {
            __syncthreads();
            if (c0 + threadIdx.x < n) {
                const auto v = pts[f + c0 + threadIdx.x];
                sx[threadIdx.x] = v.x * hinv;
                sy[threadIdx.x] = v.y * hinv;
                sz[threadIdx.x] = v.z * hinv;
                sq[threadIdx.x] = wts ? wts[f + c0 + threadIdx.x] : v.w;
                if (dip) {  // in box units the dipole term carries 1/h
                    const size_t k = 3 * (size_t)(f + c0 + threadIdx.x);
                    gx[threadIdx.x] = dip[k] * hinv;
                    gy[threadIdx.x] = dip[k + 1] * hinv;
                    gz[threadIdx.x] = dip[k + 2] * hinv;
                }
            }
            __syncthreads();
            const int m = min((int)blockDim.x, n - c0);
            if (dip) {
                for (int i = 0; i < m; ++i) {
                    const T rx = px - sx[i], ry = py - sy[i], rz = pz - sz[i];
                    const T ri = rsqrt_t<T>(rx * rx + ry * ry + rz * rz);
                    acc += sq[i] * ri + (gx[i] * rx + gy[i] * ry + gz[i] * rz) * (ri * ri * ri);
                }
            } else {
#pragma unroll 4
                for (int i = 0; i < m; ++i) {
                    const T rx = px - sx[i], ry = py - sy[i], rz = pz - sz[i];
                    acc += sq[i] * rsqrt_t<T>(rx * rx + ry * ry + rz * rz);
                }
            }
        }
        // forward: u = sum q / |UC - x| (1/h from the unit surface); adjoint of
        // L2P: h * sum w / |DE - x| with the same unit geometry
        if (j < ns) u[(size_t)b * ns + j] = adj ? acc : acc * hinv;
    }
}


// P2M, FP32 forward form: kP2mLeaves leaves per block (a leaf's ~n_s x 30
// kernel evaluations are too little work for a block of their own) and the
// particle loop on packed f32x2 arithmetic, two particles per instruction
// (the chunk's odd tail padded with a null particle: weight 0, far away).
constexpr int kP2mLeaves = 4;
__global__ void k_p2m_f32(const int32_t *__restrict__ leaves, int64_t n_leaves, const int32_t *__restrict__ lvl,
                          const int32_t *__restrict__ first, const int32_t *__restrict__ cnt,
                          const float4 *__restrict__ pts, const float *__restrict__ surf, int ns,
                          float *__restrict__ u) {
    extern __shared__ __align__(16) unsigned char p2m_sm[];
    const int nt = blockDim.x;  // a multiple of 32
    float *sx = (float *)p2m_sm, *sy = sx + nt, *sz = sy + nt, *sq = sz + nt;
    const float a = (float)kAlphaOuter;
    const int64_t l0 = (int64_t)blockIdx.x * kP2mLeaves, l1 = min(n_leaves, l0 + kP2mLeaves);
    for (int64_t li = l0; li < l1; ++li) {
        const int b = leaves[li];
        const float hinv = 1.f / box_half<float>(lvl[b]);
        const int n = cnt[b], f = first[b];
        for (int j0 = 0; j0 < ns; j0 += nt) {
            const int j = j0 + threadIdx.x;
            float px = 0.f, py = 0.f, pz = 0.f;
            if (j < ns) {
                px = a * surf[3 * j];
                py = a * surf[3 * j + 1];
                pz = a * surf[3 * j + 2];
            }
            const float2 npx = make_float2(-px, -px), npy = make_float2(-py, -py), npz = make_float2(-pz, -pz);
            float2 acc = make_float2(0.f, 0.f);
            for (int c0 = 0; c0 < n; c0 += nt) {
                __syncthreads();
                const int m = min(nt, n - c0);
                if ((int)threadIdx.x < m) {
                    const float4 v = pts[f + c0 + threadIdx.x];
                    sx[threadIdx.x] = v.x * hinv;
                    sy[threadIdx.x] = v.y * hinv;
                    sz[threadIdx.x] = v.z * hinv;
                    sq[threadIdx.x] = v.w;
                } else if ((int)threadIdx.x == m) {  // m < nt: pad the odd tail
                    sx[m] = sy[m] = sz[m] = 1e4f;
                    sq[m] = 0.f;
                }
                __syncthreads();
#pragma unroll 4
                for (int i = 0; i < m; i += 2) {
                    const float2 rx = __fadd2_rn(*reinterpret_cast<const float2 *>(sx + i), npx);
                    const float2 ry = __fadd2_rn(*reinterpret_cast<const float2 *>(sy + i), npy);
                    const float2 rz = __fadd2_rn(*reinterpret_cast<const float2 *>(sz + i), npz);
                    float2 r2 = __fmul2_rn(rx, rx);
                    r2 = __ffma2_rn(ry, ry, r2);
                    r2 = __ffma2_rn(rz, rz, r2);
                    const float2 ri = make_float2(rsqrt_t<float>(r2.x), rsqrt_t<float>(r2.y));
                    acc = __ffma2_rn(*reinterpret_cast<const float2 *>(sq + i), ri, acc);
                }
            }
            if (j < ns) u[(size_t)b * ns + j] = (acc.x + acc.y) * hinv;
        }
    }
}

// P2L: d(b)_j += (1/h_b) sum_{a in X(b)} sum_i q_i / |1.05 S_j - (x_i - c_b)/h_b|
// One block per box with an X list (the X lists are the transposed W lists, so
// these are the boxes of part_list[2]), up to 26 leaves of it: a block's length
// is the launch's.  A thread per check point (tpg of them:
// n_s rounded up to a warp; with 128 threads, two rounds over the sources, the
// second for the last 24 points of n_s = 152).  FP64, bound by the FP64 unit,
// also cuts the sources into blockDim / tpg interleaved groups, whose sums are
// added in group order.  60k Plummer, FP64: 1.18 -> 0.44 ms.
template <typename T>
__global__ void __launch_bounds__(1024, 1)
    k_p2l(int tpg, const int32_t *__restrict__ boxes, const int32_t *__restrict__ nx, const int32_t *__restrict__ xdense, const int32_t *__restrict__ lvl,
          const int32_t *__restrict__ cx, const int32_t *__restrict__ cy, const int32_t *__restrict__ cz,
          const int32_t *__restrict__ first, const int32_t *__restrict__ cnt,
          const typename Vec4<T>::type *__restrict__ pts, const T *__restrict__ surf, int ns, T *__restrict__ d,
          const T *__restrict__ wts = nullptr, int adj = 0, double *__restrict__ dbar = nullptr,
          const T *__restrict__ dip = nullptr, const int8_t *__restrict__ x_sh = nullptr) {
    // With dbar (FP32-based modes) the mean of this box's contribution goes
    // to dbar and only the mean-free remainder to d.  With dip (adjoint of
    // M2P under a loss on the gradient) every particle also carries a dipole.
    __shared__ T sx[kLeafThreads], sy[kLeafThreads], sz[kLeafThreads], sq[kLeafThreads];
    __shared__ T gx[kLeafThreads], gy[kLeafThreads], gz[kLeafThreads];
    __shared__ T cv[kMaxNs];
    __shared__ double red[32];
    const int b = boxes[blockIdx.x];
    const int lb = lvl[b];
    const T hb = box_half<T>(lb), hinv = T(1) / hb;
    const T cbx = box_center<T>(cx[b], lb), cby = box_center<T>(cy[b], lb), cbz = box_center<T>(cz[b], lb);
    const T al = (T)kAlphaInner;
    const int ng = blockDim.x / tpg, grp = threadIdx.x / tpg, j = threadIdx.x - grp * tpg;
    T px = 0, py = 0, pz = 0;
    if (j < ns) {
        px = al * surf[3 * j];
        py = al * surf[3 * j + 1];
        pz = al * surf[3 * j + 2];
    }
    T acc = 0;
    for (int e = 0; e < nx[b]; ++e) {
        const int a = xdense[(size_t)b * kMaxCoarse + e];
        const int la = lvl[a];
        T ox = box_center<T>(cx[a], la) - cbx, oy = box_center<T>(cy[a], la) - cby,
          oz = box_center<T>(cz[a], la) - cbz;
        if (x_sh) {  // the source leaf's image (periodic cell)
            T ix, iy, iz;
            image_offset<T>(x_sh[(size_t)b * kMaxCoarse + e], ix, iy, iz);
            ox += ix, oy += iy, oz += iz;
        }
        const int n = cnt[a], f = first[a];
        for (int c0 = 0; c0 < n; c0 += kLeafThreads) {
            __syncthreads();
            const int m = min(kLeafThreads, n - c0);
            for (int i = threadIdx.x; i < m; i += blockDim.x) {
                const auto v = pts[f + c0 + i];
                sx[i] = (ox + v.x) * hinv;
                sy[i] = (oy + v.y) * hinv;
                sz[i] = (oz + v.z) * hinv;
                sq[i] = wts ? wts[f + c0 + i] : v.w;
                if (dip) {
                    const size_t k = 3 * (size_t)(f + c0 + i);
                    gx[i] = dip[k] * hinv;
                    gy[i] = dip[k + 1] * hinv;
                    gz[i] = dip[k + 2] * hinv;
                }
            }
            __syncthreads();
            if (dip) {
                for (int i = grp; i < m; i += ng) {
                    const T rx = px - sx[i], ry = py - sy[i], rz = pz - sz[i];
                    const T ri = rsqrt_t<T>(rx * rx + ry * ry + rz * rz);
                    acc += sq[i] * ri + (gx[i] * rx + gy[i] * ry + gz[i] * rz) * (ri * ri * ri);
                }
            } else {
#pragma unroll 4
                for (int i = grp; i < m; i += ng) acc += sq[i] * lap_pot<T>(px - sx[i], py - sy[i], pz - sz[i]);
            }
        }
    }
    for (int g = 0; g < ng; ++g) {  // the groups' sums, in group order
        if (grp == g && j < ns) cv[j] = g == 0 ? acc : cv[j] + acc;
        __syncthreads();
    }
    if (!adj) {
        if (grp == 0 && j < ns) cv[j] *= hinv;
        __syncthreads();
    }
    if (!dbar) {
        if (grp == 0 && j < ns) d[(size_t)b * ns + j] += cv[j];
        return;
    }
    // (the mean's sum over 128 lanes, four warps, whatever the block)
    if (threadIdx.x < kLeafThreads) {
        double sum = 0.0;
        for (int k = threadIdx.x; k < ns; k += kLeafThreads) sum += (double)cv[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
    }
    __syncthreads();
    double tot = 0.0;
    for (int w = 0; w < min((int)blockDim.x, kLeafThreads) / 32; ++w) tot += red[w];  // (p <= 4: two warps)
    const double mean = tot / ns;
    for (int k = threadIdx.x; k < ns; k += blockDim.x) d[(size_t)b * ns + k] += (T)((double)cv[k] - mean);
    if (threadIdx.x == 0) dbar[b] += mean;
}

// ---------------------------------------------------------------------------
// Gathered row products of many rows in FP64 (FP32 and few rows:
// gemm_rows.cuh), out[t] (=|+=) Op in[src(t)]: a block owns NTY RT rows of one
// class and 32 RC outputs; thread (tx, ty) keeps rows RT ty .. RT ty + RT - 1
// by outputs tx + 32 c.  Operators [k][ldp]; k advances in chunks of 16 through shared
// memory with the next chunk prefetched into registers.  Bound by the FP64
// unit (two lanes per clock and SM).
// ---------------------------------------------------------------------------
constexpr int kGK = 16;

__global__ void __launch_bounds__(256) k_rows_f64(RowMap<double> g, const int32_t *__restrict__ targets,
                                                  ClassRanges cr, int n, int ldp, const double *__restrict__ in,
                                                  double *out, int accumulate) {
    constexpr int NTY = 8, RT = 8, RC = 5;
    constexpr int TT = NTY * RT, TJ = 32 * RC, NT = 32 * NTY;
    __shared__ __align__(16) double Us[kGK][TT];
    __shared__ __align__(16) double Ms[kGK][TJ];
    __shared__ int32_t tgt[TT];
    __shared__ int32_t src[TT];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int cls = blockIdx.y;
    const int j0 = (int)blockIdx.z * TJ;  // output columns [j0, j0 + TJ)
    int64_t t_begin = 0, t_end = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
        if (c == cls) t_begin = cr.b[c], t_end = cr.b[c + 1];
    const int64_t t0 = t_begin + (int64_t)blockIdx.x * TT;
    if (t0 >= t_end) return;  // uniform for the block
    if (threadIdx.x < TT) {
        const int32_t t = (t0 + threadIdx.x < t_end) ? targets[t0 + threadIdx.x] : -1;
        tgt[threadIdx.x] = t;
        src[threadIdx.x] = t >= 0 ? g.src(t) : -1;
    }
    double acc[RT][RC];
#pragma unroll
    for (int a = 0; a < RT; ++a)
#pragma unroll
        for (int c = 0; c < RC; ++c) acc[a][c] = 0.0;
    const int nk = (n + kGK - 1) / kGK;
    const double *M = g.op(cls);
    __syncthreads();
    constexpr int kRU = (TT * kGK + NT - 1) / NT, kRM = (kGK * TJ + NT - 1) / NT;
    double ru[kRU], rm[kRM];
    auto load = [&](int kc) {
        const int k0 = kc * kGK;
#pragma unroll
        for (int r = 0; r < kRU; ++r) {
            const int e = threadIdx.x + NT * r;
            const int t = e / kGK, k = e % kGK;
            ru[r] = 0.0;
            if (t < TT) {
                const int32_t sb = src[t];
                if (sb >= 0 && k0 + k < n) ru[r] = in[(size_t)sb * n + k0 + k];
            }
        }
#pragma unroll
        for (int r = 0; r < kRM; ++r) {
            const int e = threadIdx.x + NT * r;
            const int k = e / TJ, j = e - k * TJ;
            rm[r] = (k < kGK && k0 + k < n && j0 + j < n) ? M[(size_t)(k0 + k) * ldp + j0 + j] : 0.0;
        }
    };
    load(0);
    for (int kc = 0; kc < nk; ++kc) {
#pragma unroll
        for (int r = 0; r < kRU; ++r) {
            const int e = threadIdx.x + NT * r;
            if (e < TT * kGK) Us[e % kGK][e / kGK] = ru[r];
        }
#pragma unroll
        for (int r = 0; r < kRM; ++r) {
            const int e = threadIdx.x + NT * r;
            const int k = e / TJ;
            if (k < kGK) Ms[k][e - k * TJ] = rm[r];
        }
        __syncthreads();
        if (kc + 1 < nk) load(kc + 1);
#pragma unroll
        for (int k = 0; k < kGK; ++k) {
            double uv[RT], mv[RC];
#pragma unroll
            for (int a = 0; a < RT; ++a) uv[a] = Us[k][RT * ty + a];
#pragma unroll
            for (int c = 0; c < RC; ++c) mv[c] = Ms[k][tx + 32 * c];
#pragma unroll
            for (int a = 0; a < RT; ++a)
#pragma unroll
                for (int c = 0; c < RC; ++c) acc[a][c] += uv[a] * mv[c];
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < RT; ++a) {
        const int32_t t = tgt[RT * ty + a];
        if (t < 0) continue;
#pragma unroll
        for (int c = 0; c < RC; ++c) {
            const int j = j0 + tx + 32 * c;
            if (j >= n) continue;
            double *o = out + (size_t)t * n + j;
            *o = accumulate ? *o + acc[a][c] : acc[a][c];
        }
    }
}

// out[parent] (=|+=) the sum of its children's rows, in octant order (M2M and
// the adjoint of L2L: the children's products come from one row product over
// all children of a level, grouped by octant, so that absent children cost
// nothing).
template <typename T>
__global__ void k_child_sum(const int32_t *__restrict__ parents, int64_t n_p, int n, const int32_t *__restrict__ child8,
                            const T *__restrict__ prod, T *__restrict__ out, int accumulate) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_p * n) return;
    const int64_t i = idx / n;
    const int j = (int)(idx - i * n);
    const int32_t t = parents[i];
    T v = T(0);
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const int32_t c = child8[(size_t)t * 8 + s];
        if (c >= 0) v += prod[(size_t)c * n + j];
    }
    T *o = out + (size_t)t * n + j;
    *o = accumulate ? *o + v : v;
}

// ---------------------------------------------------------------------------
// Leaf evaluation, one warp per target leaf: far field (L2P from the leaf's
// downward density on DE = 2.95 h S; M2P from the upward densities on
// UE = 1.05 h S of the W-list boxes) and near field (P2P over the U list).
// All of it is one stream of (pseudo-)sources {position relative to the leaf
// centre, weight}: the segments (own surface, W surfaces, U leaves) are laid
// end to end, and the stream is staged through shared memory in chunks of
// 128.  The next chunk's loads are issued before the current chunk is
// summed, so their latency overlaps the arithmetic.
//
// Tiling <TPL, G>: the warp splits into G groups of 32/G lanes; lane m of a
// group owns targets tbase + m + (32/G) k (k < TPL) and the group takes every
// G-th source of each chunk.  Up to 64 sources per lane are summed plainly,
// then added to the totals with two-sum; the groups' totals are combined in
// FP64 with shuffles and the result overwrites res.  The tile is picked per
// leaf so that (32/G) TPL covers its targets with little waste.
//
// Only the leaf's own particles can sit at distance zero from a target (a
// particle's own position, or a coincident particle: equal positions have
// equal keys, hence the same leaf); that segment is summed with the r = 0
// test, every other one without it.  Distinct particles of different leaves
// whose separation rounds to zero in the compute type would give a
// non-finite sum: the kernel reports KIFMM_ERR_NONFINITE for them.
// ---------------------------------------------------------------------------
constexpr int kLW = 4;               // warps (target leaves) per block
constexpr int kLK = 4;               // sources per lane per chunk
constexpr int kLChunk = 32 * kLK;    // sources per staged chunk
constexpr int kLFlush = 64;          // sources per lane summed plainly before a compensated flush
constexpr int kLSeg = 32;            // segments per batch (one per lane)

template <typename T>
__device__ __forceinline__ T pow2(int e);
template <>
__device__ __forceinline__ float pow2<float>(int e) {
    return __int_as_float((127 + e) << 23);
}
template <>
__device__ __forceinline__ double pow2<double>(int e) {
    return __longlong_as_double((long long)(1023 + e) << 52);
}

// c_a - c_b along one axis for boxes (level, integer coordinate): both
// centres are odd multiples of 2^-(level+1), so the difference is an integer
// below 2^22 times 2^-(L+1) and exact in FP32.
template <typename T>
__device__ __forceinline__ T centre_diff(int ca, int la, int cb, int lb) {
    const int L = max(la, lb);
    const int na = (2 * ca + 1) << (L - la), nb = (2 * cb + 1) << (L - lb);
    return (T)(na - nb) * pow2<T>(-(L + 1));
}

template <typename T, int TPL>
struct LeafAcc {
    T tx[TPL], ty[TPL], tz[TPL];
    T part[TPL][4];             // plain partial sums since the last flush
    T acc[TPL][4], cmp[TPL][4]; // compensated totals (two-sum)
    int pend;                   // sources per lane in part (warp-uniform bound)
    // FP32: the pair loop runs on packed f32x2 arithmetic, two sources per
    // instruction: negated targets duplicated into both halves, and plain
    // partial sums per half (folded into part at each flush)
    float2 ntx[TPL], nty[TPL], ntz[TPL];
    float2 pk[TPL][4];
};

template <typename T, int TPL>
__device__ __forceinline__ void leaf_flush(LeafAcc<T, TPL> &L) {
#pragma unroll
    for (int k = 0; k < TPL; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if constexpr (sizeof(T) == 4) {
                L.part[k][c] = L.pk[k][c].x + L.pk[k][c].y;
                L.pk[k][c] = make_float2(0.f, 0.f);
            }
            T sum, err;
            two_sum<T>(L.acc[k][c], L.part[k][c], sum, err);
            L.acc[k][c] = sum;
            L.cmp[k][c] += err;
            L.part[k][c] = T(0);
        }
    L.pend = 0;
}

// One segment of the source stream: positions are r * raw + o (surfaces:
// unit-surface points; particles: r = 1, raw = position in the source leaf's
// frame), weights hw * raw weight.
template <typename T>
struct LeafSeg {
    T ox, oy, oz, r, hw;
    int base;   // first particle, or first weight of the surface
    int kind;   // 0 own surface, 1 W-list surface, 2 particles
};

template <typename T>
struct LeafSmem {
    typename Vec4<T>::type buf[2][kLChunk];
    LeafSeg<T> seg[kLSeg];
    int start[kLSeg];
};

struct LeafCtx {
    const int32_t *lvl, *cx, *cy, *cz, *first, *cnt;
    const uint32_t *u_ptr, *w_ptr;
    const int32_t *u_idx, *w_idx;
    int ns;
    const double *dbar;  // per-box mean of the downward check potential, or nullptr
    LeafTiling tile;     // tile id per remaining-target bucket
    int *status;         // device status word
    const int8_t *u_sh, *w_sh;  // image shifts of the U and W entries (periodic cell), or null
    // Forward evaluate of a free-space plan: the outputs in caller order with
    // the physical scales (coef / (4 pi side), / side^2 of the particle's
    // system), written by the pass itself next to its FP64 results; null
    // elsewhere (the results are scattered by k_finalize).
    const uint32_t *perm = nullptr;
    const int32_t *sys = nullptr;
    const double *out_scale = nullptr;
    void *pot = nullptr, *grad = nullptr;
    int out_f64 = 0;
};


// Source weights of the leaf stage.  Forward: own surface dn_dens * h_b,
// W surfaces up_dens * h_a, particles q.  Adjoint (same geometry): own
// surface u-bar, W surfaces d-bar, particles w.
template <typename T>
struct LeafW {
    const T *own;
    int own_h;
    const T *wl;
    int wl_h;
    const T *pw;  // sorted per-particle weights, or nullptr for the charges
};

// Sources j in [lo, hi) of a staged chunk with j = grp (mod G).
template <typename T, int TPL, int G, bool CHECK>
__device__ __forceinline__ void leaf_range(LeafAcc<T, TPL> &L, const typename Vec4<T>::type *buf, int lo, int hi,
                                           int grp) {
    // sources in flight per iteration: about four pair evaluations per lane
    constexpr int UNR = (sizeof(T) == 8 || TPL >= 3) ? 1 : (TPL == 2 ? 2 : 4);
#pragma unroll UNR
    for (int j = lo + ((grp - lo) & (G - 1)); j < hi; j += G) {
        const auto s = buf[j];
#pragma unroll
        for (int k = 0; k < TPL; ++k) {
            if constexpr (CHECK)
                lap_accum<T>(L.tx[k] - s.x, L.ty[k] - s.y, L.tz[k] - s.z, s.w, L.part[k][0], L.part[k][1],
                             L.part[k][2], L.part[k][3]);
            else
                lap_accum_nz<T>(L.tx[k] - s.x, L.ty[k] - s.y, L.tz[k] - s.z, s.w, L.part[k][0], L.part[k][1],
                                L.part[k][2], L.part[k][3]);
        }
    }
}

// FP32 chunks are staged as source pairs: pair p holds sources a and a + G
// with a = (p / G) 2G + p % G, as eight floats (x_a x_b y_a y_b z_a z_b w_a
// w_b), so group g (p % G = g) meets its own sources g, g + G, g + 2G, ...
// two at a time, each pair already in the register halves of the f32x2
// instructions.  Entries beyond the chunk's sources hold a null source
// (weight 0, far away), which adds exactly zero.
__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// Pairs i in [ia, ie) of group grp (pair index grp + i G).
template <int TPL, int G, bool CHECK>
__device__ __forceinline__ void leaf_pairs(LeafAcc<float, TPL> &L, const float4 *__restrict__ pairs, int ia, int ie,
                                           int grp) {
    constexpr int UNR = TPL == 1 ? 4 : 1;  // eight pair evaluations in flight per lane (the FP32 chains are latency-bound)
#pragma unroll UNR
    for (int i = ia; i < ie; ++i) {
        const int p = grp + i * G;
        const float4 A = pairs[2 * p], B = pairs[2 * p + 1];
        const float2 sx = make_float2(A.x, A.y), sy = make_float2(A.z, A.w);
        const float2 sz = make_float2(B.x, B.y), sw = make_float2(B.z, B.w);
#pragma unroll
        for (int k = 0; k < TPL; ++k) {
            // r = source - target (the gradient sum below is then + r w / r^3)
            const float2 rx = __fadd2_rn(sx, L.ntx[k]);
            const float2 ry = __fadd2_rn(sy, L.nty[k]);
            const float2 rz = __fadd2_rn(sz, L.ntz[k]);
            float2 r2 = __fmul2_rn(rx, rx);
            r2 = __ffma2_rn(ry, ry, r2);
            r2 = __ffma2_rn(rz, rz, r2);
            float2 ri;
            if constexpr (CHECK) {
                ri.x = r2.x > 0.f ? rsqrt_t<float>(r2.x) : 0.f;
                ri.y = r2.y > 0.f ? rsqrt_t<float>(r2.y) : 0.f;
            } else {
                ri.x = rsqrt_t<float>(r2.x);
                ri.y = rsqrt_t<float>(r2.y);
            }
            const float2 wr = __fmul2_rn(sw, ri);
            const float2 wr3 = __fmul2_rn(wr, __fmul2_rn(ri, ri));
            L.pk[k][0] = __fadd2_rn(L.pk[k][0], wr);
            L.pk[k][1] = __ffma2_rn(rx, wr3, L.pk[k][1]);
            L.pk[k][2] = __ffma2_rn(ry, wr3, L.pk[k][2]);
            L.pk[k][3] = __ffma2_rn(rz, wr3, L.pk[k][3]);
        }
    }
}

// A staged FP32 chunk of m sources (pair layout); [olo, ohi) are the leaf's
// own particles: the pairs of group grp that touch them take the r = 0 test.
// Sub-blocks of kLFlush / 2 pairs keep every plain partial sum to at most
// kLFlush terms.
template <int TPL, int G>
__device__ __forceinline__ void leaf_chunk_pk(LeafAcc<float, TPL> &L, const float4 *pairs, int m, int olo, int ohi,
                                              int grp) {
    const int np = grp < m ? (m - grp + 2 * G - 1) / (2 * G) : 0;
    // pair i holds this group's sources 2 i G + grp and 2 i G + grp + G
    const int i_lo = max(0, floor_div(olo - grp - G + 2 * G - 1, 2 * G));
    const int i_hi = max(0, floor_div(ohi - grp + 2 * G - 1, 2 * G));
    for (int i0 = 0; i0 < np; i0 += kLFlush / 2) {
        const int i1 = min(np, i0 + kLFlush / 2);
        const int a = max(i0, min(i1, i_lo)), e = max(a, min(i1, i_hi));
        leaf_pairs<TPL, G, false>(L, pairs, i0, a, grp);
        if (a < e) leaf_pairs<TPL, G, true>(L, pairs, a, e, grp);
        leaf_pairs<TPL, G, false>(L, pairs, e, i1, grp);
        L.pend += 2 * (i1 - i0);
        if (L.pend >= kLFlush) leaf_flush<float, TPL>(L);
    }
}

// A staged chunk of m sources; [olo, ohi) are the leaf's own particles.
// Sub-blocks of kLFlush G sources keep every plain partial sum to at most
// kLFlush terms.
template <typename T, int TPL, int G>
__device__ __forceinline__ void leaf_chunk(LeafAcc<T, TPL> &L, const typename Vec4<T>::type *buf, int m, int olo,
                                           int ohi, int grp) {
    if constexpr (sizeof(T) == 4) {
        leaf_chunk_pk<TPL, G>(L, buf, m, olo, ohi, grp);
        return;
    }
    for (int s0 = 0; s0 < m; s0 += kLFlush * G) {
        const int s1 = min(m, s0 + kLFlush * G);
        const int a = max(s0, min(s1, olo)), e = max(a, min(s1, ohi));
        leaf_range<T, TPL, G, false>(L, buf, s0, a, grp);
        if (a < e) leaf_range<T, TPL, G, true>(L, buf, a, e, grp);
        leaf_range<T, TPL, G, false>(L, buf, e, s1, grp);
        L.pend += (s1 - s0 + G - 1) / G;
        if (L.pend >= kLFlush) leaf_flush<T, TPL>(L);
    }
}

// Loads of chunk c of a batch: lane l takes stream entries c kLChunk + l + 32 i.
template <typename T>
__device__ __forceinline__ void leaf_fetch(const LeafSmem<T> &S, int c, int total, int nb,
                                           const typename Vec4<T>::type *__restrict__ pts,
                                           const T *__restrict__ surf, const LeafW<T> &W,
                                           typename Vec4<T>::type (&raw)[kLK], int (&rs)[kLK]) {
    const int lane = threadIdx.x & 31;
    // the lane's entries increase with i: one binary search, then linear steps
    int s = 0;
#pragma unroll
    for (int i = 0; i < kLK; ++i) {
        const int j = c * kLChunk + lane + 32 * i;
        rs[i] = -1;
        if (j < total) {
            if (i == 0) {
#pragma unroll
                for (int step = kLSeg / 2; step > 0; step >>= 1)
                    if (s + step < nb && S.start[s + step] <= j) s += step;
            } else {
                while (s + 1 < nb && S.start[s + 1] <= j) ++s;
            }
            const int k = j - S.start[s];
            const int kind = S.seg[s].kind, base = S.seg[s].base;
            rs[i] = s;
            if (kind == 2) {
                raw[i] = pts[base + k];
                if (W.pw) raw[i].w = W.pw[base + k];
            } else {
                raw[i].x = surf[3 * k];
                raw[i].y = surf[3 * k + 1];
                raw[i].z = surf[3 * k + 2];
                raw[i].w = (kind == 0 ? W.own : W.wl)[base + k];
            }
        }
    }
}

// Place fetched entries (segment transform applied) in staging buffer slot;
// FP32 in the pair layout of leaf_chunk_pk, with null sources past the end.
template <typename T, int G>
__device__ __forceinline__ void leaf_store(LeafSmem<T> &S, int slot, const typename Vec4<T>::type (&raw)[kLK],
                                           const int (&rs)[kLK]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < kLK; ++i) {
        typename Vec4<T>::type v;
        if (rs[i] >= 0) {
            const LeafSeg<T> g = S.seg[rs[i]];
            v.x = g.r * raw[i].x + g.ox;
            v.y = g.r * raw[i].y + g.oy;
            v.z = g.r * raw[i].z + g.oz;
            v.w = raw[i].w * g.hw;
        } else {
            if constexpr (sizeof(T) == 8) continue;
            v.x = v.y = v.z = T(1e4);  // null source: weight 0 at a finite distance
            v.w = T(0);
        }
        const int j = lane + 32 * i;
        if constexpr (sizeof(T) == 4) {
            const int r = j % (2 * G), pair = (j / (2 * G)) * G + r % G, h = r / G;
            float *P = reinterpret_cast<float *>(&S.buf[slot][0]) + 8 * pair;
            P[h] = v.x;
            P[2 + h] = v.y;
            P[4 + h] = v.z;
            P[6 + h] = v.w;
        } else {
            S.buf[slot][j] = v;
        }
    }
}

// WPP warps share a pass (all warps of the block): warp `sub` takes every
// WPP-th chunk of the stream, and the totals are added in warp order.
template <typename T, int TPL, int G, int WPP>
__device__ void leaf_pass(const LeafCtx &C, int b, int tbase, const typename Vec4<T>::type *__restrict__ pts,
                          const T *__restrict__ surf, const LeafW<T> &W, LeafSmem<T> *bufs, int sub,
                          double4 *__restrict__ res) {
    using V4 = typename Vec4<T>::type;
    LeafSmem<T> &S = bufs[sub];
    constexpr int LG = 32 / G;  // lanes per group
    const int lane = threadIdx.x & 31, grp = lane / LG, mem = lane % LG;
    const int lb = C.lvl[b], bx = C.cx[b], by = C.cy[b], bz = C.cz[b];
    const int n = C.cnt[b], f = C.first[b], ns = C.ns;
    LeafAcc<T, TPL> L;
#pragma unroll
    for (int k = 0; k < TPL; ++k) {
        const int i = tbase + mem + LG * k;
        V4 v{};
        if (i < n) v = pts[f + i];
        L.tx[k] = v.x;
        L.ty[k] = v.y;
        L.tz[k] = v.z;
        if constexpr (sizeof(T) == 4) {
            L.ntx[k] = make_float2(-(float)v.x, -(float)v.x);
            L.nty[k] = make_float2(-(float)v.y, -(float)v.y);
            L.ntz[k] = make_float2(-(float)v.z, -(float)v.z);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            L.part[k][c] = L.acc[k][c] = L.cmp[k][c] = T(0);
            L.pk[k][c] = make_float2(0.f, 0.f);
        }
    }
    L.pend = 0;
    const uint32_t w0 = C.w_ptr[b], u0 = C.u_ptr[b];
    const int nw = (int)(C.w_ptr[b + 1] - w0), nu = (int)(C.u_ptr[b + 1] - u0);
    const int nseg = 1 + nw + nu;
    for (int sb = 0; sb < nseg; sb += kLSeg) {
        // lane e describes segment sb + e of (own surface, W list, U list)
        const int e = sb + lane;
        LeafSeg<T> d{T(0), T(0), T(0), T(1), T(1), 0, 2};
        int cnt = 0, own = 0;
        if (e == 0) {
            d.r = (T)kAlphaOuter * pow2<T>(-(lb + 1));
            d.hw = W.own_h ? pow2<T>(-(lb + 1)) : T(1);
            d.base = b * ns;
            d.kind = 0;
            cnt = ns;
        } else if (e <= nw) {
            const int a = C.w_idx[w0 + e - 1], la = C.lvl[a];
            d.ox = centre_diff<T>(C.cx[a], la, bx, lb);
            d.oy = centre_diff<T>(C.cy[a], la, by, lb);
            d.oz = centre_diff<T>(C.cz[a], la, bz, lb);
            if (C.w_sh) {
                T ix, iy, iz;
                image_offset<T>(C.w_sh[w0 + e - 1], ix, iy, iz);
                d.ox += ix, d.oy += iy, d.oz += iz;
            }
            d.r = (T)kAlphaInner * pow2<T>(-(la + 1));
            d.hw = W.wl_h ? pow2<T>(-(la + 1)) : T(1);
            d.base = a * ns;
            d.kind = 1;
            cnt = ns;
        } else if (e < nseg) {
            const int a = C.u_idx[u0 + e - 1 - nw], la = C.lvl[a];
            d.ox = centre_diff<T>(C.cx[a], la, bx, lb);
            d.oy = centre_diff<T>(C.cy[a], la, by, lb);
            d.oz = centre_diff<T>(C.cz[a], la, bz, lb);
            const int sa = C.u_sh ? (int)C.u_sh[u0 + e - 1 - nw] : 13;
            if (sa != 13) {
                T ix, iy, iz;
                image_offset<T>(sa, ix, iy, iz);
                d.ox += ix, d.oy += iy, d.oz += iz;
            }
            d.base = C.first[a];
            cnt = C.cnt[a];
            own = (a == b) && sa == 13;  // another image of the leaf is not its own particles
        }
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const unsigned own_mask = __ballot_sync(0xffffffffu, own);
        int olo = 0, ohi = 0;
        if (own_mask) {
            const int o = __ffs(own_mask) - 1;
            ohi = __shfl_sync(0xffffffffu, incl, o);
            olo = ohi - __shfl_sync(0xffffffffu, cnt, o);
        }
        __syncwarp();  // the previous batch is done with seg, start and buf
        S.seg[lane] = d;
        S.start[lane] = (e < nseg) ? incl - cnt : total;
        __syncwarp();
        const int nb = min(kLSeg, nseg - sb);
        typename Vec4<T>::type raw[kLK];
        int rs[kLK];
        const int nchunks = (total + kLChunk - 1) / kLChunk;
        for (int c = WPP > 1 ? sub : 0, slot = 0; c < nchunks; c += WPP, slot ^= 1) {
            // double-buffered: the slot written here was last read two chunks ago
            leaf_fetch<T>(S, c, total, nb, pts, surf, W, raw, rs);
            leaf_store<T, G>(S, slot, raw, rs);
            __syncwarp();
            const int c0 = c * kLChunk;
            leaf_chunk<T, TPL, G>(L, S.buf[slot], min(kLChunk, total - c0), olo - c0, ohi - c0, grp);
        }
    }
    leaf_flush<T, TPL>(L);
    double totals[TPL][4];
#pragma unroll
    for (int k = 0; k < TPL; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            totals[k][c] = (double)L.acc[k][c] + (double)L.cmp[k][c];
#pragma unroll
            for (int o = 16; o >= LG; o >>= 1) totals[k][c] += __shfl_xor_sync(0xffffffffu, totals[k][c], o);
        }
    if constexpr (WPP > 1) {
        // each warp's totals through its own staging buffer (its chunks are done)
        static_assert(sizeof(S.buf) >= sizeof(double) * 32 * TPL * 4, "room for a warp's totals");
        __syncwarp();
        double *own = reinterpret_cast<double *>(&S.buf[0][0]);
#pragma unroll
        for (int k = 0; k < TPL; ++k)
#pragma unroll
            for (int c = 0; c < 4; ++c) own[(4 * k + c) * 32 + lane] = totals[k][c];
        __syncthreads();
        if (sub != 0) return;
        for (int w = 1; w < WPP; ++w) {
            const double *o = reinterpret_cast<const double *>(&bufs[w].buf[0][0]);
#pragma unroll
            for (int k = 0; k < TPL; ++k)
#pragma unroll
                for (int c = 0; c < 4; ++c) totals[k][c] += o[(4 * k + c) * 32 + lane];
        }
    }
#pragma unroll
    for (int k = 0; k < TPL; ++k) {
        double(&tot)[4] = totals[k];
        if (C.dbar) tot[0] += C.dbar[b];  // the constant part of the local expansion
        const int i = tbase + mem + LG * k;
        if (grp == 0 && i < n) {
            res[f + i] = make_double4(tot[0], tot[1], tot[2], tot[3]);
            if (!isfinite(tot[0] + tot[1] + tot[2] + tot[3])) set_status(C.status, KIFMM_ERR_NONFINITE);
            if (C.pot || C.grad) {  // the finalisation, as k_finalize does it
                const uint32_t j = C.perm[f + i];
                const int sy = C.sys[b];
                const double c1 = C.out_scale[2 * sy], c2 = C.out_scale[2 * sy + 1];
                if (C.out_f64) {
                    if (C.pot) ((double *)C.pot)[j] = c1 * tot[0];
                    if (C.grad) {
                        double *g = (double *)C.grad + 3 * (size_t)j;
                        g[0] = c2 * tot[1];
                        g[1] = c2 * tot[2];
                        g[2] = c2 * tot[3];
                    }
                } else {
                    if (C.pot) ((float *)C.pot)[j] = (float)(c1 * tot[0]);
                    if (C.grad) {
                        float *g = (float *)C.grad + 3 * (size_t)j;
                        g[0] = (float)(c2 * tot[1]);
                        g[1] = (float)(c2 * tot[2]);
                        g[2] = (float)(c2 * tot[3]);
                    }
                }
            }
        }
    }
}
// Leaf work items: a leaf is covered greedily by passes (leaf, first
// target); the pass over r remaining targets uses the plan table's variant
// for r (bucket (r - 1) / 8) and covers (32 / G) TPL of them, so e.g. 40
// targets become a 32-target pass and an 8-target pass with four source
// groups, keeping every lane busy.  One kernel per variant, each with the
// registers its tile needs; k_leaf_partition lists the items of each
// variant (order within a list is immaterial: passes are independent).
__global__ void k_leaf_partition(int64_t n_leaves, const int32_t *__restrict__ leaves,
                                 const int32_t *__restrict__ cnt, LeafTiling tile, int64_t cap,
                                 int2 *__restrict__ lists, int32_t *__restrict__ counts) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const bool valid = i < n_leaves;
    const int b = valid ? leaves[i] : -1;
    const int n = valid ? cnt[b] : 0;
    // places for all of a leaf's passes at once: leaves stay in order in every
    // list (coarse leaves, with the longest source lists, first), where places
    // taken pass by pass put a coarse leaf's last passes at the end
    int mine[kLeafTiles];
#pragma unroll
    for (int u = 0; u < kLeafTiles; ++u) mine[u] = 0;
    for (int t0 = 0; t0 < n;) {
        const int v = leaf_variant(tile, n - t0);
#pragma unroll
        for (int u = 0; u < kLeafTiles; ++u) mine[u] += u == v ? 1 : 0;
        t0 += (32 / leaf_tile_groups(v)) * leaf_tile_tpl(v);
    }
    __syncwarp();
    int at[kLeafTiles];
#pragma unroll
    for (int u = 0; u < kLeafTiles; ++u) {
        at[u] = 0;
        if (!__any_sync(0xffffffffu, mine[u] > 0)) continue;
        int incl = mine[u];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        int base = 0;
        if (lane == 31) base = atomicAdd(&counts[u], incl);
        at[u] = __shfl_sync(0xffffffffu, base, 31) + incl - mine[u];
    }
    for (int t0 = 0; t0 < n;) {
        const int v = leaf_variant(tile, n - t0);
#pragma unroll
        for (int u = 0; u < kLeafTiles; ++u)
            if (u == v) lists[(int64_t)u * cap + at[u]++] = make_int2(b, t0);
        t0 += (32 / leaf_tile_groups(v)) * leaf_tile_tpl(v);
    }
}

// Each warp (FP64: each block) takes the next pass from a shared counter as it
// finishes one (passes differ in length by their source lists; a fixed stride
// left the last warps running alone).  Every pass writes only its own targets,
// so the order passes are taken in does not change any result.
//
// FP64 is bound by the FP64 unit (two lanes per clock and SM, some 19
// operations per pair), so a pass of one warp is long: 32 targets of a leaf
// with 6000 sources take 3.5 ms, and a 60k Plummer cloud spent two thirds of
// its leaf stage waiting for the last of them.  The four warps of a block
// therefore share each pass (that cloud, p = 6: the whole step 12.3 -> 9.0 ms;
// 4096 points, p = 4: 2.06 -> 1.43 ms).
template <typename T>
__host__ __device__ constexpr int leaf_blocks_per_sm(int tpl) {
    return sizeof(T) == 4 ? (tpl == 1 ? 5 : 4) : 3;
}
template <typename T, int TPL, int G>
__global__ void __launch_bounds__(32 * kLW, leaf_blocks_per_sm<T>(TPL))
    k_leaf_all(LeafCtx C, const int2 *__restrict__ list, const int32_t *__restrict__ count, int32_t *next,
               const typename Vec4<T>::type *__restrict__ pts, const T *__restrict__ surf, LeafW<T> W,
               double4 *__restrict__ res) {
    __shared__ LeafSmem<T> bufs[kLW];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nl = *count;
    if constexpr (sizeof(T) == 8) {
        __shared__ int taken;
        while (true) {
            __syncthreads();  // the previous pass is done with taken and the buffers
            if (threadIdx.x == 0) taken = atomicAdd(next, 1);
            __syncthreads();
            if (taken >= nl) break;
            const int2 it = list[taken];
            leaf_pass<T, TPL, G, kLW>(C, it.x, it.y, pts, surf, W, bufs, warp, res);
        }
    } else {
        while (true) {
            int li = 0;
            if (lane == 0) li = atomicAdd(next, 1);
            li = __shfl_sync(0xffffffffu, li, 0);
            if (li >= nl) break;
            const int2 it = list[li];
            leaf_pass<T, TPL, G, 1>(C, it.x, it.y, pts, surf, W, bufs, warp, res);
        }
    }
}

template <typename T, int TPL, int G>
void leaf_launch_variant(const Plan &P, const LeafCtx &C, int v, const typename Vec4<T>::type *pts, const T *surf,
                         const LeafW<T> &W, double4 *res, cudaStream_t caller) {
    // on the variant's own stream, after the partition; joined back below
    cudaStream_t s = P.leaf_streams[v];
    cudaStreamWaitEvent(s, P.leaf_fork, 0);
    constexpr int occ = leaf_blocks_per_sm<T>(TPL);
    const int64_t want = sizeof(T) == 8 ? P.n_leaves : (P.n_leaves + kLW - 1) / kLW;
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)P.num_sms * occ));
    ++g_launches, k_leaf_all<T, TPL, G><<<g, 32 * kLW, 0, s>>>(C, P.leaf_vlist + (int64_t)v * P.leaf_item_cap,
                                                                P.leaf_vcnt + v, P.leaf_vcnt + 8 + v, pts, surf,
                                                                W, res);
    cudaEventRecord(P.leaf_join[v], s);
    cudaStreamWaitEvent(caller, P.leaf_join[v], 0);
}

// All leaves: work items by variant, then one launch per variant the table
// uses, each on its own stream so that the short variants' tails (a pass of
// one warp over a leaf's whole source list) overlap the long one.
template <typename T>
void leaf_launch(const Plan &P, const LeafCtx &C, const typename Vec4<T>::type *pts, const T *surf,
                 const LeafW<T> &W, double4 *res, cudaStream_t s) {
    if (P.n_leaves == 0) return;
    cudaMemsetAsync(P.leaf_vcnt, 0, sizeof(int32_t) * 16, s);  // counts and next-pass counters
    ++g_launches, k_leaf_partition<<<(unsigned)((P.n_leaves + 255) / 256), 256, 0, s>>>(
                      P.n_leaves, P.leaves, P.cnt, C.tile, P.leaf_item_cap, P.leaf_vlist, P.leaf_vcnt);
    cudaEventRecord(P.leaf_fork, s);
    bool used[kLeafTiles] = {false};
    for (int i = 0; i < kLeafBuckets; ++i) used[C.tile.get(i)] = true;
    if (used[0]) leaf_launch_variant<T, 1, 4>(P, C, 0, pts, surf, W, res, s);
    if (used[1]) leaf_launch_variant<T, 2, 4>(P, C, 1, pts, surf, W, res, s);
    if (used[2]) leaf_launch_variant<T, 1, 2>(P, C, 2, pts, surf, W, res, s);
    if (used[3]) leaf_launch_variant<T, 2, 2>(P, C, 3, pts, surf, W, res, s);
    if (used[4]) leaf_launch_variant<T, 1, 1>(P, C, 4, pts, surf, W, res, s);
    if (used[5]) leaf_launch_variant<T, 2, 1>(P, C, 5, pts, surf, W, res, s);
}

// Scatter to caller order with 1/(4 pi), coef and physical units.
template <typename TO>
__global__ void k_finalize(int64_t n, const double4 *__restrict__ res, const uint32_t *__restrict__ perm,
                           const int64_t *__restrict__ off, int S, const double *__restrict__ out_scale,
                           TO *pot, TO *grad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= (int64_t)j) lo = mid; else hi = mid - 1;
    }
    const double c1 = out_scale[2 * lo], c2 = out_scale[2 * lo + 1];  // coef / (4 pi side), / side^2
    const double4 r = res[i];
    if (pot) pot[j] = (TO)(c1 * r.x);
    if (grad) {
        grad[3 * j] = (TO)(c2 * r.y);
        grad[3 * j + 1] = (TO)(c2 * r.z);
        grad[3 * j + 2] = (TO)(c2 * r.w);
    }
}

// Energy partial sums over chunks that never straddle systems (sorted order).
template <typename T>
__global__ void k_energy_chunks(const int64_t *__restrict__ chunks, const double4 *__restrict__ res,
                                const typename Vec4<T>::type *__restrict__ pts, double *partial) {
    __shared__ double red[256];
    const int64_t a = chunks[2 * blockIdx.x], e = chunks[2 * blockIdx.x + 1];
    double s = 0.0;
    for (int64_t i = a + threadIdx.x; i < e; i += blockDim.x) s += (double)pts[i].w * res[i].x;
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

__global__ void k_energy_sum(const int32_t *__restrict__ chunk_start, const double *__restrict__ partial,
                             const double *__restrict__ lo_side, double coef, int S, double *energy) {
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    double e = 0.0;
    for (int c = chunk_start[s]; c < chunk_start[s + 1]; ++c) e += partial[c];
    energy[s] = 0.5 * coef * kInv4Pi / lo_side[s * 4 + 3] * e;
}

// Clump force and torque, FP64 accumulation, one thread per clump.
template <typename TO>
__global__ void k_clump(int64_t nc, const int64_t *__restrict__ off, const TO *__restrict__ xyz,
                        const TO *__restrict__ q, const TO *__restrict__ grad, const TO *__restrict__ ref,
                        TO *force, TO *torque) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    double F[3] = {0, 0, 0}, Tq[3] = {0, 0, 0};
    const double rx = ref[3 * c], ry = ref[3 * c + 1], rz = ref[3 * c + 2];
    for (int64_t k = off[c]; k < off[c + 1]; ++k) {
        const double qk = q[k];
        const double f0 = -qk * (double)grad[3 * k], f1 = -qk * (double)grad[3 * k + 1],
                     f2 = -qk * (double)grad[3 * k + 2];
        const double dx = (double)xyz[3 * k] - rx, dy = (double)xyz[3 * k + 1] - ry,
                     dz = (double)xyz[3 * k + 2] - rz;
        F[0] += f0;
        F[1] += f1;
        F[2] += f2;
        Tq[0] += dy * f2 - dz * f1;
        Tq[1] += dz * f0 - dx * f2;
        Tq[2] += dx * f1 - dy * f0;
    }
    for (int d = 0; d < 3; ++d) {
        force[3 * c + d] = (TO)F[d];
        torque[3 * c + d] = (TO)Tq[d];
    }
}


inline unsigned grid_for(int64_t n, int block) { return (unsigned)((n + block - 1) / block); }

// k_p2m launch shape: a thread per check point, four staged values per thread.
inline int p2m_threads(const Plan &P) { return (P.ns + 31) / 32 * 32; }
// k_p2l: a thread per check point and, in FP64, up to four source groups.
template <typename T>
inline int p2l_threads(const Plan &P) {
    const int t = p2m_threads(P);
    return sizeof(T) == 8 ? t * std::max(1, std::min(4, 640 / t)) : t;
}
template <typename T>
inline size_t p2m_smem(const Plan &P) { return 7 * sizeof(T) * (size_t)p2m_threads(P); }

constexpr int kRowsSmallMax = 200 * 1024;  // shared memory of a small tile (FP64: n_s up to 512)

// Elements of an operator block of n inputs and ld outputs (padded).
inline int64_t op_block(int n, int ld) { return (int64_t)gemm_nkp(n) * gemm_ldp(ld); }

template <typename T, bool VEC>
void rows_small_launch(const RowMap<T> &g, const int32_t *targets, const ClassRanges &cr, int64_t most, int ncls,
                       bool few, int n, int ld, const T *in, T *out, int accumulate, double *dbar, cudaStream_t s) {
    const int nkp = gemm_nkp(n), ldp = gemm_ldp(ld), rw = few ? 1 : 4;
    const dim3 grid(grid_for(most, 4 * rw), ncls, grid_for(ld, kSmallCols));
    const size_t smem = rows_small_smem<T>(nkp, rw);
    if (few)
        ++g_launches, k_rows_small<T, VEC, 1><<<grid, kRThreads, smem, s>>>(g, targets, cr, n, nkp, ldp, in, out,
                                                                           accumulate, dbar);
    else
        ++g_launches, k_rows_small<T, VEC, 4><<<grid, kRThreads, smem, s>>>(g, targets, cr, n, nkp, ldp, in, out,
                                                                           accumulate, dbar);
}

template <bool VEC>
void rows_launch_f32(const RowMap<float> &g, const int32_t *targets, const ClassRanges &cr, int64_t most, int ncls,
                     bool big, bool few, int n, int ld, const float *in, float *out, int accumulate, double *dbar,
                     cudaStream_t s) {
    const int nkp = gemm_nkp(n), ldp = gemm_ldp(ld), nc = gemm_nc(ld);
    if (!big) return rows_small_launch<float, VEC>(g, targets, cr, most, ncls, few, n, ld, in, out, accumulate, dbar, s);
    const dim3 grid(grid_for(most, 64), ncls, ldp / (32 * nc));
    switch (nc) {
        case 1: ++g_launches, k_rows_big<1, VEC><<<grid, kRThreads, 0, s>>>(g, targets, cr, n, nkp, ldp, in, out, accumulate, dbar); break;
        case 2: ++g_launches, k_rows_big<2, VEC><<<grid, kRThreads, 0, s>>>(g, targets, cr, n, nkp, ldp, in, out, accumulate, dbar); break;
        case 3: ++g_launches, k_rows_big<3, VEC><<<grid, kRThreads, 0, s>>>(g, targets, cr, n, nkp, ldp, in, out, accumulate, dbar); break;
        case 4: ++g_launches, k_rows_big<4, VEC><<<grid, kRThreads, 0, s>>>(g, targets, cr, n, nkp, ldp, in, out, accumulate, dbar); break;
        default: ++g_launches, k_rows_big<5, VEC><<<grid, kRThreads, 0, s>>>(g, targets, cr, n, nkp, ldp, in, out, accumulate, dbar); break;
    }
}

// out[t] (=|+=) Op in[src(t)] for the rows targets[starts[c] .. starts[c + 1])
// of class c < ncls; ld = n, or n + 1 with the mean row (FP32-based modes).
// The big tile once its blocks fill the GPU, the small one below (a level of
// few boxes is latency-bound).
template <typename T>
void rows(Plan &P, const RowMap<T> &g, const int32_t *targets, const int64_t *starts, int ncls, const T *in, T *out,
          int accumulate, cudaStream_t s, int ld = 0, double *dbar = nullptr) {
    ClassRanges cr;
    int64_t most = 0, total = 0;
    for (int c = 0; c <= 8; ++c) cr.b[c] = starts[std::min(c, ncls)];
    for (int c = 0; c < ncls; ++c) {
        most = std::max<int64_t>(most, starts[c + 1] - starts[c]);
        total += starts[c + 1] - starts[c];
    }
    if (most <= 0) return;
    const int n = P.ns;
    if (ld == 0) ld = n;
    // blocks of 16 rows by 32 outputs
    const int64_t small_blocks = (int64_t)grid_for(total, 16) * grid_for(ld, kSmallCols);
    const bool few = small_blocks < (sizeof(T) == 4 ? 1 : 4) * (int64_t)P.num_sms;
    if constexpr (sizeof(T) == 4) {
        const bool big = (int64_t)grid_for(total, 64) * (gemm_ldp(ld) / (32 * gemm_nc(ld))) >= P.num_sms;
        if (n % 4 == 0)
            rows_launch_f32<true>(g, targets, cr, most, ncls, big, few, n, ld, in, out, accumulate, dbar, s);
        else
            rows_launch_f32<false>(g, targets, cr, most, ncls, big, few, n, ld, in, out, accumulate, dbar, s);
    } else if ((int64_t)grid_for(total, 64) * grid_for(n, 160) >= 2 * P.num_sms ||
               rows_small_smem<double>(gemm_nkp(n)) > (size_t)kRowsSmallMax) {
        const dim3 grid(grid_for(most, 64), ncls, grid_for(n, 160));
        ++g_launches, k_rows_f64<<<grid, 256, 0, s>>>(g, targets, cr, n, gemm_ldp(n), in, out, accumulate);
    } else {
        rows_small_launch<double, true>(g, targets, cr, most, ncls, few, n, n, in, out, accumulate, nullptr, s);
    }
}

// The same operator for the rows targets[a .. e).
template <typename T>
void rows_one(Plan &P, const T *op, const int32_t *targets, int64_t a, int64_t e, const T *in, T *out,
              cudaStream_t s) {
    const int64_t st[2] = {a, e};
    rows<T>(P, RowMap<T>{nullptr, op, 0, false}, targets, st, 1, in, out, 0, s);
}

// out[b] (=|+=) sum over the children c of b of Op_{octant(c)} in[c], for the
// boxes b of level l that have children; prod: scratch rows.
template <typename T>
void rows_children(Plan &P, int l, const T *ops, const T *in, T *prod, T *out, int accumulate, cudaStream_t s) {
    rows<T>(P, RowMap<T>{nullptr, ops, op_block(P.ns, P.ns), true}, P.part_list[3],
            P.part_start[3].data() + 8 * (l + 1), 8, in, prod, 0, s);
    const int64_t a = P.part_start[1][1 + l], np = P.part_start[1][2 + l] - a;
    if (np > 0)
        ++g_launches, k_child_sum<T><<<grid_for(np * P.ns, 256), 256, 0, s>>>(P.part_list[1] + a, np, P.ns, P.child8,
                                                                              prod, out, accumulate);
}

// out[b] += Op_{octant(b)} in[parent(b)] for the boxes b of level l.
template <typename T>
void rows_parent(Plan &P, int l, const T *ops, const T *in, T *out, cudaStream_t s, int ld = 0,
                 double *dbar = nullptr) {
    rows<T>(P, RowMap<T>{P.parent, ops, op_block(P.ns, ld ? ld : P.ns), true}, P.part_list[3],
            P.part_start[3].data() + 8 * l, 8, in, out, 1, s, ld, dbar);
}

// Periodic cell (Sec. 2.4): the images beyond the 26 nearest act on the
// root's downward check potential, d(root) += F u(root), with F the
// far-image composite; FP64 sums, one block.  With dbar (FP32-based modes)
// the mean goes to dbar and the mean-free rest to d.  n_s^2 FP64 products on
// one SM's two FP64 lanes (6 us at n_s = 152); each output's sum is cut into
// blockDim / n_s parts so that the loads overlap (one part: 48 us).
template <typename T>
__global__ void __launch_bounds__(1024) k_far_root(int ns, const double *__restrict__ Ft, const double *__restrict__ u,
                                                   T *__restrict__ d, double *__restrict__ dbar) {
    __shared__ double v[kMaxNs];
    __shared__ double pv[1024];
    __shared__ double red[32];
    const int parts = max(1, (int)blockDim.x / ns), part = threadIdx.x / ns, jp = threadIdx.x - part * ns;
    const int chunk = (ns + parts - 1) / parts;
    static_assert(kMaxNs <= 1024, "a thread per output");
    double acc = 0.0;
    if (part < parts)
        for (int k = part * chunk; k < min(ns, (part + 1) * chunk); ++k) acc += Ft[(size_t)k * ns + jp] * u[k];
    pv[threadIdx.x] = acc;
    __syncthreads();
    for (int j = threadIdx.x; j < ns; j += blockDim.x) {
        double tot = 0.0;
        for (int q = 0; q < parts; ++q) tot += pv[q * ns + j];
        v[j] = tot;
    }
    __syncthreads();
    double mean = 0.0;
    if (dbar) {
        double sum = 0.0;
        for (int j = threadIdx.x; j < ns; j += blockDim.x) sum += v[j];
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
        __syncthreads();
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
        mean = tot / ns;
        if (threadIdx.x == 0) dbar[0] += mean;
    }
    for (int j = threadIdx.x; j < ns; j += blockDim.x) d[j] += (T)(v[j] - mean);
}

// Periodic cell: the uniform potential term of the conducting-boundary
// lattice sum that the root's equivalent density does not carry, (2 pi / 3)
// (Q2 of the particles - Q2 of the density) for the unit cell (V = 1), Q2 the
// trace of the second moment about the cell centre.  The particles' Q2 is
// the sum of the per-leaf sums in leaf order, the density's is g . u(root).
// One block, fixed summation order.
__global__ void k_moment_term(int64_t nl, const double *__restrict__ leaf_q2, int ns, const double *__restrict__ g,
                              const double *__restrict__ u_root, double *pshift) {
    __shared__ double red[2][32];
    double a = 0.0, b = 0.0;
    for (int64_t i = threadIdx.x; i < nl; i += blockDim.x) a += leaf_q2[i];
    for (int j = threadIdx.x; j < ns; j += blockDim.x) b += g[j] * u_root[j];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = a;
        red[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double qa = 0.0, qb = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) qa += red[0][w], qb += red[1][w];
        *pshift = (2.0 * 3.14159265358979323846 / 3.0) * (qa - qb);
    }
}

// FP32-based periodic plans: the root's upward check potential in FP64 from
// its children's (M2M composites in FP64, stored [k][j]); a root that is a
// leaf keeps its own.  8 n_s^2 FP64 products at two lanes per clock and SM:
// eight outputs per block spread them over the SMs (one block: 330 us at
// n_s = 152), 32 threads sharing each output's 8 n_s terms.
constexpr int kRootCols = 8;
__global__ void __launch_bounds__(32 * kRootCols) k_root_up64(int ns, const int32_t *__restrict__ child8,
                                                              const int32_t *__restrict__ nchild,
                                                              const double *__restrict__ m2m64,
                                                              const float *__restrict__ u, double *__restrict__ u64) {
    __shared__ double red[32][kRootCols];
    const int c = threadIdx.x % kRootCols, p = threadIdx.x / kRootCols;
    const int j = blockIdx.x * kRootCols + c;
    double acc = 0.0;
    if (nchild[0] == 0) {
        if (j < ns && p == 0) acc = (double)u[j];
    } else if (j < ns) {
        const int o = p >> 2;  // four threads per child octant
        const int32_t ch = child8[o];
        if (ch >= 0) {
            const double *M = m2m64 + (size_t)o * ns * ns + j;
            for (int k = p & 3; k < ns; k += 4) acc += M[(size_t)k * ns] * (double)u[(size_t)ch * ns + k];
        }
    }
    red[p][c] = acc;
    __syncthreads();
    if (threadIdx.x < kRootCols && j < ns) {
        double tot = 0.0;
        for (int q = 0; q < 32; ++q) tot += red[q][threadIdx.x];
        u64[j] = tot;
    }
}

__global__ void k_add_shift(int64_t n, const double *__restrict__ pshift, double4 *__restrict__ res) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) res[i].x += *pshift;
}

template <typename T>
cudaError_t evaluate_t(Plan &P, void *pot, void *grad, double *energy, cudaStream_t s) {
    using V4 = typename Vec4<T>::type;
    const int ns = P.ns;
    const T *surf = P.f64 ? (const T *)P.surf64 : (const T *)P.surf32;
    T *u = (T *)P.u_chk, *d = (T *)P.d_chk, *tmp = (T *)P.tmp_chk;
    const V4 *pts = (const V4 *)P.pts;
    double4 *res = (double4 *)P.res;
    // upward pass
    stage_begin(P, KIFMM_STAGE_P2M, s);
    if constexpr (sizeof(T) == 4)
        ++g_launches, k_p2m_f32<<<(unsigned)((P.n_leaves + kP2mLeaves - 1) / kP2mLeaves), p2m_threads(P),
                                  4 * sizeof(float) * (size_t)p2m_threads(P), s>>>(P.leaves, P.n_leaves, P.lvl,
                                                                                   P.first, P.cnt, pts, surf, ns, u);
    else
        ++g_launches, k_p2m<T><<<(unsigned)P.n_leaves, p2m_threads(P), p2m_smem<T>(P), s>>>(
                          P.leaves, P.lvl, P.first, P.cnt, pts, surf, ns, u);
    stage_end(P, KIFMM_STAGE_P2M, s);
    stage_begin(P, KIFMM_STAGE_M2M, s);
    for (int l = P.max_level - 1; l >= 0; --l)
        rows_children<T>(P, l, (const T *)P.m2m_t, u, tmp, u, 0, s);
    stage_end(P, KIFMM_STAGE_M2M, s);
    KIFMM_CUDA_TRY(cudaGetLastError());
    // interactions
    stage_begin(P, KIFMM_STAGE_M2L, s);
    KIFMM_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(T) * (size_t)P.nb * ns, s));
    const bool split_mean = !P.f64;  // FP32-based modes: d = dbar (FP64) + mean-free FP32 vector
    if (split_mean) KIFMM_CUDA_TRY(cudaMemsetAsync(P.dbar, 0, sizeof(double) * (size_t)P.nb, s));
    const bool tensor = (P.desc.precision == KIFMM_MIXED_FP16);
    if (tensor) {
        KIFMM_CUDA_TRY(m2l_tensor(P, s));
    } else {
        if constexpr (sizeof(T) == 4) {
            if (m2l_uses_simt(P)) KIFMM_CUDA_TRY(m2l_simt(P, u, d, P.dbar, s));
            else KIFMM_CUDA_TRY(m2l_exact(P, 0, u, d, 0, P.dbar, s));
        } else {
            KIFMM_CUDA_TRY(m2l_exact(P, 0, u, d, 0, nullptr, s));
        }
    }
    stage_end(P, KIFMM_STAGE_M2L, s);
    if (P.n_x > 0) {
        stage_begin(P, KIFMM_STAGE_P2L, s);
        ++g_launches, k_p2l<T><<<(unsigned)P.part_start[2][1], p2l_threads<T>(P), 0, s>>>(
                          p2m_threads(P), P.part_list[2], P.nx, P.xdense, P.lvl, P.cx, P.cy, P.cz, P.first, P.cnt, pts, surf, ns, d,
                          nullptr, 0, split_mean ? P.dbar : nullptr, nullptr, P.periodic ? P.x_sh : nullptr);
        stage_end(P, KIFMM_STAGE_P2L, s);
    }
    // the root's upward check potential in FP64 (periodic cell)
    const double *u_root = nullptr;
    if (P.periodic) {
        if constexpr (sizeof(T) == 8) {
            u_root = (const double *)u;
        } else {
            ++g_launches, k_root_up64<<<grid_for(ns, kRootCols), 32 * kRootCols, 0, s>>>(ns, P.child8, P.nchild, P.m2m64, u, P.u_root64);
            u_root = P.u_root64;
        }
        // the far images, on the root (box 0) before the downward pass
        ++g_launches, k_far_root<T><<<1, 1024, 0, s>>>(ns, P.far_t, u_root, d, split_mean ? P.dbar : nullptr);
    }
    // downward pass: per level, per octant class of the child
    stage_begin(P, KIFMM_STAGE_L2L, s);
    for (int l = 1; l <= P.max_level; ++l)
        rows_parent<T>(P, l, (const T *)P.l2l_t, d, d, s, P.op_ld, split_mean ? P.dbar : nullptr);
    stage_end(P, KIFMM_STAGE_L2L, s);
    KIFMM_CUDA_TRY(cudaGetLastError());
    // leaves: equivalent densities (two-step pseudo-inverse), then L2P + M2P + P2P
    stage_begin(P, KIFMM_STAGE_LEAF, s);
    if (P.n_w > 0) {
        rows_one<T>(P, (const T *)P.up_w_t, P.part_list[2], 0, P.part_start[2][1], u, tmp, s);
        rows_one<T>(P, (const T *)P.up_v_t, P.part_list[2], 0, P.part_start[2][1], tmp, (T *)P.up_dens, s);
    }
    rows_one<T>(P, (const T *)P.dn_w_t, P.leaves, 0, P.n_leaves, d, tmp, s);
    rows_one<T>(P, (const T *)P.dn_v_t, P.leaves, 0, P.n_leaves, tmp, (T *)P.dn_dens, s);
    stage_end(P, KIFMM_STAGE_LEAF, s);
    stage_begin(P, KIFMM_STAGE_P2P, s);
    LeafCtx C{P.lvl, P.cx, P.cy, P.cz, P.first, P.cnt, P.u_ptr, P.w_ptr, P.u_idx, P.w_idx, ns,
              split_mean ? P.dbar : nullptr, P.leaf_tile, P.status, P.periodic ? P.u_sh : nullptr,
              P.periodic ? P.w_sh : nullptr};
    // free space: the leaf pass writes the outputs itself (a periodic cell
    // adds the uniform shift to the results afterwards, then k_finalize)
    const bool fused_out = !P.periodic && (pot || grad);
    if (fused_out) {
        C.perm = P.perm;
        C.sys = P.sys;
        C.out_scale = P.out_scale;
        C.pot = pot;
        C.grad = grad;
        C.out_f64 = P.io_f64 ? 1 : 0;
    }
    const LeafW<T> W{(const T *)P.dn_dens, 1, (const T *)P.up_dens, 1, nullptr};
    if (!P.tuned_leaf && tuning_wanted(P, s)) {
        // time the default table and every candidate on this tree; keep the fastest
        float best = 1e30f;
        LeafTiling pick = P.leaf_tile;
        leaf_launch<T>(P, C, pts, surf, W, res, s);  // warm the caches first
        for (int c = -1; c < kLeafTilingCandidates; ++c) {
            LeafCtx Cc = C;
            if (c >= 0) Cc.tile = leaf_tiling_candidate(c);
            if (c >= 0 && Cc.tile.packed == C.tile.packed) continue;  // the default, timed
            float ms = 1e30f;
            for (int rep = 0; rep < 2; ++rep)  // best of two
                ms = std::min(ms, time_launch(s, [&] { leaf_launch<T>(P, Cc, pts, surf, W, res, s); }));
            if (ms < best) {
                best = ms;
                pick = Cc.tile;
            }
        }
        P.leaf_tile = pick;
        C.tile = pick;
        P.tuned_leaf = true;
    }
    leaf_launch<T>(P, C, pts, surf, W, res, s);
    if (P.periodic) {
        ++g_launches, k_moment_term<<<1, 256, 0, s>>>(P.n_leaves, P.leaf_q2, ns, P.far_g, u_root, P.pshift);
        ++g_launches, k_add_shift<<<grid_for(P.n, 256), 256, 0, s>>>(P.n, P.pshift, res);
    }
    stage_end(P, KIFMM_STAGE_P2P, s);
    KIFMM_CUDA_TRY(cudaGetLastError());
    // outputs
    stage_begin(P, KIFMM_STAGE_OUT, s);
    if ((pot || grad) && !fused_out) {
        if (P.io_f64)
            ++g_launches, k_finalize<double><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, (double *)pot,
                              (double *)grad);
        else
            ++g_launches, k_finalize<float><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, (float *)pot,
                              (float *)grad);
    }
    if (energy) {
        ++g_launches, k_energy_chunks<T><<<(unsigned)P.n_energy_chunks, 256, 0, s>>>(P.energy_chunks, res, pts,
                                                                                   P.energy_partial);
        ++g_launches, k_energy_sum<<<grid_for(P.n_sys, 64), 64, 0, s>>>(P.energy_chunk_start, P.energy_partial,
                                                                         P.lo_side, P.coef, P.n_sys, energy);
    }
    stage_end(P, KIFMM_STAGE_OUT, s);
    P.fwd_valid = P.fwd_res_valid = true;
    return cudaGetLastError();
}

// Per-particle system (the last offset at or below the caller index j).
__device__ __forceinline__ int system_of(const int64_t *__restrict__ off, int S, uint32_t j) {
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= (int64_t)j) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Adjoint weights in sorted order: ws = dL/dpot + (1/2) dL/dU_s q (the energy
// U_s = 1/2 sum q pot of the particle's system s, through its pot); with an
// energy loss the forward potential (root units) is kept for the explicit
// (1/2) dL/dU pot term of dq, since the transposed passes overwrite it.
template <typename TI, typename T>
__global__ void k_adj_weights(int64_t n, const uint32_t *__restrict__ perm, const int64_t *__restrict__ off, int S,
                              const typename Vec4<T>::type *__restrict__ pts, const TI *__restrict__ w,
                              const double *__restrict__ dLdU, const double4 *__restrict__ res, T *__restrict__ ws,
                              double *__restrict__ fwd_pot) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    double v = w ? (double)w[j] : 0.0;
    if (dLdU) {
        v += 0.5 * dLdU[system_of(off, S, j)] * (double)pts[i].w;
        fwd_pot[i] = res[i].x;
    }
    ws[i] = (T)v;
}

// dq = c1 (psi + pd) (+ 1/2 dL/dU c1 pot), dx = w_tot grad + c2 (q grad(psi + pd) + hg),
// c1 = coef / (4 pi side), c2 = c1 / side; w_tot = dL/dpot + 1/2 dL/dU q.
template <typename TO, typename T>
__global__ void k_finalize_adj(int64_t n, const double4 *__restrict__ res, const uint32_t *__restrict__ perm,
                               const int64_t *__restrict__ off, int S, const double *__restrict__ out_scale,
                               const typename Vec4<T>::type *__restrict__ pts, const TO *__restrict__ w,
                               const double *__restrict__ dLdU, const double *__restrict__ fwd_pot,
                               const double4 *__restrict__ hg, const double4 *__restrict__ pd,
                               const TO *__restrict__ grad, TO *dq, TO *dx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    const int s = system_of(off, S, j);
    const double c1 = out_scale[2 * s], c2 = out_scale[2 * s + 1];  // coef / (4 pi side), / side^2
    double4 r = res[i];
    if (pd) {
        const double4 e = pd[i];
        r.x += e.x, r.y += e.y, r.z += e.z, r.w += e.w;
    }
    const double q = (double)pts[i].w;
    const double hu = dLdU ? 0.5 * dLdU[s] : 0.0;
    if (dq) dq[j] = (TO)(c1 * r.x + (dLdU ? hu * c1 * fwd_pot[i] : 0.0));
    if (dx) {
        const double wj = (w ? (double)w[j] : 0.0) + hu * q;
        double t[3] = {c2 * q * r.y, c2 * q * r.z, c2 * q * r.w};
        if (hg) {
            const double4 h = hg[i];
            t[0] += c2 * h.x, t[1] += c2 * h.y, t[2] += c2 * h.z;
        }
        if (grad)
            for (int d = 0; d < 3; ++d) t[d] += wj * (double)grad[3 * j + d];
        dx[3 * j] = (TO)t[0];
        dx[3 * j + 1] = (TO)t[1];
        dx[3 * j + 2] = (TO)t[2];
    }
}

// Sums of many terms: FP64 as they are, FP32 compensated (two-sum of every
// term, about 48 bits), in place of FP64 sums of FP32 terms: ten of those per
// pair, conversions included, kept the FP64 unit (two lanes per clock and SM)
// busy for 2.4 ms on 100k particles.
template <typename T>
struct TermSum;
template <>
struct TermSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ double total() const { return s; }
};
template <>
struct TermSum<float> {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float x) {  // (no contraction into the term's own product)
        const float t = __fadd_rn(s, x), bb = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(x, bb)));
        s = t;
    }
    __device__ __forceinline__ double total() const { return (double)s + (double)c; }
};

// The U-list particles of leaf b, laid end to end and staged by the whole
// block, kLeafThreads at a time: load(slot, particle, ox, oy, oz) stages one
// (its leaf's centre relative to b's) and says whether it needs care, body(m,
// care) sums m staged ones, care for the whole block if one of them needs it.
template <typename T>
struct UStage {
    T ox[kLeafThreads], oy[kLeafThreads], oz[kLeafThreads];
    int first[kLeafThreads], start[kLeafThreads + 1], wsum[kLeafThreads / 32];
};
template <typename T, class Load, class Body>
__device__ __forceinline__ void for_u_sources(const LeafCtx &C, int b, UStage<T> &S, Load &&load, Body &&body) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int lb = C.lvl[b], bx = C.cx[b], by = C.cy[b], bz = C.cz[b];
    const uint32_t u0 = C.u_ptr[b];
    const int nu = (int)(C.u_ptr[b + 1] - u0);
    for (int sb = 0; sb < nu; sb += kLeafThreads) {
        __syncthreads();  // the previous batch is done with the segment arrays
        int c = 0;
        if (sb + tid < nu) {
            const int a = C.u_idx[u0 + sb + tid], la = C.lvl[a];
            S.ox[tid] = centre_diff<T>(C.cx[a], la, bx, lb);
            S.oy[tid] = centre_diff<T>(C.cy[a], la, by, lb);
            S.oz[tid] = centre_diff<T>(C.cz[a], la, bz, lb);
            S.first[tid] = C.first[a];
            c = C.cnt[a];
        }
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) S.wsum[warp] = incl;
        __syncthreads();
        for (int w = 0; w < warp; ++w) incl += S.wsum[w];
        S.start[tid + 1] = incl;
        if (tid == 0) S.start[0] = 0;
        __syncthreads();
        const int total = S.start[kLeafThreads];
        for (int c0 = 0; c0 < total; c0 += kLeafThreads) {
            __syncthreads();
            bool care = false;
            if (c0 + tid < total) {
                int lo = 0, hi = kLeafThreads;  // the last segment that starts at or before c0 + tid
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (S.start[mid] <= c0 + tid) lo = mid; else hi = mid;
                }
                care = load(tid, S.first[lo] + c0 + tid - S.start[lo], S.ox[lo], S.oy[lo], S.oz[lo]);
            }
            care = __syncthreads_or(care);
            body(min(kLeafThreads, total - c0), care);
        }
    }
}

// ---------------------------------------------------------------------------
// The Stokeslet (the tensor kernel Eq. 1 admits; Stokes flow, Sec. 2.4):
// G(r) = I / |r| + r r^T / |r|^3, the 1 / (8 pi) and coef applied at the
// output.  Sources carry forces, surfaces 3-vector densities (expansion
// vectors of 3 n_s values, point-major), targets receive velocities.  The
// same homogeneity as 1/r (degree -1), so the box-unit scalings carry over.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void stokes_acc(T rx, T ry, T rz, T fx, T fy, T fz, T &ux, T &uy, T &uz) {
    const T ri = rsqrt_t<T>(rx * rx + ry * ry + rz * rz);
    const T rf = (rx * fx + ry * fy + rz * fz) * (ri * ri * ri);
    ux += fx * ri + rx * rf;
    uy += fy * ri + ry * rf;
    uz += fz * ri + rz * rf;
}

// P2M: u(b)_{3j+a} = sum_i G_a.(UC_j - x_i) f_i, box units then 1/h; one
// block per leaf, a thread per check point, forces staged through shared memory.
template <typename T>
__global__ void k_p2m_stokes(const int32_t *__restrict__ leaves, const int32_t *__restrict__ lvl,
                             const int32_t *__restrict__ first, const int32_t *__restrict__ cnt,
                             const typename Vec4<T>::type *__restrict__ pts, const T *__restrict__ frc,
                             const T *__restrict__ surf, int npt, T *__restrict__ u) {
    __shared__ T sx[kLeafThreads], sy[kLeafThreads], sz[kLeafThreads], sfx[kLeafThreads], sfy[kLeafThreads],
        sfz[kLeafThreads];
    const int b = leaves[blockIdx.x];
    const T h = box_half<T>(lvl[b]), hinv = T(1) / h;
    const int n = cnt[b], f = first[b];
    const T a = (T)kAlphaOuter;
    for (int j0 = 0; j0 < npt; j0 += blockDim.x) {
        const int j = j0 + threadIdx.x;
        T px = 0, py = 0, pz = 0, ux = 0, uy = 0, uz = 0;
        if (j < npt) px = a * surf[3 * j], py = a * surf[3 * j + 1], pz = a * surf[3 * j + 2];
        for (int c0 = 0; c0 < n; c0 += kLeafThreads) {
            __syncthreads();
            for (int k = threadIdx.x; k < kLeafThreads && c0 + k < n; k += blockDim.x) {
                const auto v = pts[f + c0 + k];
                sx[k] = v.x * hinv, sy[k] = v.y * hinv, sz[k] = v.z * hinv;
                const size_t o = 3 * (size_t)(f + c0 + k);
                sfx[k] = frc[o], sfy[k] = frc[o + 1], sfz[k] = frc[o + 2];
            }
            __syncthreads();
            const int m = min(kLeafThreads, n - c0);
            for (int i = 0; i < m; ++i) stokes_acc<T>(px - sx[i], py - sy[i], pz - sz[i], sfx[i], sfy[i], sfz[i], ux, uy, uz);
        }
        if (j < npt) {
            T *o = u + (size_t)b * 3 * npt + 3 * j;
            o[0] = ux * hinv, o[1] = uy * hinv, o[2] = uz * hinv;
        }
    }
}

// P2L: d(b) += the forces of the leaves of X(b) on b's downward check surface.
template <typename T>
__global__ void k_p2l_stokes(const int32_t *__restrict__ boxes, const int32_t *__restrict__ nx, const int32_t *__restrict__ xdense,
                             const int32_t *__restrict__ lvl, const int32_t *__restrict__ cx,
                             const int32_t *__restrict__ cy, const int32_t *__restrict__ cz,
                             const int32_t *__restrict__ first, const int32_t *__restrict__ cnt,
                             const typename Vec4<T>::type *__restrict__ pts, const T *__restrict__ frc,
                             const T *__restrict__ surf, int npt, T *__restrict__ d) {
    __shared__ T sx[kLeafThreads], sy[kLeafThreads], sz[kLeafThreads], sfx[kLeafThreads], sfy[kLeafThreads],
        sfz[kLeafThreads];
    const int b = boxes[blockIdx.x];
    const int lb = lvl[b];
    const T hb = box_half<T>(lb), hinv = T(1) / hb;
    const T al = (T)kAlphaInner;
    for (int j0 = 0; j0 < npt; j0 += blockDim.x) {
        const int j = j0 + threadIdx.x;
        T px = 0, py = 0, pz = 0, ux = 0, uy = 0, uz = 0;
        if (j < npt) px = al * surf[3 * j], py = al * surf[3 * j + 1], pz = al * surf[3 * j + 2];
        for (int e = 0; e < nx[b]; ++e) {
            const int a = xdense[(size_t)b * kMaxCoarse + e], la = lvl[a];
            const T ox = centre_diff<T>(cx[a], la, cx[b], lb), oy = centre_diff<T>(cy[a], la, cy[b], lb),
                    oz = centre_diff<T>(cz[a], la, cz[b], lb);
            const int n = cnt[a], f = first[a];
            for (int c0 = 0; c0 < n; c0 += kLeafThreads) {
                __syncthreads();
                for (int k = threadIdx.x; k < kLeafThreads && c0 + k < n; k += blockDim.x) {
                    const auto v = pts[f + c0 + k];
                    sx[k] = (ox + v.x) * hinv, sy[k] = (oy + v.y) * hinv, sz[k] = (oz + v.z) * hinv;
                    const size_t o = 3 * (size_t)(f + c0 + k);
                    sfx[k] = frc[o], sfy[k] = frc[o + 1], sfz[k] = frc[o + 2];
                }
                __syncthreads();
                const int m = min(kLeafThreads, n - c0);
                for (int i = 0; i < m; ++i)
                    stokes_acc<T>(px - sx[i], py - sy[i], pz - sz[i], sfx[i], sfy[i], sfz[i], ux, uy, uz);
            }
        }
        if (j < npt) {
            T *o = d + (size_t)b * 3 * npt + 3 * j;
            o[0] += ux * hinv, o[1] += uy * hinv, o[2] += uz * hinv;
        }
    }
}

// Leaves: L2P (own downward density on the 2.95 h_b surface), M2P (the W
// boxes' upward densities on their 1.05 h_a surfaces) and P2P (the U-list
// particles' forces, r = 0 skipped); root units; one block per leaf, up to 32
// targets at a time with the sources dealt out to its warps and lane groups as
// in k_adj_leaf.
template <typename T>
__global__ void __launch_bounds__(kLeafThreads) k_leaf_stokes(LeafCtx C, const int32_t *__restrict__ leaves,
                                                              const typename Vec4<T>::type *__restrict__ pts,
                                                              const T *__restrict__ frc, const T *__restrict__ surf,
                                                              int npt, const T *__restrict__ dn_dens,
                                                              const T *__restrict__ up_dens, double4 *__restrict__ res) {
    using V4 = typename Vec4<T>::type;
    __shared__ V4 src[kLeafThreads], sf[kLeafThreads];
    __shared__ UStage<T> U;
    __shared__ double red[kLeafThreads / 32 - 1][3][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = leaves[blockIdx.x];
    const int lb = C.lvl[b], bx = C.cx[b], by = C.cy[b], bz = C.cz[b], n = C.cnt[b], f = C.first[b];
    const T hb = box_half<T>(lb);
    const uint32_t w0 = C.w_ptr[b];
    const int nw = (int)(C.w_ptr[b + 1] - w0);
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int rest = min(32, n - t0);
        const int ng = rest <= 8 ? 4 : (rest <= 16 ? 2 : 1), lg = 32 / ng;  // lane groups, lanes per group
        const int grp = lane / lg, i = t0 + lane - grp * lg;
        const bool valid = i < n;
        T x = 0, y = 0, z = 0;
        if (valid) {
            const V4 v = pts[f + i];
            x = v.x, y = v.y, z = v.z;
        }
        TermSum<T> vx, vy, vz;
        const int k_first = warp * ng + grp, k_step = ng * (kLeafThreads / 32);
        auto add = [&](T rx, T ry, T rz, const V4 &w) {
            const T r2 = rx * rx + ry * ry + rz * rz;
            // the particle itself and coincident points add nothing
            const T ri = r2 > T(0) ? rsqrt_t<T>(r2) : T(0);
            const T rf = (rx * w.x + ry * w.y + rz * w.z) * (ri * ri * ri);
            vx.add(w.x * ri + rx * rf);
            vy.add(w.y * ri + ry * rf);
            vz.add(w.z * ri + rz * rf);
        };
        auto sum = [&](int m) {
            for (int k = k_first; k < m; k += k_step) {
                const V4 v = src[k];
                add(x - v.x, y - v.y, z - v.z, sf[k]);
            }
        };
        // a surface of forces: points o + r S_k, forces h wts[3 k ..]
        auto surface = [&](T ox, T oy, T oz, T r, const T *wts, T h) {
            for (int c0 = 0; c0 < npt; c0 += kLeafThreads) {
                __syncthreads();
                const int k = c0 + tid;
                if (k < npt) {
                    V4 v, w;
                    v.x = ox + r * surf[3 * k], v.y = oy + r * surf[3 * k + 1], v.z = oz + r * surf[3 * k + 2], v.w = T(0);
                    w.x = wts[3 * k] * h, w.y = wts[3 * k + 1] * h, w.z = wts[3 * k + 2] * h, w.w = T(0);
                    src[tid] = v;
                    sf[tid] = w;
                }
                __syncthreads();
                sum(min(kLeafThreads, npt - c0));
            }
        };
        surface(T(0), T(0), T(0), (T)kAlphaOuter * hb, dn_dens + (size_t)b * 3 * npt, hb);
        for (int e = 0; e < nw; ++e) {
            const int a = C.w_idx[w0 + e], la = C.lvl[a];
            const T ha = box_half<T>(la);
            surface(centre_diff<T>(C.cx[a], la, bx, lb), centre_diff<T>(C.cy[a], la, by, lb),
                    centre_diff<T>(C.cz[a], la, bz, lb), (T)kAlphaInner * ha, up_dens + (size_t)a * 3 * npt, ha);
        }
        for_u_sources<T>(
            C, b, U,
            [&](int slot, int j, T ox, T oy, T oz) {
                const V4 v = pts[j];
                V4 p, w;
                p.x = ox + v.x, p.y = oy + v.y, p.z = oz + v.z, p.w = T(0);
                w.x = frc[3 * (size_t)j], w.y = frc[3 * (size_t)j + 1], w.z = frc[3 * (size_t)j + 2], w.w = T(0);
                src[slot] = p;
                sf[slot] = w;
                return false;
            },
            [&](int m, bool) { sum(m); });
        // lane groups, then warps, in order
        double tot[3] = {vx.total(), vy.total(), vz.total()};
#pragma unroll
        for (int q = 0; q < 3; ++q)
            for (int o = 16; o >= lg; o >>= 1) tot[q] += __shfl_xor_sync(0xffffffffu, tot[q], o);
        if (warp > 0) {
#pragma unroll
            for (int q = 0; q < 3; ++q) red[warp - 1][q][lane] = tot[q];
        }
        __syncthreads();
        if (warp == 0 && grp == 0 && valid) {
            for (int w = 0; w < kLeafThreads / 32 - 1; ++w)
#pragma unroll
                for (int q = 0; q < 3; ++q) tot[q] += red[w][q][lane];
            res[f + i] = make_double4(tot[0], tot[1], tot[2], 0.0);
            if (!isfinite(tot[0] + tot[1] + tot[2])) set_status(C.status, KIFMM_ERR_NONFINITE);
        }
    }
}

// Velocities in the caller's order: coef / (8 pi side) times the root-unit sums.
template <typename TO>
__global__ void k_finalize_stokes(int64_t n, const double4 *__restrict__ res, const uint32_t *__restrict__ perm,
                                  const int64_t *__restrict__ off, int S, const double *__restrict__ out_scale,
                                  TO *__restrict__ vel) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= (int64_t)j) lo = mid; else hi = mid - 1;
    }
    const double c = 0.5 * out_scale[2 * lo];  // coef / (4 pi side) / 2
    const double4 r = res[i];
    vel[3 * (size_t)j] = (TO)(c * r.x);
    vel[3 * (size_t)j + 1] = (TO)(c * r.y);
    vel[3 * (size_t)j + 2] = (TO)(c * r.z);
}

template <typename T>
cudaError_t evaluate_stokes_t(Plan &P, void *vel, cudaStream_t s) {
    using V4 = typename Vec4<T>::type;
    const int ns = P.ns, npt = P.nsurf;
    const T *surf = P.f64 ? (const T *)P.surf64 : (const T *)P.surf32;
    T *u = (T *)P.u_chk, *d = (T *)P.d_chk, *tmp = (T *)P.tmp_chk;
    const V4 *pts = (const V4 *)P.pts;
    const T *frc = (const T *)P.frc;
    double4 *res = (double4 *)P.res;
    const unsigned thr = (unsigned)std::min(kLeafThreads, (npt + 31) / 32 * 32);
    stage_begin(P, KIFMM_STAGE_P2M, s);
    ++g_launches, k_p2m_stokes<T><<<(unsigned)P.n_leaves, thr, 0, s>>>(P.leaves, P.lvl, P.first, P.cnt, pts, frc,
                                                                       surf, npt, u);
    stage_end(P, KIFMM_STAGE_P2M, s);
    stage_begin(P, KIFMM_STAGE_M2M, s);
    for (int l = P.max_level - 1; l >= 0; --l)
        rows_children<T>(P, l, (const T *)P.m2m_t, u, tmp, u, 0, s);
    stage_end(P, KIFMM_STAGE_M2M, s);
    stage_begin(P, KIFMM_STAGE_M2L, s);
    KIFMM_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(T) * (size_t)P.nb * ns, s));
    if constexpr (sizeof(T) == 4) KIFMM_CUDA_TRY(m2l_simt(P, u, d, nullptr, s));
    else KIFMM_CUDA_TRY(m2l_exact(P, 0, u, d, 0, nullptr, s));
    stage_end(P, KIFMM_STAGE_M2L, s);
    if (P.n_x > 0) {
        stage_begin(P, KIFMM_STAGE_P2L, s);
        ++g_launches, k_p2l_stokes<T><<<(unsigned)P.part_start[2][1], thr, 0, s>>>(P.part_list[2], P.nx, P.xdense, P.lvl, P.cx, P.cy, P.cz,
                                                                       P.first, P.cnt, pts, frc, surf, npt, d);
        stage_end(P, KIFMM_STAGE_P2L, s);
    }
    stage_begin(P, KIFMM_STAGE_L2L, s);
    for (int l = 1; l <= P.max_level; ++l)
        rows_parent<T>(P, l, (const T *)P.l2l_t, d, d, s);
    stage_end(P, KIFMM_STAGE_L2L, s);
    KIFMM_CUDA_TRY(cudaGetLastError());
    stage_begin(P, KIFMM_STAGE_LEAF, s);
    if (P.n_w > 0) {
        rows_one<T>(P, (const T *)P.up_w_t, P.part_list[2], 0, P.part_start[2][1], u, tmp, s);
        rows_one<T>(P, (const T *)P.up_v_t, P.part_list[2], 0, P.part_start[2][1], tmp, (T *)P.up_dens, s);
    }
    rows_one<T>(P, (const T *)P.dn_w_t, P.leaves, 0, P.n_leaves, d, tmp, s);
    rows_one<T>(P, (const T *)P.dn_v_t, P.leaves, 0, P.n_leaves, tmp, (T *)P.dn_dens, s);
    stage_end(P, KIFMM_STAGE_LEAF, s);
    stage_begin(P, KIFMM_STAGE_P2P, s);
    LeafCtx C{P.lvl, P.cx, P.cy, P.cz, P.first, P.cnt, P.u_ptr, P.w_ptr, P.u_idx, P.w_idx, ns, nullptr,
              P.leaf_tile, P.status, nullptr, nullptr};
    ++g_launches, k_leaf_stokes<T><<<(unsigned)P.n_leaves, kLeafThreads, 0, s>>>(
                      C, P.leaves, pts, frc, surf, npt, (const T *)P.dn_dens, (const T *)P.up_dens, res);
    stage_end(P, KIFMM_STAGE_P2P, s);
    stage_begin(P, KIFMM_STAGE_OUT, s);
    if (vel) {
        if (P.io_f64)
            ++g_launches, k_finalize_stokes<double><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, (double *)vel);
        else
            ++g_launches, k_finalize_stokes<float><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, (float *)vel);
    }
    stage_end(P, KIFMM_STAGE_OUT, s);
    P.fwd_valid = P.fwd_res_valid = true;
    return cudaGetLastError();
}


// Weights of a loss on the gradient, in sorted order and root units: the
// caller's dL/dgrad divided by the side of the particle's system (the
// gradient in caller units is the root-unit gradient over the side).
template <typename TI, typename T>
__global__ void k_gather_g(int64_t n, const uint32_t *__restrict__ perm, const int64_t *__restrict__ off, int S,
                           const double *__restrict__ lo_side, const TI *__restrict__ g, T *__restrict__ gs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t j = perm[i];
    int lo = 0, hi = S - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= (int64_t)j) lo = mid; else hi = mid - 1;
    }
    const double side = lo_side[4 * lo + 3];
#pragma unroll
    for (int d = 0; d < 3; ++d) gs[3 * i + d] = (T)((double)g[3 * j + d] / side);
}

// The leaf-level terms of a loss on the gradient, one block per leaf b, root
// units:
//  hg[i]  = H_i g_i, the Hessian of the forward field at particle i applied
//           to its own dipole (the gradient's dependence on the particle's
//           position), from b's forward sources: its downward equivalent
//           density on the 2.95 h_b surface, the upward densities of its W
//           boxes on their 1.05 h_a surfaces, and the U-list particles;
//  pd[i]  = (psi, grad psi) at particle i of the dipoles g_j of the U-list
//           particles j != i (the near field of the transposed gradient).
// With H = grad grad (1/r), r = x_i - y:  H g = (3 (r.g) r - r^2 g) / r^5;
// a dipole g at y gives psi(x) = g . r / r^3, grad psi = g / r^3 - 3 (g.r) r / r^5.
//
// Some 85 FP32 operations per pair bound it.  Up to 32 targets at a time, one
// per lane of every warp (8 or 16 targets: four or two lanes each), so that a
// leaf of 24 uses all four warps: the sources (surfaces; then the U list's
// particles laid end to end) are staged 128 at a time and dealt out to the
// warps and lane groups, whose sums are added in order at the end.
template <typename T>
__global__ void __launch_bounds__(kLeafThreads, sizeof(T) == 8 ? 5 : 8)
    k_adj_leaf(LeafCtx C, const int32_t *__restrict__ leaves, const typename Vec4<T>::type *__restrict__ pts,
               const T *__restrict__ surf, const T *__restrict__ dn_dens, const T *__restrict__ up_dens,
               const T *__restrict__ gs, double4 *__restrict__ hg, double4 *__restrict__ pd) {
    using V4 = typename Vec4<T>::type;
    __shared__ V4 src[kLeafThreads], dip[kLeafThreads];
    __shared__ UStage<T> U;
    __shared__ double red[kLeafThreads / 32 - 1][7][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = leaves[blockIdx.x];
    const int lb = C.lvl[b], bx = C.cx[b], by = C.cy[b], bz = C.cz[b], n = C.cnt[b], f = C.first[b], ns = C.ns;
    const T hb = box_half<T>(lb);
    const uint32_t w0 = C.w_ptr[b];
    const int nw = (int)(C.w_ptr[b + 1] - w0);
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int rest = min(32, n - t0);
        const int ng = rest <= 8 ? 4 : (rest <= 16 ? 2 : 1), lg = 32 / ng;  // lane groups, lanes per group
        const int grp = lane / lg, i = t0 + lane - grp * lg;
        const bool valid = i < n;
        T x = 0, y = 0, z = 0, g0 = 0, g1 = 0, g2 = 0;
        if (valid) {
            const V4 v = pts[f + i];
            x = v.x, y = v.y, z = v.z;
            g0 = gs[3 * (size_t)(f + i)], g1 = gs[3 * (size_t)(f + i) + 1], g2 = gs[3 * (size_t)(f + i) + 2];
        }
        TermSum<T> h0, h1, h2, p0, p1, p2, p3;
        const int k_first = warp * ng + grp, k_step = ng * (kLeafThreads / 32);
        // Hessian of one monopole w at offset r = x_i - y, applied to a dipole
        auto hess = [&](T rx, T ry, T rz, T w, T ri2, T ri3, T d0, T d1, T d2) {
            const T rg3 = T(3) * (rx * d0 + ry * d1 + rz * d2) * ri2;
            h0.add(w * ri3 * (rg3 * rx - d0));
            h1.add(w * ri3 * (rg3 * ry - d1));
            h2.add(w * ri3 * (rg3 * rz - d2));
        };
        // a surface of monopoles: points o + r S_k, weights h wts[k]
        auto surface = [&](T ox, T oy, T oz, T r, const T *wts, T h) {
            for (int c0 = 0; c0 < ns; c0 += kLeafThreads) {
                __syncthreads();
                if (c0 + tid < ns) {
                    V4 v;
                    v.x = ox + r * surf[3 * (c0 + tid)];
                    v.y = oy + r * surf[3 * (c0 + tid) + 1];
                    v.z = oz + r * surf[3 * (c0 + tid) + 2];
                    v.w = wts[c0 + tid] * h;
                    src[tid] = v;
                }
                __syncthreads();
                const int m = min(kLeafThreads, ns - c0);
                for (int k = k_first; k < m; k += k_step) {
                    const V4 v = src[k];
                    const T rx = x - v.x, ry = y - v.y, rz = z - v.z;
                    const T ri = rsqrt_t<T>(rx * rx + ry * ry + rz * rz), ri2 = ri * ri;
                    hess(rx, ry, rz, v.w, ri2, ri * ri2, g0, g1, g2);
                }
            }
        };
        // m staged particles; the particle itself and coincident points add
        // nothing, by a zero weight.  Where a dipole is not finite (care) the
        // pair's dipoles are zero as well, since zero times them would be NaN.
        // (Leaving the pair out by a branch: 270 -> 295 us on 100k particles.)
        auto near_field = [&](int m, auto care) {
            for (int k = k_first; k < m; k += k_step) {
                const V4 v = src[k];
                V4 d = dip[k];
                const T rx = x - v.x, ry = y - v.y, rz = z - v.z;
                const T r2 = rx * rx + ry * ry + rz * rz;
                const T ri = r2 > T(0) ? rsqrt_t<T>(r2) : T(0), ri2 = ri * ri, ri3 = ri * ri2;
                T d0 = g0, d1 = g1, d2 = g2;
                if (decltype(care)::value && !(r2 > T(0))) d0 = d1 = d2 = d.x = d.y = d.z = T(0);
                hess(rx, ry, rz, v.w, ri2, ri3, d0, d1, d2);
                const T gr = d.x * rx + d.y * ry + d.z * rz;
                const T gr3 = T(3) * gr * ri2;
                p0.add(gr * ri3);
                p1.add(ri3 * (d.x - gr3 * rx));
                p2.add(ri3 * (d.y - gr3 * ry));
                p3.add(ri3 * (d.z - gr3 * rz));
            }
        };
        const bool odd = __syncthreads_or(!isfinite(g0 + g1 + g2));  // some target's dipole
        // own downward equivalent surface (weights dn_dens h_b), then the W
        // boxes' upward equivalent surfaces (weights up_dens h_a)
        surface(T(0), T(0), T(0), (T)kAlphaOuter * hb, dn_dens + (size_t)b * ns, hb);
        for (int e = 0; e < nw; ++e) {
            const int a_ = C.w_idx[w0 + e], la = C.lvl[a_];
            const T ha = box_half<T>(la);
            surface(centre_diff<T>(C.cx[a_], la, bx, lb), centre_diff<T>(C.cy[a_], la, by, lb),
                    centre_diff<T>(C.cz[a_], la, bz, lb), (T)kAlphaInner * ha, up_dens + (size_t)a_ * ns, ha);
        }
        for_u_sources<T>(
            C, b, U,
            [&](int slot, int j, T ox, T oy, T oz) {
                const V4 v = pts[j];
                V4 p, d;
                p.x = ox + v.x, p.y = oy + v.y, p.z = oz + v.z, p.w = v.w;
                d.x = gs[3 * (size_t)j], d.y = gs[3 * (size_t)j + 1], d.z = gs[3 * (size_t)j + 2], d.w = T(0);
                src[slot] = p;
                dip[slot] = d;
                return !isfinite(d.x + d.y + d.z);
            },
            [&](int m, bool care) {
                if (sizeof(T) == 8 || care || odd) near_field(m, std::true_type{});
                else near_field(m, std::false_type{});
            });
        // lane groups, then warps, in order
        double tot[7] = {h0.total(), h1.total(), h2.total(), p0.total(), p1.total(), p2.total(), p3.total()};
#pragma unroll
        for (int q = 0; q < 7; ++q)
            for (int o = 16; o >= lg; o >>= 1) tot[q] += __shfl_xor_sync(0xffffffffu, tot[q], o);
        if (warp > 0)
#pragma unroll
            for (int q = 0; q < 7; ++q) red[warp - 1][q][lane] = tot[q];
        __syncthreads();
        if (warp == 0 && grp == 0 && valid) {
            for (int w = 0; w < kLeafThreads / 32 - 1; ++w)
#pragma unroll
                for (int q = 0; q < 7; ++q) tot[q] += red[w][q][lane];
            hg[f + i] = make_double4(tot[0], tot[1], tot[2], 0.0);
            pd[f + i] = make_double4(tot[3], tot[4], tot[5], tot[6]);
        }
    }
}

// Transposed passes with the tree frozen: psi = A^T w (Sec. 2.2 operators,
// transposed in reverse order), then the adjoint outputs.
template <typename T>
cudaError_t backward_t(Plan &P, const void *w_user, const void *g_user, const double *dLdU, const void *grad_user,
                       void *dq, void *dx, cudaStream_t s) {
    using V4 = typename Vec4<T>::type;
    const int ns = P.ns;
    const int64_t blk = op_block(ns, ns);
    const T *surf = P.f64 ? (const T *)P.surf64 : (const T *)P.surf32;
    T *ub = (T *)P.u_chk, *db = (T *)P.d_chk, *tmp = (T *)P.tmp_chk;
    // scratch of their own: the forward's equivalent densities stay intact
    // (the Hessian term reads them, and a second backward may follow)
    T *e1 = (T *)P.adj_e1, *e2 = (T *)P.adj_e2, *ws = (T *)P.w_sorted;
    T *gs = g_user ? (T *)P.g_sorted : nullptr;
    const T *adjp = (const T *)P.adj_pinv;
    const V4 *pts = (const V4 *)P.pts;
    double4 *res = (double4 *)P.res;
    double4 *hg = g_user ? (double4 *)P.adj_hg : nullptr, *pd = g_user ? (double4 *)P.adj_pd : nullptr;
    double *fwd_pot = dLdU ? P.adj_pot : nullptr;
    if (P.io_f64)
        ++g_launches, k_adj_weights<double, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                          P.n, P.perm, P.sys_off_d, P.n_sys, pts, (const double *)w_user, dLdU, res, ws, fwd_pot);
    else
        ++g_launches, k_adj_weights<float, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                          P.n, P.perm, P.sys_off_d, P.n_sys, pts, (const float *)w_user, dLdU, res, ws, fwd_pot);
    LeafCtx C{P.lvl, P.cx, P.cy, P.cz, P.first, P.cnt, P.u_ptr, P.w_ptr, P.u_idx, P.w_idx, ns, nullptr,
              P.leaf_tile, P.status, nullptr, nullptr};
    if (g_user) {
        if (P.io_f64)
            ++g_launches, k_gather_g<double, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, P.perm, P.sys_off_d, P.n_sys, P.lo_side, (const double *)g_user, gs);
        else
            ++g_launches, k_gather_g<float, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                              P.n, P.perm, P.sys_off_d, P.n_sys, P.lo_side, (const float *)g_user, gs);
        // the forward field's Hessian term and the dipoles' near field (reads
        // the last evaluate's equivalent densities)
        ++g_launches, k_adj_leaf<T><<<(unsigned)P.n_leaves, kLeafThreads, 0, s>>>(
                          C, P.leaves, pts, surf, (const T *)P.dn_dens, (const T *)P.up_dens, gs, hg, pd);
    }
    // L2P^T: h * sum w / |DE - x| (+ the dipoles) at each leaf, then d-bar = W_dn^T V_dn^T (.)
    KIFMM_CUDA_TRY(cudaMemsetAsync(db, 0, sizeof(T) * (size_t)P.nb * ns, s));
    KIFMM_CUDA_TRY(cudaMemsetAsync(ub, 0, sizeof(T) * (size_t)P.nb * ns, s));
    ++g_launches, k_p2m<T><<<(unsigned)P.n_leaves, p2m_threads(P), p2m_smem<T>(P), s>>>(P.leaves, P.lvl, P.first, P.cnt, pts, surf,
                                                                        ns, e1, ws, 1, gs);
    rows_one<T>(P, adjp + 3 * blk, P.leaves, 0, P.n_leaves, e1, tmp, s);
    rows_one<T>(P, adjp + 2 * blk, P.leaves, 0, P.n_leaves, tmp, db, s);
    // M2P^T: W-list sources a receive h_a * sum w / |UE_a - x| (+ dipoles) from the leaves of X(a)
    if (P.n_x > 0) {
        KIFMM_CUDA_TRY(cudaMemsetAsync(e2, 0, sizeof(T) * (size_t)P.nb * ns, s));
        ++g_launches, k_p2l<T><<<(unsigned)P.part_start[2][1], p2l_threads<T>(P), 0, s>>>(
                          p2m_threads(P), P.part_list[2], P.nx, P.xdense, P.lvl, P.cx, P.cy, P.cz, P.first, P.cnt, pts, surf, ns, e2,
                          ws, 1, nullptr, gs);
        rows_one<T>(P, adjp + 1 * blk, P.part_list[2], 0, P.part_start[2][1], e2, tmp, s);
        rows_one<T>(P, adjp, P.part_list[2], 0, P.part_start[2][1], tmp, ub, s);
    }
    // L2L^T, bottom-up
    for (int l = P.max_level - 1; l >= 0; --l)
        rows_children<T>(P, l, (const T *)P.adj_l2l, db, tmp, db, 1, s);
    // M2L^T (V lists are symmetric; operator at the negated offset, transposed)
    KIFMM_CUDA_TRY(m2l_exact(P, 1, db, ub, 1, nullptr, s));
    // M2M^T, top-down
    for (int l = 1; l <= P.max_level; ++l)
        rows_parent<T>(P, l, (const T *)P.adj_m2m, ub, ub, s);
    // P2M^T (own UC surface, u-bar), P2L^T (W boxes' DC surfaces, d-bar), P2P^T (weights w)
    const LeafW<T> W{ub, 0, db, 0, ws};
    leaf_launch<T>(P, C, pts, surf, W, res, s);
    if (P.io_f64)
        ++g_launches, k_finalize_adj<double, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                          P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, pts, (const double *)w_user, dLdU,
                          fwd_pot, hg, pd, (const double *)grad_user, (double *)dq, (double *)dx);
    else
        ++g_launches, k_finalize_adj<float, T><<<grid_for(P.n, 256), 256, 0, s>>>(
                          P.n, res, P.perm, P.sys_off_d, P.n_sys, P.out_scale, pts, (const float *)w_user, dLdU,
                          fwd_pot, hg, pd, (const float *)grad_user, (float *)dq, (float *)dx);
    P.fwd_res_valid = false;  // res now holds the adjoint field
    return cudaGetLastError();
}

}  // namespace

cudaError_t rows_setup() {
    const auto dyn = cudaFuncAttributeMaxDynamicSharedMemorySize;
    // the longest rows: FP32 the Stokeslet's at p = 8; FP64 those whose tile fits
    const int f32 = (int)rows_small_smem<float>(gemm_nkp(3 * (6 * 7 * 7 + 2)));
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_rows_small<double, true, 4>, dyn, kRowsSmallMax));
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_rows_small<double, true, 1>, dyn, kRowsSmallMax));
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_rows_small<float, true, 4>, dyn, f32));
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_rows_small<float, true, 1>, dyn, f32));
    KIFMM_CUDA_TRY(cudaFuncSetAttribute(k_rows_small<float, false, 4>, dyn, f32));
    return cudaFuncSetAttribute(k_rows_small<float, false, 1>, dyn, f32);
}

cudaError_t run_backward(Plan &P, const void *w, const void *g, const double *dLdU, const void *grad, void *dq,
                         void *dx, cudaStream_t s) {
    return P.f64 ? backward_t<double>(P, w, g, dLdU, grad, dq, dx, s)
                 : backward_t<float>(P, w, g, dLdU, grad, dq, dx, s);
}

cudaError_t run_evaluate(Plan &P, void *pot, void *grad, double *energy, cudaStream_t s) {
    if (P.stokes) return P.f64 ? evaluate_stokes_t<double>(P, pot, s) : evaluate_stokes_t<float>(P, pot, s);
    return P.f64 ? evaluate_t<double>(P, pot, grad, energy, s) : evaluate_t<float>(P, pot, grad, energy, s);
}

cudaError_t run_clump_reduce(Plan &P, int64_t n_clumps, const int64_t *offs, const void *xyz, const void *q,
                             const void *grad, const void *ref, void *force, void *torque, cudaStream_t s) {
    if (n_clumps == 0) return cudaSuccess;
    if (P.io_f64)
        ++g_launches, k_clump<double><<<grid_for(n_clumps, 128), 128, 0, s>>>(n_clumps, offs, (const double *)xyz, (const double *)q,
                                                               (const double *)grad, (const double *)ref,
                                                               (double *)force, (double *)torque);
    else
        ++g_launches, k_clump<float><<<grid_for(n_clumps, 128), 128, 0, s>>>(n_clumps, offs, (const float *)xyz, (const float *)q,
                                                              (const float *)grad, (const float *)ref,
                                                              (float *)force, (float *)torque);
    return cudaGetLastError();
}

}  // namespace kifmm
