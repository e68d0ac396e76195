// batched.cu -- singular values of many small matrices of uneven shapes in one
// persistent launch (the batched form of the method of Section 5.1.1).
//
//  1. prep kernel (one block): orders the batch by (class, cost), most expensive first
//     (a counting sort), so that blocks draw similar matrices together and the long ones
//     start first.  Everything stays on the device, so the whole call can be captured into a
//     CUDA graph.
//  2. persistent kernel (one block of 16 warps per SM): each block takes units of work from an
//     atomic counter; a unit is one matrix for all 16 warps, two for 8 warps each, four for 4,
//     or sixteen for one warp each, by the classes below.
//
// A matrix (or its transpose, M >= N) lives in the registers of its warps: lane l of
// warp w holds rows l, l + 32, ... of columns w, w + NW, ... .
//   - M beyond the rows the registers hold: R of the QR factorisation first, by chunks of rows.
//     R (packed, shared memory) and a chunk are reduced to the next R column by column; a column
//     belongs to one warp, so a step is: the owner publishes column j, one barrier, every warp
//     forms its dot products, reduces them over its lanes and updates its columns.
//   - One-stage Householder bidiagonalisation of the register tile (band width 1: the band stage
//     degenerates for these sizes): the left reflector as above; the right one needs each row's
//     sum over the warps (two barriers).
//   - The bidiagonal's values by multisection on Sturm counts (FP32; sturm.cuh), with all
//     threads of the matrix.
// Columns are taken in order k NW + w0 with k unrolled, so that register indices are
// constants, finished columns and rows drop out of the loops, and the code of one k serves NW
// columns.
//
// What bounds it: the chain of a column (one to three barriers and a reduction over the lanes,
// about 700 cycles) for the small classes, multiply-add issue for the large ones.  Before, the
// matrix lived in shared memory or, above 48K elements, in global memory, and every reflector
// streamed it twice.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <utility>

#include "../../include/nla.h"
#include "common.cuh"
#include "house.cuh"
#include "kernels.cuh"
#include "sturm.cuh"
#include "trace.h"
#include "tuned.h"

namespace {

constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kBuckets = 5;      // size buckets of the tuned table, by element count
constexpr int kBucketElems = 48 * 1024;
constexpr int kClasses = 5;      // 0: N <= 256, 1: N <= 192 (16 warps), 2: N <= 128 (8), 3: N <= 64 (4), 4: N <= 32 (1)
constexpr int kCostBins = 128;   // per class, quarters of a power of two of the cost

// Least threads per matrix for each size bucket (the tuned table's group sizes): a matrix is
// given to the smallest class that holds its N and has as many threads.
struct BatchCfg {
    int group[kBuckets];
};

nla_status berr(nla_status s, const char *m) {
    nla_set_last_error(m);
    return s;
}

__host__ __device__ inline int class_warps(int c) { return c <= 1 ? 16 : c == 2 ? 8 : c == 3 ? 4 : 1; }

__device__ int class_of(long m, long n, const BatchCfg &cfg) {
    const long N = min(m, n), elems = m * n;
    int b = 0;
    while (b < kBuckets - 1 && elems > (long)kBucketElems >> (kBuckets - 2 - b)) ++b;
    const int by_n = N > 192 ? 0 : N > 128 ? 1 : N > 64 ? 2 : N > 32 ? 3 : 4;
    int c = 4;
    while (c > 1 && (c > by_n || 32 * class_warps(c) < cfg.group[b])) --c;
    return min(c, by_n);
}

// ---------------------------------------------------------------- prep
__global__ void batched_prep_kernel(int batch, const int *dM, const int *dN, int *order, unsigned int *ctl, BatchCfg cfg) {
    __shared__ unsigned int bins[kClasses * kCostBins];
    const int tid = threadIdx.x, nt = blockDim.x;
    const auto bin_of = [&](int i) {
        const long m = max(dM[i], 0), n = max(dN[i], 0), N = min(m, n);
        // flops to within the ordering's needs; +1: empty matrices come last
        const float cost = (float)(m * n) * (float)N + 1.f;
        return class_of(m, n, cfg) * kCostBins + kCostBins - 1 - min(kCostBins - 1, (int)(4.f * __log2f(cost)));
    };
    for (int i = tid; i < kClasses * kCostBins; i += nt) bins[i] = 0u;
    __syncthreads();
    for (int i = tid; i < batch; i += nt) atomicAdd(&bins[bin_of(i)], 1u);
    __syncthreads();
    if (tid < 32) {  // exclusive prefix sum: 20 bins a lane
        constexpr int per = kClasses * kCostBins / 32;
        unsigned int sum = 0;
        for (int q = 0; q < per; ++q) sum += bins[tid * per + q];
        unsigned int inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (tid >= o) inc += v;
        }
        unsigned int at = inc - sum;
        for (int q = 0; q < per; ++q) {
            const unsigned int c = bins[tid * per + q];
            bins[tid * per + q] = at;
            at += c;
        }
    }
    __syncthreads();
    if (tid <= kClasses) ctl[8 + tid] = tid < kClasses ? bins[tid * kCostBins] : (unsigned)batch;
    if (tid == 0) ctl[0] = 0u;
    __syncthreads();
    for (int i = tid; i < batch; i += nt) order[atomicAdd(&bins[bin_of(i)], 1u)] = i;
}

// ---------------------------------------------------------------- one matrix by NW warps
// Reflector of [alpha; x] with ||x||^2 = xn2: beta, tau, scale = 1 / (alpha - beta), u0 = alpha - beta.
__device__ __forceinline__ void reflector(float alpha, float xn2, float &beta, float &tau, float &scale, float &u0) {
    beta = alpha, tau = 0.f, scale = 0.f, u0 = 0.f;
    if (xn2 > 0.f) {
        float r, rs;
        nla::sqrt_and_inverse(fmaf(alpha, alpha, xn2), r, rs);
        beta = alpha >= 0.f ? -r : r;
        tau = fmaf(fabsf(alpha), rs, 1.f);
        u0 = alpha - beta;
        scale = nla::inverse(u0);
    }
}

constexpr int pow2_ceil(int x) {
    int p = 1;
    while (p < x) p *= 2;
    return p;
}

// Sums of v[0..P-1] over the lanes; lane l is left with the sum of v[l / (32 / P)].
template <int P>
__device__ __forceinline__ float reduce_scatter(float (&v)[P], int lane) {
    int o = 16;
#pragma unroll
    for (int h = P / 2; h >= 1; h /= 2, o /= 2) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const float send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    for (; o >= 1; o /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

template <class F, int... K>
__device__ __forceinline__ void static_for_impl(F &&f, std::integer_sequence<int, K...>) {
    (f(std::integral_constant<int, K>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void static_for(F &&f) {
    static_for_impl(static_cast<F &&>(f), std::make_integer_sequence<int, N>{});
}

// NW warps, tiles of 32 RR rows x NW RC columns for the bidiagonalisation, of which the first
// RCS columns of every warp live in shared memory (they are the first to be finished), and
// 32 QR rows in a chunk of the QR reduction.
template <int NW_, int RR_, int RC_, int RCS_, int QR_>
struct Cls {
    static constexpr int NW = NW_, RR = RR_, RC = RC_, RCS = RCS_, QR = QR_;
    static constexpr int NMAX = NW * RC, RH = 32 * RR;
    // shared floats of a worker; R packed by columns: entry (i, c) at c (c + 1) / 2 + i
    static constexpr int kPacked = (NMAX * (NMAX + 1) / 2 + 3) & ~3;
    static constexpr int kColsAt = RCS ? ((RCS * NW * (RCS * NW + 1) / 2 + 31) & ~31) : 0;  // shared columns, after R's first ones
    static constexpr int kBig = RCS && kColsAt + RCS * NW * RH > kPacked ? kColsAt + RCS * NW * RH : kPacked;
    static constexpr int kPart = RH + 32 / NW;  // conflict-free for two threads a row
    static constexpr int kFloats = kBig + 2 * 32 * (RR > QR ? RR : QR) + 2 * NW * RC + (NW > 1 ? NW * kPart : 0) + 2 * RH + 32 + 2 * NMAX +
                                   2 * NMAX;
};

template <class C>
struct Worker {
    static constexpr int NW = C::NW, RC = C::RC, RCS = C::RCS, RH = C::RH;
    float *big, *us, *rowb, *mbuf, *part, *ys, *a1s, *misc, *d, *e, *t2;
    int w, lane, bar;

    __device__ Worker(float *sm, int warp, int lane_) : w(warp % NW), lane(lane_), bar(1 + warp / NW) {
        constexpr int rows = 32 * (C::RR > C::QR ? C::RR : C::QR);
        big = sm;
        us = big + C::kBig;
        rowb = us + 2 * rows;
        mbuf = rowb + NW * RC;
        part = mbuf + NW * RC;
        ys = part + (NW > 1 ? NW * C::kPart : 0);
        a1s = ys + RH;
        misc = a1s + RH;  // [0..1] alpha by parity, [2] right alpha, [16 ..] the warps' partial norms
        t2 = misc + 32;
        d = t2 + 2 * C::NMAX;
        e = d + C::NMAX;
        rowb += w * RC;
        mbuf += w * RC;
    }
    __device__ __forceinline__ void sync() const {
        if (NW == 1)
            __syncwarp();
        else
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(32 * NW) : "memory");
    }

    // Left reflector step on columns of group k: with u (rows of column j, zero where it does not
    // reach), form the coefficients m_c of every column c > j of the warp and subtract u m_c.
    // row(q): entry (j, c) of the warp's column k + q before the step; set_row(q, w): what happens
    // to it.  Returns through mk[] the coefficients (zero for finished columns).
    template <int K, int RR, class Get, class Row, class SetRow>
    __device__ __forceinline__ void left_coeffs(const float (&u)[RR], int r0, int w0, float alpha, Get get, Row row,
                                                SetRow set_row, float (&mk)[RC], float &beta, float &u0) {
        constexpr int CNT = RC - K, P = pow2_ceil(CNT);
        float z[P], nrm = 0.f;
#pragma unroll
        for (int q = 0; q < P; ++q) z[q] = 0.f;
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            if (r < r0) continue;
            nrm = fmaf(u[r], u[r], nrm);
#pragma unroll
            for (int q = 0; q < CNT; ++q) z[q] = fmaf(u[r], get(r, K + q), z[q]);
        }
        nrm = nla::warp_sum(nrm);
        const float zs = reduce_scatter<P>(z, lane);
        const int q = lane / (32 / P);
        float tau, scale;
        reflector(alpha, nrm, beta, tau, scale, u0);
        const bool live = q < CNT && (q > 0 || w > w0);
        const float wc = live ? tau * fmaf(scale, zs, row(min(q, CNT - 1))) : 0.f;
        if (lane % (32 / P) == 0 && q < CNT) {
            mbuf[K + q] = scale * wc;
            if (live) set_row(q, wc);
        }
        __syncwarp();
#pragma unroll
        for (int t = K; t < RC; ++t) mk[t] = mbuf[t];
    }

    // R (packed in big) <- R of the QR factorisation of [R; A], A = rows in the tile.
    __device__ void qr_chunk(float (&a)[C::QR][RC], int N) {
        constexpr int RR = C::QR, rows = 32 * RR;
        static_for<RC>([&](auto kc) {
            constexpr int K = decltype(kc)::value;
#pragma unroll 1
            for (int w0 = 0; w0 < NW; ++w0) {
                const int j = K * NW + w0;
                if (j >= N) break;
                float *ub = us + (j & 1) * rows, *rjj = big + j * (j + 1) / 2 + j;
                if (w == w0) {
#pragma unroll
                    for (int r = 0; r < RR; ++r) ub[32 * r + lane] = a[r][K];
                    if (lane == 0) misc[j & 1] = *rjj;
                }
                sync();
                float u[RR], mk[RC], beta, u0;
#pragma unroll
                for (int r = 0; r < RR; ++r) u[r] = ub[32 * r + lane];
                const auto rjc = [&](int q) -> float & {
                    const int c = w + NW * (K + q);
                    return big[c * (c + 1) / 2 + j];
                };
                left_coeffs<K, RR>(u, 0, w0, misc[j & 1], [&](int r, int t) { return a[r][t]; },
                                   [&](int q) { return q > 0 || w > w0 ? rjc(q) : 0.f; },
                                   [&](int q, float wc) { rjc(q) -= wc; }, mk, beta, u0);
                if (w == w0 && lane == 0) *rjj = beta;
#pragma unroll
                for (int r = 0; r < RR; ++r)
#pragma unroll
                    for (int t = K; t < RC; ++t) a[r][t] = fmaf(-u[r], mk[t], a[r][t]);
                if (NW == 1) __syncwarp();
            }
        });
    }

    // Bidiagonalisation of the tile (M x N, M <= RH): d, e.
    __device__ void bidiag(float (&a)[C::RR][RC - RCS], int N) {
        constexpr int RR = C::RR;
        float *const sc = big + C::kColsAt + w * RH + lane;  // column w + NW t, t < RCS, at sc + t NW RH
        const auto get = [&](int r, int t) -> float & { return t < RCS ? sc[t * NW * RH + 32 * r] : a[r][t < RCS ? 0 : t - RCS]; };
        static_for<RC>([&](auto kc) {
            constexpr int K = decltype(kc)::value, R0 = K * NW / 32;  // rows 32 R0 .. are not finished
#pragma unroll 1
            for (int w0 = 0; w0 < NW; ++w0) {
                const int j = K * NW + w0, jl = j % 32;
                if (j >= N) break;
                // ---- left reflector of column j
                if (w == w0) {
#pragma unroll
                    for (int r = R0; r < RR; ++r) {
                        const float v = get(r, K);
                        us[32 * r + lane] = r > R0 || lane > jl ? v : 0.f;
                        if (r == R0 && lane == jl) misc[0] = v;
                    }
                }
                if (lane == jl) {
#pragma unroll
                    for (int t = K; t < RC; ++t) rowb[t] = get(R0, t);
                }
                sync();
                float u[RR], mk[RC], beta, u0;
#pragma unroll
                for (int r = R0; r < RR; ++r) u[r] = us[32 * r + lane];
                left_coeffs<K, RR>(u, R0, w0, misc[0], get, [&](int q) { return rowb[K + q]; }, [](int, float) {}, mk, beta, u0);
                if (lane == jl) u[R0] = u0;  // row j: its entries drop by w_c = u_0 m_c
#pragma unroll
                for (int r = R0; r < RR; ++r)
#pragma unroll
                    for (int t = K; t < RC; ++t) {
                        float &x = get(r, t);
                        x = fmaf(-u[r], mk[t], x);
                    }
                if (w == w0 && lane == 0) d[j] = beta;
                if (j + 1 >= N) break;
                // ---- right reflector of row j: entries x_c, c > j; alpha = x_{j+1} in warp w1, column k or k + 1
                const bool wrap = w0 + 1 == NW;
                const int w1 = wrap ? 0 : w0 + 1;
                __syncwarp();
                if (lane == jl) {
#pragma unroll
                    for (int t = K; t < RC; ++t) rowb[t] = t > K || w > w0 ? get(R0, t) : 0.f;
                }
                __syncwarp();
                float x[RC], y[RR], pn = 0.f;
#pragma unroll
                for (int t = K; t < RC; ++t) x[t] = rowb[t];
                constexpr int K1 = K + 1 < RC ? K + 1 : K;
                if (w == w1) {
                    if (lane == 0) misc[2] = wrap ? x[K1] : x[K];
#pragma unroll
                    for (int r = R0; r < RR; ++r) a1s[32 * r + lane] = wrap ? get(r, K1) : get(r, K);
                    if (wrap)
                        x[K1] = 0.f;
                    else
                        x[K] = 0.f;
                }
#pragma unroll
                for (int r = R0; r < RR; ++r) {
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int t = K; t < RC; t += 2) {
                        s0 = fmaf(get(r, t), x[t], s0);
                        if (t + 1 < RC) s1 = fmaf(get(r, t + 1), x[t + 1], s1);
                    }
                    y[r] = s0 + s1;
                }
#pragma unroll
                for (int t = K; t < RC; ++t) pn = fmaf(x[t], x[t], pn);
                if constexpr (NW > 1) {
#pragma unroll
                    for (int r = R0; r < RR; ++r) part[w * C::kPart + 32 * r + lane] = y[r];
                    if (lane == 0) misc[16 + w] = pn;
                    sync();
                    // two threads a row add the warps' sums
                    const int t = w * 32 + lane, row = 32 * R0 + (t >> 1);
                    if (row < RH) {
                        float s = 0.f;
#pragma unroll
                        for (int q = 0; q < NW / 2; ++q) s += part[((t & 1) * (NW / 2) + q) * C::kPart + row];
                        static_assert(RH % 16 == 0, "a warp's 16 rows exist together");
                        s += __shfl_xor_sync(0xffffffffu, s, 1);
                        if ((t & 1) == 0) ys[row] = s;
                    }
                    sync();
                    pn = 0.f;
#pragma unroll
                    for (int q = 0; q < NW; ++q) pn += misc[16 + q];
#pragma unroll
                    for (int r = R0; r < RR; ++r) y[r] = ys[32 * r + lane];
                } else {
                    __syncwarp();
                }
                float tau, scale;
                reflector(misc[2], pn, beta, tau, scale, u0);
                if (w == w0 && lane == 0) e[j] = beta;
                if (w == w1) {
                    if (wrap)
                        x[K1] = u0;
                    else
                        x[K] = u0;
                }
#pragma unroll
                for (int r = R0; r < RR; ++r) {
                    const float m = scale * (tau * fmaf(scale, y[r], a1s[32 * r + lane]));
#pragma unroll
                    for (int t = K; t < RC; ++t) {
                        float &v = get(r, t);
                        v = fmaf(-m, x[t], v);
                    }
                }
                if (NW == 1) __syncwarp();
            }
        });
    }

    // Values of the bidiagonal (d, e) by multisection, L lanes per value; S descending.
    __device__ void values(int N, float *S) {
        const int t = w * 32 + lane;
        sync();
        float b = 0.f;
        for (int i = t; i < N; i += 32 * NW) {
            const float el = i > 0 ? fabsf(e[i - 1]) : 0.f, er = i + 1 < N ? fabsf(e[i]) : 0.f;
            b = fmaxf(b, fabsf(d[i]) + fmaxf(el, er));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, o));
        if (NW > 1) {
            if (lane == 0) misc[16 + w] = b;
            sync();
#pragma unroll
            for (int q = 0; q < NW; ++q) b = fmaxf(b, misc[16 + q]);
        }
        if (!(b > 0.f)) {  // zero
            for (int i = t; i < N; i += 32 * NW) S[i] = 0.f;
            return;
        }
        // B is scaled by 2^-ex, in two factors that are normal numbers, to a bound in [0.5, 1)
        int ex;
        frexpf(b, &ex);
        const float f1 = ldexpf(1.f, -(ex / 2)), f2 = ldexpf(1.f, -(ex - ex / 2));
        for (int i = t; i < 2 * N - 1; i += 32 * NW) {
            const float v = ((i & 1) ? e[i >> 1] : d[i >> 1]) * f1 * f2;
            t2[i] = fmaxf(v * v, nla::kT2FloorF);
        }
        sync();
        int L = 1;
        while (L < 32 && N * L * 2 <= 32 * NW) L *= 2;
        const int idx = t / L, l = t % L, gbase = lane & ~(L - 1);
        const unsigned full = L == 32 ? 0xffffffffu : (1u << L) - 1, gmask = full << gbase;
        if (idx < N) {  // uniform over the group of L lanes
            const int j = N - 1 - idx;
            const float frac = (float)(l + 1) / (float)(L + 1);
            float lo = 0.f, hi = 1.f;
            for (int round = 0; round < 64 && hi - lo > 0x1p-23f; ++round) {
                const float x = fmaf(hi - lo, frac, lo);
                const bool below = nla::sturm_neg(2 * N - 1, t2, x) - N <= j;
                const unsigned m = (__ballot_sync(gmask, below) >> gbase) & full;
                const int f = m == full ? L : __ffs(~m) - 1;  // first point whose count passes j
                const float xf = __shfl_sync(gmask, x, gbase + min(f, L - 1));
                const float xp = __shfl_sync(gmask, x, gbase + max(f - 1, 0));
                if (f < L) hi = xf;
                if (f > 0) lo = xp;
            }
            if (l == 0) S[idx] = 0.5f * (lo + hi) / f1 / f2;
        }
    }

    // The matrix A (m x n, column-major, lda): M >= N after transposition (tr).
    __device__ void run(const float *A, int M, int N, int lda, bool tr, float *S) {
        const auto entry = [&](int i, int c) {
            return i < M && c < N ? (tr ? A[c + (size_t)i * lda] : A[i + (size_t)c * lda]) : 0.f;
        };
        constexpr int RR = C::RR;
        const bool qr = M > RH;
        if (qr) {
            for (int i = w * 32 + lane; i < N * (N + 1) / 2; i += 32 * NW) big[i] = 0.f;
            for (int base = 0; base < M; base += 32 * C::QR) {
                float a[C::QR][RC];
#pragma unroll
                for (int t = 0; t < RC; ++t)
#pragma unroll
                    for (int r = 0; r < C::QR; ++r) a[r][t] = entry(base + 32 * r + lane, w + NW * t);
                sync();
                qr_chunk(a, N);
            }
            sync();
        }
        float a[RR][RC - RCS];
#pragma unroll
        for (int t = RCS; t < RC; ++t)
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const int i = 32 * r + lane, c = w + NW * t;
                a[r][t - RCS] = qr ? (i <= c && c < N ? big[c * (c + 1) / 2 + i] : 0.f) : entry(i, c);
            }
        if constexpr (RCS > 0) {
            sync();  // R's later columns are in registers: the shared columns may take their place
            float *const sc = big + C::kColsAt + w * RH + lane;
#pragma unroll
            for (int t = 0; t < RCS; ++t)
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    const int i = 32 * r + lane, c = w + NW * t;
                    sc[t * NW * RH + 32 * r] = qr ? (i <= c && c < N ? big[c * (c + 1) / 2 + i] : 0.f) : entry(i, c);
                }
        }
        bidiag(a, N);
        values(N, S);
        sync();
    }
};

// Tile shapes.  256 columns do not fit the registers beside their addresses, hence six columns a
// warp in shared memory (seven and eight measured 5 and 7 % slower at 256 x 256).  us for one
// unit (one SM's 16 warps), square / 4:1 tall: N = 256 615 / 1908, 192 305 / 848, 128 (two
// matrices) 211 / 541, 64 (four) 104 / 192, 32 (sixteen) 99 / 151.  Rows per chunk of the QR:
// larger chunks only paid for the two smallest classes (64 rows a chunk: 237 and 172 us).
// The 10,000-matrix workload (n ~ U{8..256}, m/n ~ U[1, 4]): 186.0 ms with the matrices in
// shared or global memory, 33.7 ms with these; 300 small ones (n <= 64): 726 -> 184 us.
using Class0 = Cls<16, 8, 16, 6, 4>;
using Class1 = Cls<16, 6, 12, 0, 6>;
using Class2 = Cls<8, 4, 16, 0, 4>;
using Class3 = Cls<4, 2, 16, 0, 4>;
using Class4 = Cls<1, 1, 32, 0, 2>;

constexpr int worker_floats() {
    int f = Class0::kFloats;
    f = std::max(f, Class1::kFloats);
    f = std::max(f, 2 * Class2::kFloats);
    f = std::max(f, 4 * Class3::kFloats);
    return std::max(f, 16 * Class4::kFloats);
}

template <class C>
__device__ __noinline__ void run_worker(float *smem, int warp, int lane, const float *A, int M, int N, int lda, bool tr, float *S) {
    Worker<C> wk(smem + warp / C::NW * C::kFloats, warp, lane);
    wk.run(A, M, N, lda, tr, S);
}

// One matrix by one block of C::NW warps.
template <class C>
__global__ void __launch_bounds__(32 * C::NW, 1)
one_svd_kernel(const float *A, int M, int N, int lda, int tr, float *S, int *info) {
    extern __shared__ __align__(16) float smem[];
    run_worker<C>(smem, threadIdx.x >> 5, threadIdx.x & 31, A, M, N, lda, tr != 0, S);
    if (threadIdx.x == 0) *info = 0;
}

template <class C>
cudaError_t one_launch(const float *A, int M, int N, int lda, bool tr, float *S, int *info, cudaStream_t st) {
    static nla::PerDeviceOnce attr;
    constexpr int smem = C::kFloats * (int)sizeof(float);
    attr.run([] {
        cudaFuncSetAttribute(one_svd_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        cudaGetLastError();
    });
    one_svd_kernel<C><<<1, 32 * C::NW, smem, st>>>(A, M, N, lda, tr ? 1 : 0, S, info);
    return cudaGetLastError();
}

__global__ void __launch_bounds__(kThreads, 1)
batched_svd_kernel(const int *__restrict__ dM, const int *__restrict__ dN, const int *__restrict__ dLda,
                   float *const *dA, float *const *dS, const int *__restrict__ order, unsigned int *ctl,
                   int max_m, int max_n, int *dInfo) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int sh_unit;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    while (true) {
        if (tid == 0) sh_unit = (int)atomicAdd(ctl, 1u);
        __syncthreads();
        int unit = sh_unit, cls = 0, first = 0, per = 1, end = 0;
        for (; cls < kClasses; ++cls) {
            first = (int)ctl[8 + cls];
            end = (int)ctl[8 + cls + 1];
            per = kWarps / class_warps(cls);
            const int units = (end - first + per - 1) / per;
            if (unit < units) break;
            unit -= units;
        }
        if (cls == kClasses) break;
        const int pos = first + unit * per + warp / class_warps(cls);
        if (pos < end) {
            const int i = order[pos];
            const int m = dM[i], n = dN[i], lda = dLda[i];
            const int M = max(m, n), N = min(m, n);
            // Large matrices beyond the declared bounds are refused.  The bounds may be those of m_i and n_i
            // or of the larger and the smaller dimension; up to max_m max_n entries are accepted either way.
            const bool within = (m <= max_m && n <= max_n) || (long)M * N <= kBucketElems ||
                                (long)((M + 3) & ~3) * N <= (long)((max(max_m, 1) + 3) & ~3) * max(max_n, 1);
            const bool ok = N <= 256 && within;
            if (ok && N > 0) {
                const float *A = dA[i];
                float *S = dS[i];
                const bool tr = m < n;
                switch (cls) {
                    case 0: run_worker<Class0>(smem, warp, lane, A, M, N, lda, tr, S); break;
                    case 1: run_worker<Class1>(smem, warp, lane, A, M, N, lda, tr, S); break;
                    case 2: run_worker<Class2>(smem, warp, lane, A, M, N, lda, tr, S); break;
                    case 3: run_worker<Class3>(smem, warp, lane, A, M, N, lda, tr, S); break;
                    default: run_worker<Class4>(smem, warp, lane, A, M, N, lda, tr, S); break;
                }
            }
            if (lane == 0 && warp % class_warps(cls) == 0) dInfo[i] = ok ? 0 : -NLA_ERR_UNSUPPORTED;
        }
        __syncthreads();
    }
}

}  // namespace

namespace nla {

// us on GB300, fitted to N = 16 .. 256 and M / N = 1 .. 64: this file's one-block form against the
// two-stage reduction of a whole GPU, whose chains of steps cost about 3.4 us a column however
// small the matrix is (N = 64, M = 64: 80 against 209; M = 1,024: 465 against 245; N = 256: 610
// against 965 square, 1,244 against 1,004 at 512 rows).
bool small_svd_pays(int m, int n) {
    const float M = (float)std::max(m, n), N = (float)std::min(m, n);
    if (N > 256.f || M > 65536.f) return false;
    const auto chunks = [&](float tile, float rows) { return M > tile ? ceilf(M / rows) : 0.f; };
    const float one = N <= 64.f    ? 1.3f + 0.8f * chunks(64.f, 128.f)
                      : N <= 128.f ? 1.3f + 0.55f * chunks(128.f, 128.f)
                      : N <= 192.f ? 1.65f + 0.7f * chunks(192.f, 192.f)
                                   : 2.4f + 0.62f * chunks(256.f, 128.f);
    return one * N < 0.9f * (3.35f * N + 0.0016f * N * N + 0.00035f * M * N);
}

// Singular values of the column-major m x n matrix (read only), min(m, n) <= 256.
cudaError_t small_svd(const float *A, int m, int n, int lda, float *S, int *info, cudaStream_t st) {
    const int M = std::max(m, n), N = std::min(m, n);
    const bool tr = m < n;
    if (N > 192) return one_launch<Class0>(A, M, N, lda, tr, S, info, st);
    if (N > 128) return one_launch<Class1>(A, M, N, lda, tr, S, info, st);
    if (N > 64) return one_launch<Class2>(A, M, N, lda, tr, S, info, st);
    return one_launch<Class3>(A, M, N, lda, tr, S, info, st);  // (one warp alone is slower up to 32, too: 82 against 41 us)
}

// Group sizes per bucket installed by the tuner table (bucket b -> least threads per matrix).
int g_batched_group[kBuckets] = {0, 0, 0, 0, 0};
}

extern "C" {

nla_status nla_gesvd_vals_batched_workspace(int batch, nla_dtype dtype, int max_m, int max_n, size_t *bytes) {
    if (!bytes || batch < 0 || max_m < 0 || max_n < 0) return berr(NLA_ERR_ARG, "bad arguments");
    if (dtype != NLA_F32) return berr(NLA_ERR_UNSUPPORTED, "the batched kernel supports FP32 only");
    *bytes = 256 + ((size_t)std::max(batch, 1) * 4 + 255) / 256 * 256;  // control words, order
    return NLA_OK;
}

nla_status nla_gesvd_vals_batched(int batch, nla_dtype dtype, const int *dM, const int *dN, const int *dLda,
                                  void *const *dA_array, void *const *dS_array, int max_m, int max_n, void *dWork,
                                  size_t work_bytes, int *dInfo, const nla_opts *opts, nla_stream_t stream) {
    (void)opts;
    if (dtype != NLA_F32) return berr(NLA_ERR_UNSUPPORTED, "the batched kernel supports FP32 only");
    if (batch < 0 || max_m < 0 || max_n < 0) return berr(NLA_ERR_ARG, "negative size");
    if (batch == 0) return NLA_OK;
    if (std::min(max_m, max_n) > 256) return berr(NLA_ERR_UNSUPPORTED, "min(m_i, n_i) must be <= 256");
    if (!dM || !dN || !dLda || !dA_array || !dS_array || !dInfo || !dWork)
        return berr(NLA_ERR_ARG, "null device pointer");
    size_t need = 0;
    nla_gesvd_vals_batched_workspace(batch, dtype, max_m, max_n, &need);
    if (work_bytes < need) return berr(NLA_ERR_WORKSPACE, "workspace too small");
    if (((uintptr_t)dWork) % 256) return berr(NLA_ERR_WORKSPACE, "workspace not 256-byte aligned");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    char *w = reinterpret_cast<char *>(dWork);
    unsigned int *ctl = reinterpret_cast<unsigned int *>(w);
    int *order = reinterpret_cast<int *>(w + 256);
    BatchCfg cfg;
    for (int b = 0; b < kBuckets; ++b) {
        const int g = nla::g_batched_group[b];
        cfg.group[b] = g >= 32 && g <= 256 && 256 % g == 0 ? g : 32;
    }
    static nla::PerDeviceOnce attr;
    constexpr size_t smem = (size_t)worker_floats() * sizeof(float);
    attr.run([&] {
        cudaFuncSetAttribute(batched_svd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaGetLastError();
    });
    {
        nla::TraceScope ts(nla::kTrBatched, st);
        batched_prep_kernel<<<1, 1024, 0, st>>>(batch, dM, dN, order, ctl, cfg);
        const int blocks = std::min(nla::device_sm_count(), batch);
        batched_svd_kernel<<<blocks, kThreads, smem, st>>>(dM, dN, dLda, (float *const *)dA_array, (float *const *)dS_array,
                                                           order, ctl, max_m, max_n, dInfo);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return berr(NLA_ERR_CUDA, cudaGetErrorString(e));
    return NLA_OK;
}

}  // extern "C"
