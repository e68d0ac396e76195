// update_strip.cu -- FP32 trailing update of a small trailing block in one launch (Algorithm
// 2, both sides): X <- (I - V T V^T)^T X (side 0, QR) and X <- X (I - V T V^T) (side 1, LQ).
//
// A block owns a strip of C lines (columns of X on the QR side, rows on the LQ side) over the
// whole long dimension L, keeps it in shared memory, and does all three steps on it: W = V^T
// strip, W' = T^T W, strip -= V W'.  X is read and written once (8 bytes an element where the
// two-kernel path moves 12), nothing crosses blocks (no split sums, no tickets), and a
// trailing update is one launch instead of two.
//
// Threads: G groups of 512 / G threads over the long dimension.  Step 1 gives a group NB / G of
// the reflectors for all C lines, step 3 C / G of the lines with all reflectors: 64
// accumulators or coefficients in registers either way, 64 FMAs per 8 to 20 shared-memory reads.
// V is staged by chunks of the long dimension, reflector-major, one chunk ahead in registers;
// step 3 takes the chunks in reverse order, starting with the one that is still there.
//
// Bound: shared-memory reads and the FMA pipe per strip (about equal), so a strip's time grows
// with L only, and re-reading V per strip from L2; above two thousand or so the two-kernel path's
// larger tiles win.  Measured with band 16, us per side averaged over the steps of a square
// matrix, two kernels -> this one where it is chosen: n = 256 21 -> 8, 1,024 24 -> 9.7, 2,048 27 ->
// 16.4, 4,096 35.6 -> 30.1.  Lines per strip (4 / 8 / 16) at n = 1,024: 11.1 / 10.0 / 12.4.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace nla {

namespace {

constexpr int kStripThreads = 512;

template <int NB>
constexpr int strip_chunk() {
    return 8192 / NB;  // 16 elements of V per thread
}
template <int NB>
constexpr int strip_vld() {
    return strip_chunk<NB>() + 2;  // 2 mod 8: the LQ side's transposing stores hit distinct banks
}

// Halving exchanges over the warp's lanes: lane l is left with the sums of entries 2 l and 2 l + 1.
template <int H>
NLA_DEV void fold(float (&a)[64], int lane) {
    const bool up = (lane & (H / 2)) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        const float send = up ? a[i] : a[i + H], keep = up ? a[i + H] : a[i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, H / 2);
    }
    if constexpr (H > 2) fold<H / 2>(a, lane);
}

size_t strip_smem(int NB, int C, int L) {
    const size_t lp = (size_t)((L + 3) & ~3);
    const size_t vs = (size_t)2 * NB * (8192 / NB + 2);
    return sizeof(float) * (C * lp + vs + 16 * 64 + 2 * NB * C + NB * NB);
}

template <int SIDE, int NB, int C>
__global__ void __launch_bounds__(kStripThreads, 1)
strip_kernel(float *__restrict__ X, long ldx, int lines, int L, const float *__restrict__ V, long ldv,
             const float *__restrict__ Tm, int vec) {
    pdl_wait();
    pdl_trigger();
    constexpr int NT = kStripThreads, G = C * NB / 64, LT = NT / G, KPG = NB / G, CU = C / G;
    constexpr int LC = strip_chunk<NB>(), LDV = strip_vld<NB>();
    static_assert(G >= 1 && KPG * C == 64 && CU * NB == 64 && LT % 32 == 0, "shape");
    extern __shared__ __align__(16) float sm[];
    const int lp = (L + 3) & ~3;
    float *Xs = sm;                      // C x lp: Xs[c * lp + l]
    float *Vs = Xs + (size_t)C * lp;     // two chunks, NB x LDV each
    float *part = Vs + 2 * NB * LDV;     // 16 warps x 64
    float *Ws = part + 16 * 64, *Wp = Ws + NB * C, *Ts = Wp + NB * C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c0 = blockIdx.x * C, nc = min(C, lines - c0);
    const int nchunk = (L + LC - 1) / LC;

    // one chunk of V, 16 elements a thread.  QR: V(l, k) = V[l + k ldv], four consecutive l of a
    // reflector per read; LQ: V(l, k) = V[k + l ldv], four consecutive reflectors of an l.
    float vr[16];
    const auto fetch = [&](int ch) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = tid + NT * i;  // of LC * NB / 4
            const int k = SIDE == 0 ? e / (LC / 4) : e % (NB / 4) * 4;
            const int l = ch * LC + (SIDE == 0 ? e % (LC / 4) * 4 : e / (NB / 4));
            const float *p = SIDE == 0 ? V + l + (long)k * ldv : V + k + (long)l * ldv;
            if (vec && (SIDE == 0 ? l + 3 < L : l < L)) {
                const float4 f = *reinterpret_cast<const float4 *>(p);
                vr[4 * i] = f.x, vr[4 * i + 1] = f.y, vr[4 * i + 2] = f.z, vr[4 * i + 3] = f.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) vr[4 * i + u] = (SIDE == 0 ? l + u : l) < L ? p[u] : 0.f;
            }
        }
    };
    // into buffer `buf`, as the unit lower trapezoid it stands for
    const auto stage = [&](int ch, int buf) {
        float *vs = Vs + buf * NB * LDV;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int e = tid + NT * i;
            const int k = SIDE == 0 ? e / (LC / 4) : e % (NB / 4) * 4;
            const int l = SIDE == 0 ? e % (LC / 4) * 4 : e / (NB / 4);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int kk = SIDE == 0 ? k : k + u, ll = SIDE == 0 ? l + u : l, gl = ch * LC + ll;
                float v = vr[4 * i + u];
                if (gl <= kk) v = gl == kk ? 1.f : 0.f;
                vs[kk * LDV + ll] = v;
            }
        }
    };
    fetch(0);
    // ---- the strip and T into shared memory
    if (SIDE == 0) {
        for (int i = tid; i < C * (lp / 4); i += NT) {
            const int c = i / (lp / 4), l = i % (lp / 4) * 4;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            const float *p = X + l + (long)(c0 + c) * ldx;
            if (c < nc) {
                if (vec && l + 3 < L) {
                    f = *reinterpret_cast<const float4 *>(p);
                } else {
                    f.x = p[0];
                    f.y = l + 1 < L ? p[1] : 0.f;
                    f.z = l + 2 < L ? p[2] : 0.f;
                    f.w = l + 3 < L ? p[3] : 0.f;
                }
            }
            *reinterpret_cast<float4 *>(Xs + c * lp + l) = f;
        }
    } else {
        for (int i = tid; i < C / 4 * L; i += NT) {
            const int l = i % L, c = i / L * 4;
            const float *p = X + c0 + c + (long)l * ldx;
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (vec && c + 3 < nc) {
                f = *reinterpret_cast<const float4 *>(p);
            } else {
                f.x = c < nc ? p[0] : 0.f;
                f.y = c + 1 < nc ? p[1] : 0.f;
                f.z = c + 2 < nc ? p[2] : 0.f;
                f.w = c + 3 < nc ? p[3] : 0.f;
            }
            Xs[c * lp + l] = f.x, Xs[(c + 1) * lp + l] = f.y, Xs[(c + 2) * lp + l] = f.z, Xs[(c + 3) * lp + l] = f.w;
        }
    }
    for (int i = tid; i < NB * NB; i += NT) Ts[i] = Tm[i];
    stage(0, 0);
    __syncthreads();
    const int grp = tid / LT, lt = tid % LT;
    // ---- W = V^T strip: reflectors grp * KPG ..
    {
        float acc[64];  // reflector k, line c at k C + c
#pragma unroll
        for (int i = 0; i < 64; ++i) acc[i] = 0.f;
        for (int ch = 0; ch < nchunk; ++ch) {
            if (ch + 1 < nchunk) fetch(ch + 1);
            const float *vs = Vs + (ch & 1) * NB * LDV + grp * KPG * LDV;
            const int lend = min(LC, L - ch * LC);
#pragma unroll 2
            for (int l = lt; l < lend; l += LT) {
                float v[KPG], x[C];
#pragma unroll
                for (int k = 0; k < KPG; ++k) v[k] = vs[k * LDV + l];
#pragma unroll
                for (int c = 0; c < C; ++c) x[c] = Xs[c * lp + ch * LC + l];
#pragma unroll
                for (int k = 0; k < KPG; ++k)
#pragma unroll
                    for (int c = 0; c < C; ++c) acc[k * C + c] = fmaf(v[k], x[c], acc[k * C + c]);
            }
            if (ch + 1 < nchunk) stage(ch + 1, (ch + 1) & 1);
            __syncthreads();
        }
        fold<32>(acc, lane);
        *reinterpret_cast<float2 *>(part + warp * 64 + 2 * lane) = make_float2(acc[0], acc[1]);
    }
    __syncthreads();
    // ---- the group's warps, then W' = T^T W
    for (int i = tid; i < NB * C; i += NT) {
        const int k = i / C, c = i % C, g = k / KPG;
        float s = 0.f;
#pragma unroll
        for (int w = 0; w < LT / 32; ++w) s += part[(g * (LT / 32) + w) * 64 + (k % KPG) * C + c];
        Ws[i] = s;
    }
    __syncthreads();
    for (int i = tid; i < NB * C; i += NT) {
        const int k = i / C, c = i % C;
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < NB; ++q) s = q <= k ? fmaf(Ts[q + k * NB], Ws[q * C + c], s) : s;
        Wp[i] = s;
    }
    __syncthreads();
    // ---- strip -= V W': lines grp * CU ..
    float w[NB][CU];
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int c = 0; c < CU; ++c) w[k][c] = Wp[k * C + grp * CU + c];
    for (int ch = nchunk - 1; ch >= 0; --ch) {
        if (ch > 0) fetch(ch - 1);
        const float *vs = Vs + (ch & 1) * NB * LDV;
        const int lend = min(LC, L - ch * LC);
#pragma unroll 2
        for (int l = lt; l < lend; l += LT) {
            // (summed first: the sums are small beside x, so x is rounded once per update)
            float x[CU];
#pragma unroll
            for (int c = 0; c < CU; ++c) x[c] = 0.f;
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                const float v = vs[k * LDV + l];
#pragma unroll
                for (int c = 0; c < CU; ++c) x[c] = fmaf(v, w[k][c], x[c]);
            }
#pragma unroll
            for (int c = 0; c < CU; ++c) x[c] = Xs[(grp * CU + c) * lp + ch * LC + l] - x[c];
            const int gl = ch * LC + l;
            if (SIDE == 0) {
#pragma unroll
                for (int c = 0; c < CU; ++c)
                    if (grp * CU + c < nc) X[gl + (long)(c0 + grp * CU + c) * ldx] = x[c];
            } else {
                float *p = X + c0 + grp * CU + (long)gl * ldx;
                if (CU == 4 && vec && grp * CU + 3 < nc) {
                    *reinterpret_cast<float4 *>(p) = make_float4(x[0], x[1 % CU], x[2 % CU], x[3 % CU]);
                } else {
#pragma unroll
                    for (int c = 0; c < CU; ++c)
                        if (grp * CU + c < nc) p[c] = x[c];
                }
            }
        }
        if (ch > 0) {
            stage(ch - 1, (ch - 1) & 1);
            __syncthreads();
        }
    }
}

template <int SIDE, int NB, int C>
cudaError_t strip_launch(float *X, long ldx, int lines, int L, const float *V, long ldv, const float *Tm, cudaStream_t st) {
    auto kern = strip_kernel<SIDE, NB, C>;
    static PerDeviceOnce once;
    allow_max_smem(kern, once);
    const int vec = ldx % 4 == 0 && ldv % 4 == 0 && reinterpret_cast<uintptr_t>(X) % 16 == 0 &&
                    reinterpret_cast<uintptr_t>(V) % 16 == 0;
    return launch_pdl(kern, dim3((lines + C - 1) / C), dim3(kStripThreads), strip_smem(NB, C, L), st, X, ldx, lines, L, V, ldv, Tm,
                      vec);
}

}  // namespace

// X (M x N) updated on `side` by the nb reflectors V (side 0: V(r, k) = V[r + k ldv], side 1:
// V(c, k) = V[k + c ldv]); cudaErrorNotSupported where the two-kernel path is the better one.
cudaError_t trail_strip(int side, float *X, long ldx, int M, int N, const float *V, long ldv, int nb, const float *Tm,
                        cudaStream_t st) {
    if ((nb != 16 && nb != 32) || M <= 0 || N <= 0) return cudaErrorNotSupported;
    const int lines = side == 0 ? N : M, L = side == 0 ? M : N, sms = device_sm_count();
    constexpr size_t kBudget = 226 * 1024;
    // us, fitted to 256 .. 3,072 squares: a block takes a fixed 6 us and its share of shared-memory
    // reads, and only one fits an SM, so what counts is the number of waves
    int C = 0;
    float best = 23.f + 2.4e-6f * (float)lines * (float)L;  // the two-kernel path
    for (int c = 4; c <= (nb == 16 ? 16 : 8); c *= 2) {
        if (strip_smem(nb, c, L) > kBudget) break;
        const int waves = ((lines + c - 1) / c + sms - 1) / sms;
        const float t = (float)waves * (6.f + 2.8e-5f * (float)nb * (float)c * (float)L);
        if (t < best) best = t, C = c;
    }
    if (C == 0) return cudaErrorNotSupported;
#define NLA_GO(SIDE, NB, CC) return strip_launch<SIDE, NB, CC>(X, ldx, lines, L, V, ldv, Tm, st)
    if (nb == 16) {
        if (side == 0) {
            if (C == 16) NLA_GO(0, 16, 16);
            if (C == 8) NLA_GO(0, 16, 8);
            NLA_GO(0, 16, 4);
        }
        if (C == 16) NLA_GO(1, 16, 16);
        if (C == 8) NLA_GO(1, 16, 8);
        NLA_GO(1, 16, 4);
    }
    if (side == 0) {
        if (C == 8) NLA_GO(0, 32, 8);
        NLA_GO(0, 32, 4);
    }
    if (C == 8) NLA_GO(1, 32, 8);
    NLA_GO(1, 32, 4);
#undef NLA_GO
}

}  // namespace nla
