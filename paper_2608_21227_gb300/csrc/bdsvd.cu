// bdsvd.cu -- stage 3: singular values of the upper bidiagonal B(d, e).
//
// Section 5.1.1 ends the reduction at "diagonal form"; here the bidiagonal's
// singular values are found by bisection, which is data-parallel (one thread
// per singular value) where QR iteration is sequential.  The eigenvalues of
// the 2n x 2n Golub-Kahan tridiagonal TGK (zero diagonal, off-diagonals
// t = d_0, e_0, d_1, e_1, ..., d_{n-1}) are +-sigma_i, so for x > 0 the number
// of singular values below x is negcount(TGK - x I) - n, where negcount counts
// the negative pivots of the LDL^T factorisation of TGK - x I (Sylvester's law
// of inertia), counted here as the sign changes of its leading minors (sturm.cuh).
//
// GB300's FP64 pipe issues a small fraction of the FP32 rate, so the search is
// split:
//   prep:   B is scaled by a power of two so its Gershgorin bound is <= 1
//           (exact), and the squares t_i^2 are stored once in FP64 and FP32;
//   coarse: multisection with FP32 Sturm counts.  A group of kl lanes owns one
//           value and counts at kl interior points of its bracket per round, so
//           a round shrinks the bracket (kl+1)-fold where bisection halves it.
//           An FP32 count is the exact count of a matrix whose off-diagonals
//           differ relatively by a few FP32 rounding errors, so it can only
//           misplace values within 2^-22 (the scaled bound is 1).  For FP32
//           output that is the answer: the reduction before it has the same
//           absolute error level.  For FP64 output the coarse bracket stops at
//           2^-19 and is widened by 2^-20 on both sides, which keeps the value
//           inside it;
//   fine:   (FP64 output) multisection with FP64 counts to 2^-51 of the bound,
//           kl lanes per value (kl = 1, plain bisection, for large n; more lanes
//           when few values would leave most SMs idle).
//
// What bounds it: a count is a chain of 2n dependent terms, a term one FMA deep and
// about five instructions (FP32) or 2.25 FP64-pipe instructions.  The pivot form this
// replaced divided once per term.  Measured on GB300, whole stage, pivot form -> minors:
// FP32 output n = 1024 0.52 -> 0.13 ms, n = 8192 4.9 -> 1.6 ms; FP64 output n = 256
// 1.30 -> 0.38 ms, n = 2048 16.7 -> 4.7 ms.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"
#include "sturm.cuh"

namespace nla {

constexpr int kBisectThreads = 32;  // fine phase: one warp per block spreads the FP64 work over all SMs
constexpr int kMsThreads = 128;

size_t bdsvd_scratch_bytes(int n) {
    const size_t m = (size_t)(n > 0 ? 2 * n : 1);
    return 256 + m * sizeof(double) + ((m * sizeof(float) + 255) / 256) * 256 + (size_t)(n > 0 ? n : 1) * 8;
}

// One block: Gershgorin bound, power-of-two scale, squared scaled off-diagonals.
__global__ void bd_prep_kernel(int n, const double *__restrict__ d, const double *__restrict__ e, double *hdr,
                               double *t2, float *t2f) {
    __shared__ double wb[32];
    __shared__ double sh_scale;
    double bnd = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double di = fabs(d[i]);
        double el = i > 0 ? fabs(e[i - 1]) : 0.0, er = i + 1 < n ? fabs(e[i]) : 0.0;
        bnd = fmax(bnd, di + fmax(el, er));
    }
    bnd = warp_max(bnd);
    if ((threadIdx.x & 31) == 0) wb[threadIdx.x >> 5] = bnd;
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b = fmax(b, wb[w]);
        int ex = 0;
        if (b > 0.0) frexp(b, &ex);  // b * 2^-ex in [0.5, 1)
        sh_scale = ldexp(1.0, -ex);
        hdr[0] = sh_scale;
        hdr[1] = b;
    }
    __syncthreads();
    const double s = sh_scale;
    for (int i = threadIdx.x; i < 2 * n - 1; i += blockDim.x) {
        double t = (i & 1) ? e[i >> 1] : d[i >> 1];
        t *= s;
        t2[i] = fmax(t * t, kT2FloorD);
        t2f[i] = fmaxf((float)(t * t), kT2FloorF);
    }
}

// Multisection with FP32 counts on [0, 1]: group g of kl lanes (a power of two <= 32)
// finds the g-th largest value.  Invariant: count(lo) - n <= j < count(hi) - n, i.e. the
// j-th smallest value lies in [lo, hi).  Each round every lane counts at its
// own interior point; the bracket becomes the first interval of consecutive
// points over which the count passes j.
template <typename T>
__global__ void __launch_bounds__(kMsThreads)
coarse_kernel(int n, const double *__restrict__ hdr, const float *__restrict__ t2f, float stop,
              float2 *__restrict__ br, T *__restrict__ S, int kl) {
    const int idx = (blockIdx.x * blockDim.x + threadIdx.x) / kl;
    const int l = threadIdx.x % kl;
    const int gbase = (threadIdx.x & 31) & ~(kl - 1);
    const unsigned full = kl == 32 ? 0xffffffffu : (1u << kl) - 1;
    const unsigned gmask = full << gbase;
    if (idx >= n) return;  // uniform over the group
    const int n2 = 2 * n - 1;
    const int j = n - 1 - idx;
    const float frac = (float)(l + 1) / (float)(kl + 1);
    float lo = 0.f, hi = 1.f;
    for (int round = 0; round < 64 && hi - lo > stop; ++round) {
        const float x = fmaf(hi - lo, frac, lo);
        const bool below = sturm_neg(n2, t2f, x) - n <= j;
        const unsigned m = (__ballot_sync(gmask, below) >> gbase) & full;
        const int f = m == full ? kl : __ffs(~m) - 1;  // first point whose count passes j; kl if none
        const float xf = __shfl_sync(gmask, x, gbase + min(f, kl - 1));
        const float xp = __shfl_sync(gmask, x, gbase + max(f - 1, 0));
        if (f < kl) hi = xf;
        if (f > 0) lo = xp;
    }
    if (l == 0) {
        if (S)
            S[idx] = (T)(0.5 * ((double)lo + (double)hi) / hdr[0]);
        else
            br[idx] = make_float2(lo, hi);
    }
}

// FP64 search from the widened coarse bracket: a group of kl lanes (a power of two,
// kl <= 32) per value counts at kl interior points per round (kl = 1: bisection).
// Few values leave most SMs idle, so the host gives each value more lanes then.
template <typename T>
__global__ void __launch_bounds__(kBisectThreads)
fine_kernel(int n, const double *__restrict__ hdr, const double *__restrict__ t2, const float2 *__restrict__ br,
            T *__restrict__ S, double fine_tol, int kl) {
    const int idx = (blockIdx.x * blockDim.x + threadIdx.x) / kl;
    const int l = threadIdx.x % kl;
    const int gbase = (threadIdx.x & 31) & ~(kl - 1);
    const unsigned gmask = (kl == 32 ? 0xffffffffu : ((1u << kl) - 1)) << gbase;
    if (idx >= n) return;  // uniform over the group
    const double s = hdr[0];
    const int n2 = 2 * n - 1;
    const int j = n - 1 - idx;  // idx-th largest == j-th smallest; counts below x are negcount - n
    const float2 b = br[idx];
    double dlo = fmax(0.0, (double)b.x - 0x1p-20), dhi = fmin(1.0, (double)b.y + 0x1p-20);
    const double frac = (double)(l + 1) / (double)(kl + 1);
    for (int it = 0; it < 80; ++it) {
        const double x = fma(dhi - dlo, frac, dlo);
        // stop at the tolerance or when the points no longer separate (FP64 spacing)
        const bool done = dhi - dlo <= fine_tol || !(x > dlo && x < dhi);
        if (__any_sync(gmask, done)) break;
        const bool below = sturm_neg(n2, t2, x) - n <= j;
        const unsigned full = gmask >> gbase;
        const unsigned m = (__ballot_sync(gmask, below) >> gbase) & full;
        const int f = m == full ? kl : __ffs(~m) - 1;  // first point whose count passes j; kl if none
        const double xf = __shfl_sync(gmask, x, gbase + min(f, kl - 1));
        const double xp = __shfl_sync(gmask, x, gbase + max(f - 1, 0));
        if (f < kl) dhi = xf;
        if (f > 0) dlo = xp;
    }
    if (l == 0) S[idx] = (T)(0.5 * (dlo + dhi) / s);
}

template <typename T>
cudaError_t bdsvd_bisect(int n, const double *d, const double *e, T *S, void *scratch, int *info, cudaStream_t st) {
    (void)info;
    if (n <= 0) return cudaSuccess;
    char *w = reinterpret_cast<char *>(scratch);
    double *hdr = reinterpret_cast<double *>(w);
    double *t2 = reinterpret_cast<double *>(w + 256);
    float *t2f = reinterpret_cast<float *>(w + 256 + (size_t)2 * n * sizeof(double));
    float2 *br = reinterpret_cast<float2 *>(w + 256 + (size_t)2 * n * sizeof(double) +
                                            (((size_t)2 * n * sizeof(float) + 255) / 256) * 256);
    bd_prep_kernel<<<1, 1024, 0, st>>>(n, d, e, hdr, t2, t2f);
    // lanes per value of the FP32 phase: the largest power of two <= 32 that keeps the
    // warps within two per SM sub-partition (one warp is bound by its chain of terms, two
    // fill the issue slots; more lanes shorten the search but count more in all)
    const long sub = 4L * device_sm_count() * 32;  // lanes of one warp per sub-partition
    int cl = 1;
    while (cl < 32 && (long)n * cl * 2 <= 2 * sub) cl *= 2;
    const int cblocks = (int)(((long)n * cl + kMsThreads - 1) / kMsThreads);
    if (sizeof(T) == 4) {
        coarse_kernel<T><<<cblocks, kMsThreads, 0, st>>>(n, hdr, t2f, 0x1p-23f, nullptr, S, cl);
        return cudaGetLastError();
    }
    coarse_kernel<T><<<cblocks, kMsThreads, 0, st>>>(n, hdr, t2f, 0x1p-19f, br, nullptr, cl);
    // lanes per value: the largest power of two <= 32 that keeps n * kl / 32 warps
    // within one per SM sub-partition (the FP64 count is bound by that pipe)
    int kl = 1;
    while (kl < 32 && (long)n * kl * 2 <= sub) kl *= 2;
    const long fthreads = (long)n * kl;
    fine_kernel<T><<<(int)((fthreads + kBisectThreads - 1) / kBisectThreads), kBisectThreads, 0, st>>>(
        n, hdr, t2, br, S, 0x1p-51, kl);
    return cudaGetLastError();
}

template cudaError_t bdsvd_bisect<double>(int, const double *, const double *, double *, void *, int *, cudaStream_t);
template cudaError_t bdsvd_bisect<float>(int, const double *, const double *, float *, void *, int *, cudaStream_t);

}  // namespace nla
