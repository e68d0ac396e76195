// panel.cu -- Householder panel factorisation (the GEQRT/TSQRT step of
// Algorithm 1: "QR sweep" on a tile column, "LQ sweep" on a tile row).
//
// One cooperative launch factors an M x nb panel (nb <= 64).  The panel is
// split into row chunks, one per block, held in shared memory for the whole
// factorisation, so the panel is read from and written to global memory once.
// Column j needs one grid-wide reduction: every block contributes partial sums
// of ||x||^2 and of x . a_c for the columns c > j right of it (x = column j
// below the diagonal), the partials meet in global memory behind a counter
// barrier, and each block then finishes the reflector redundantly and updates
// its own rows.  The dot products are taken before beta is known, using
// v = [1; x / (alpha - beta)] so that v . a_c = a_jc + (x . a_c) / (alpha - beta);
// that is what makes one barrier per column enough.
//
// After the last column a second reduction forms G = V^T V and block 0 builds
// the compact-WY factor T (H_1 ... H_nb = I - V T V^T, T upper triangular,
// T_jj = tau_j, T(0:j, j) = -tau_j T(0:j, 0:j) G(0:j, j)), which the trailing
// update (Algorithm 2) consumes.
//
// Householder convention (LAPACK-style): beta = -sign(alpha) ||[alpha; x]||,
// sign(0) = +1, tau = (beta - alpha) / beta; a zero x gives tau = 0, H = I.
// This grid variant takes norms and cross-block sums in FP64 in every precision
// mode; the cluster variant below takes them in the panel's own precision (FP64 for
// the FP64 and mixed-precision paths, FP32 for the plain FP32 path).
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdlib>

#include "common.cuh"
#include "kernels.cuh"
#include "house.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

namespace nla {

constexpr int kPanelThreads = 256;
constexpr int kNbMax = 64;
constexpr int kPanelRowsTarget = 256;  // rows per block when the panel is long enough

size_t panel_part_doubles(int P) {
    return (size_t)2 * P * (kNbMax + 1) + (size_t)P * kNbMax * kNbMax + 2 * kNbMax;
}

int current_device() {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return dev;
}

int device_sm_count() {
    static PerDeviceValue<int> sms;
    return sms.get([] {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, std::max(current_device(), 0)) != cudaSuccess)
            cudaGetLastError();
        return n > 0 ? n : 1;
    });
}

int panel_max_ctas() { return device_sm_count(); }

// NLA_PDL=0: plain stream order.  With the panels and the small updates down to 8 to 20 us the
// launch gaps show (ms per FP32 SVD, off / on: 1024 5.28 / 4.66, 3001 x 1537 10.7 / 9.8, 8192
// 114.5 / 109.2).
bool pdl_enabled() {
    static const bool on = [] {
        const char *v = getenv("NLA_PDL");
        return !v || atoi(v) != 0;
    }();
    return on;
}

template <typename T>
__global__ void __launch_bounds__(kPanelThreads)
panel_kernel(T *__restrict__ P, long rs, long cs, int M, int nb, int R, T *__restrict__ tau,
             T *__restrict__ Tm, unsigned int *bar, double *part, int *info) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *S = reinterpret_cast<T *>(smem_raw);  // R x nb, column c at S + c*R
    // G = V^T V and T (nb x nb each, row-major, ld nb) after the panel rows
    double *Gs = reinterpret_cast<double *>(smem_raw + (((size_t)R * nb * sizeof(T) + 15) & ~(size_t)15));
    double *Ts = Gs + (size_t)nb * nb;
    __shared__ double red[kNbMax + 1];
    __shared__ double rowv[kNbMax + 1];
    __shared__ T wcoef[kNbMax + 1];
    __shared__ double sh_tau, sh_beta, sh_scale;
    __shared__ int sh_fail;

    const int p = blockIdx.x, nP = gridDim.x, tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int r0 = p * R;
    const int nr = max(0, min(M, r0 + R) - r0);
    const int kmax = min(nb, M);
    double *colpart = part;                                    // [2][nP][kNbMax+1]
    double *gpart = part + (size_t)2 * nP * (kNbMax + 1);      // [nP][kNbMax*kNbMax]
    double *rowbuf = gpart + (size_t)nP * kNbMax * kNbMax;     // [2][kNbMax]

    if (tid == 0) sh_fail = 0;
    if (p == 0)
        for (int j = kmax + tid; j < nb; j += blockDim.x) tau[j] = T(0);

    // ---- load the block's rows of the panel into shared memory
    if (cs == 1) {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int c = idx % nb, rr = idx / nb;
            S[(size_t)c * R + rr] = P[(long)(r0 + rr) * rs + c];
        }
    } else {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int rr = idx % nr, c = idx / nr;
            S[(size_t)c * R + rr] = P[(long)(r0 + rr) * rs + (long)c * cs];
        }
    }
    __syncthreads();

    for (int j = 0; j < kmax; ++j) {
        const int buf = j & 1;
        const int nitem = nb - j;  // item 0: ||x||^2; item t > 0: x . a_{j+t}
        const int rr_lo = max(0, j + 1 - r0);
        double *cp = colpart + ((size_t)buf * nP + p) * (kNbMax + 1);
        const T *xj = S + (size_t)j * R;
        for (int it = warp; it < nitem; it += nwarps) {
            if (it == 0) {
                T s = T(0);
                for (int rr = rr_lo + lane; rr < nr; rr += 32) s += xj[rr] * xj[rr];
                s = warp_sum(s);
                if (lane == 0) cp[0] = (double)s;
            } else {
                const T *ac = S + (size_t)(j + it) * R;
                T s = T(0);
                for (int rr = rr_lo + lane; rr < nr; rr += 32) s += xj[rr] * ac[rr];
                s = warp_sum(s);
                if (lane == 0) cp[it] = (double)s;
            }
        }
        if (j >= r0 && j < r0 + nr)
            for (int c = j + tid; c < nb; c += blockDim.x)
                rowbuf[buf * kNbMax + (c - j)] = (double)S[(size_t)c * R + (j - r0)];
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            atomicAdd(bar, 1u);
            if (!spin_until_geq(bar, (unsigned)(j + 1) * (unsigned)nP, info, 32)) sh_fail = 1;
            __threadfence();
        }
        __syncthreads();
        if (sh_fail) return;

        // fixed-order sum of the partials (deterministic across runs): each item is
        // split over `sub` threads whose independent loads are in flight together
        {
            const int sub = nitem <= 32 ? 8 : 4;  // 256 threads cover up to 64 items
            const int it = tid / sub, part = tid % sub;
            double s = 0.0;
            if (it < nitem) {
                const double *base = colpart + (size_t)buf * nP * (kNbMax + 1) + it;
#pragma unroll 8
                for (int q = part; q < nP; q += sub) s += ld_cg(base + (size_t)q * (kNbMax + 1));
            }
            for (int o = sub >> 1; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, sub);
            if (it < nitem && part == 0) {
                red[it] = s;
                rowv[it] = ld_cg(rowbuf + buf * kNbMax + it);
            }
        }
        __syncthreads();
        if (tid == 0) {
            double alpha = rowv[0], xn2 = red[0];
            double tj = 0.0, beta = alpha, scale = 0.0;
            if (xn2 > 0.0) {
                double r = sqrt(alpha * alpha + xn2);
                beta = alpha >= 0.0 ? -r : r;
                tj = (beta - alpha) / beta;
                scale = 1.0 / (alpha - beta);
            }
            sh_tau = tj;
            sh_beta = beta;
            sh_scale = scale;
            if (p == 0) tau[j] = (T)tj;
        }
        __syncthreads();
        const double tj = sh_tau, sc = sh_scale;
        for (int it = 1 + tid; it < nitem; it += blockDim.x) wcoef[it] = (T)(tj * (rowv[it] + sc * red[it]));
        __syncthreads();
        if (tj != 0.0) {
            const T scT = (T)sc;
            for (int rr = rr_lo + tid; rr < nr; rr += blockDim.x) {
                T v = S[(size_t)j * R + rr] * scT;  // reflector entry v_r
                for (int c = j + 1; c < nb; ++c) S[(size_t)c * R + rr] -= v * wcoef[c - j];
                S[(size_t)j * R + rr] = v;
            }
            if (j >= r0 && j < r0 + nr) {  // row j itself: v_j = 1
                for (int c = j + 1 + tid; c < nb; c += blockDim.x) S[(size_t)c * R + (j - r0)] -= wcoef[c - j];
                if (tid == 0) S[(size_t)j * R + (j - r0)] = (T)sh_beta;
            }
        }
        __syncthreads();
    }

    // ---- write the factored rows back
    if (cs == 1) {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int c = idx % nb, rr = idx / nb;
            P[(long)(r0 + rr) * rs + c] = S[(size_t)c * R + rr];
        }
    } else {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int rr = idx % nr, c = idx / nr;
            P[(long)(r0 + rr) * rs + (long)c * cs] = S[(size_t)c * R + rr];
        }
    }

    // ---- partial Gram matrix G(i, k) = v_i . v_k (i < k) over this block's rows.
    // v_c has an implicit 1 in row c and zeros above it.
    double *gp = gpart + (size_t)p * kNbMax * kNbMax;
    for (int it = warp; it < nb * nb; it += nwarps) {
        int i = it / nb, k = it % nb;
        if (i >= k || k >= kmax) continue;
        T s = T(0);
        for (int rr = (k > r0 ? ((k - r0) & ~31) : 0) + lane; rr < nr; rr += 32) {  // rows below k only
            const int r = r0 + rr;
            if (r < k) continue;
            const T vk = (r == k) ? T(1) : S[(size_t)k * R + rr];
            s += S[(size_t)i * R + rr] * vk;  // r >= k > i: stored tail
        }
        s = warp_sum(s);
        if (lane == 0) gp[i * kNbMax + k] = (double)s;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(bar, 1u);

    if (p == 0) {
        if (tid == 0 && !spin_until_geq(bar, (unsigned)(kmax + 1) * (unsigned)nP, info)) sh_fail = 1;
        __syncthreads();
        if (sh_fail) return;
        for (int it = tid; it < nb * nb; it += blockDim.x) {
            int i = it / nb, k = it % nb;
            double s = 0.0;
            if (i < k && k < kmax)
                for (int q = 0; q < nP; ++q) s += ld_cg(gpart + (size_t)q * kNbMax * kNbMax + i * kNbMax + k);
            Gs[i * nb + k] = s;
            Ts[i * nb + k] = 0.0;
        }
        __syncthreads();
        for (int k = 0; k < nb; ++k) {
            double tk = (k < kmax) ? (double)tau[k] : 0.0;
            double t = 0.0;
            if (tid < k)
                for (int q = tid; q < k; ++q) t += Ts[tid * nb + q] * Gs[q * nb + k];
            __syncthreads();
            if (tid < k) Ts[tid * nb + k] = -tk * t;
            if (tid == k) Ts[k * nb + k] = tk;
            __syncthreads();
        }
        for (int it = tid; it < nb * nb; it += blockDim.x) {
            int i = it % nb, k = it / nb;
            Tm[i + (size_t)k * nb] = (T)Ts[i * nb + k];
        }
    }
    // ---- the last block out resets the counters for the next launch
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        unsigned int prev = atomicAdd(bar + 1, 1u);
        if (prev == (unsigned)nP - 1) {
            atomicExch(bar, 0u);
            atomicExch(bar + 1, 0u);
            __threadfence();
        }
    }
}

// ------------------------------------------------------------------ cluster variant
// Same algorithm with the panel spread over one thread-block cluster (up to 16
// blocks on one GPC).  Per column each block pushes its partial sums (and the
// owner block row j) into every block's shared memory over distributed shared
// memory and arrives on every block's mbarrier; a block waits only on its own
// barrier, so the exchange costs one remote write latency instead of a
// cluster-wide barrier plus remote reads.
constexpr int kClusterThreads = 512;

NLA_DEV uint32_t cluster_addr(const void *local, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(tc::smem_u32(local)), "r"(rank));
    return r;
}
NLA_DEV void mbar_arrive_remote(uint32_t cluster_mbar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_mbar) : "memory");
}
NLA_DEV bool mbar_try_wait_cluster(uint64_t *mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(tc::smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// One element global -> shared as an asynchronous copy (completed by cp.async.wait_all).
template <typename T>
NLA_DEV void cp_async_4or8(T *dst_smem, const T *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(tc::smem_u32(dst_smem)), "l"(src),
                 "n"((int)sizeof(T))
                 : "memory");
}

// Dot product of two columns over rows [lo, hi) of the block, four independent
// partial sums per lane, then a warp reduction.
template <typename T>
NLA_DEV T warp_dot(const T *x, const T *y, int lo, int hi, int lane) {
    T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
    int r = lo + lane;
    for (; r + 96 < hi; r += 128) {
        a0 += x[r] * y[r];
        a1 += x[r + 32] * y[r + 32];
        a2 += x[r + 64] * y[r + 64];
        a3 += x[r + 96] * y[r + 96];
    }
    for (; r < hi; r += 32) a0 += x[r] * y[r];
    return warp_sum((a0 + a1) + (a2 + a3));
}

template <typename T>
__global__ void __launch_bounds__(kClusterThreads)
panel_cluster_kernel(T *__restrict__ P, long rs, long cs, int M, int nb, int R, T *__restrict__ tau,
                     T *__restrict__ Tm, int *info) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cg::cluster_group cluster = cg::this_cluster();
    const int p = (int)cluster.block_rank(), nP = (int)cluster.num_blocks();
    T *S = reinterpret_cast<T *>(smem_raw);  // R x nb
    // Per column j the blocks exchange nb partial sums over their rows below j:
    //   item 0            ||x||^2                     (x = column j below row j)
    //   item t in 1..nb-1-j   x . a_{j+t}             (trailing columns)
    //   item nb-j+i, i < j    x . v_i                 (finished reflectors: G(i, j))
    // and the owner of row j pushes row j at the same positions (a_j,j+t and v_i[j]).
    __shared__ T inbox[2][16][kNbMax];  // by column parity and source block
    __shared__ T rowin[2][kNbMax];
    __shared__ T mypart[kNbMax];
    __shared__ T wcoef[kNbMax];
    __shared__ T taus[kNbMax];  // block 0: tau_j, for T after the column loop
    // block 0: T(i, k), i <= k, at Tsh[i + k*nb] and G(i, k) = v_i . v_k, i < k, transposed
    // into the strictly lower part, at Tsh[k + i*nb]
    __shared__ T Tsh[kNbMax * kNbMax];
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ T sh_tau, sh_beta, sh_scale;
    __shared__ int sh_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int r0 = p * R;
    const int nr = max(0, min(M, r0 + R) - r0);
    const int kmax = min(nb, M);
    if (tid == 0) {
        tc::mbar_init(&mbar[0], nP);
        tc::mbar_init(&mbar[1], nP);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh_abort = 0;
    }
    if (p == 0) {
        for (int j = kmax + tid; j < nb; j += blockDim.x) tau[j] = T(0);
        for (int i = tid; i < nb * nb; i += blockDim.x) Tsh[i] = T(0);
    }
    // the block's rows into shared memory: every copy in flight at once (one memory latency)
    if (cs == 1) {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int c = idx % nb, rr = idx / nb;
            cp_async_4or8(&S[(size_t)c * R + rr], &P[(long)(r0 + rr) * rs + c]);
        }
    } else {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int rr = idx % nr, c = idx / nr;
            cp_async_4or8(&S[(size_t)c * R + rr], &P[(long)(r0 + rr) * rs + (long)c * cs]);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    cluster.sync();  // every block's barriers are initialised before the first remote arrive
    for (int j = 0; j < kmax; ++j) {
        const int buf = j & 1;
        const int ntr = nb - j;  // items 0 .. ntr-1: norm and trailing columns; ntr .. nb-1: G(i, j)
        const int rr_lo = max(0, j + 1 - r0);
        const T *xj = S + (size_t)j * R;
        for (int it = warp; it < nb; it += nwarps) {
            const int col = it < ntr ? j + it : it - ntr;
            const T d = warp_dot<T>(xj, S + (size_t)col * R, rr_lo, nr, lane);
            if (lane == 0) mypart[it] = d;
        }
        __syncthreads();
        // push this block's partials (and row j, by its owner) to every block of the cluster
        const int owner = j / R;
        for (int idx = tid; idx < nP * nb; idx += blockDim.x) {
            const int q = idx / nb, it = idx % nb;
            cluster.map_shared_rank(&inbox[buf][p][0], q)[it] = mypart[it];
            if (p == owner) {
                const int col = it < ntr ? j + it : it - ntr;
                cluster.map_shared_rank(&rowin[buf][0], q)[it] = S[(size_t)col * R + (j - r0)];
            }
        }
        __syncthreads();  // all of this block's pushes precede its arrivals
        if (tid < nP) mbar_arrive_remote(cluster_addr(&mbar[buf], tid));
        // warp 0: wait for every block's partials, sum them in a fixed order, form the
        // reflector, the coefficients w_c = tau v . a_c and (block 0) column j of T
        if (warp == 0) {
            if (lane == 0 && !sh_abort) {
                const uint32_t par = (uint32_t)((j >> 1) & 1);
                if (!mbar_try_wait_cluster(&mbar[buf], par)) {
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait_cluster(&mbar[buf], par)) {
                        if (global_ns() - t0 > kSpinBudgetNs) {
                            if (info) atomicExch(info, kInfoTimeout);
                            sh_abort = 1;
                            break;
                        }
                    }
                }
            }
            __syncwarp();  // lane 0's acquire orders the warp's reads below
            const int i0 = lane, i1 = lane + 32;  // nb <= kNbMax = 64
            T s0 = T(0), s1 = T(0), w0 = T(0), w1 = T(0);
#pragma unroll
            for (int q = 0; q < 16; ++q) {  // (the cluster size as a predicate: the loads issue together)
                if (q < nP && i0 < nb) s0 += inbox[buf][q][i0];
                if (q < nP && i1 < nb) s1 += inbox[buf][q][i1];
            }
            if (i0 < nb) w0 = rowin[buf][i0];
            if (i1 < nb) w1 = rowin[buf][i1];
            const T alpha = __shfl_sync(0xffffffffu, w0, 0), xn2 = __shfl_sync(0xffffffffu, s0, 0);
            T tj = T(0), beta = alpha, scale = T(0);
            if (xn2 > T(0)) {
                if constexpr (sizeof(T) == 4) {  // a few ulp, far inside the FP32 path's tolerance
                    const float q = alpha * alpha + xn2;
                    const float r = q * rsqrtf(q);
                    beta = alpha >= 0.f ? -r : r;
                    tj = __fdividef(beta - alpha, beta);
                    scale = __fdividef(1.f, alpha - beta);
                } else {
                    const T r = sqrt(alpha * alpha + xn2);
                    beta = alpha >= T(0) ? -r : r;
                    tj = (beta - alpha) / beta;
                    scale = T(1) / (alpha - beta);
                }
            }
            if (lane == 0) {
                sh_tau = tj;
                sh_beta = beta;
                sh_scale = scale;
                if (p == 0) {
                    tau[j] = tj;
                    taus[j] = tj;
                }
            }
            if (i0 >= 1 && i0 < ntr) wcoef[i0] = tj * (w0 + scale * s0);
            if (i1 < ntr) wcoef[i1] = tj * (w1 + scale * s1);
            if (p == 0) {  // G(i, j) = v_i . v_j = v_i[j] + x . v_i / (alpha - beta), i < j; T after the loop
                if (i0 >= ntr && i0 < nb) Tsh[j + (i0 - ntr) * nb] = w0 + scale * s0;
                if (i1 >= ntr && i1 < nb) Tsh[j + (i1 - ntr) * nb] = w1 + scale * s1;
            }
        }
        __syncthreads();
        const T tj = sh_tau, scT = sh_scale;
        if (tj != T(0)) {
            // columns in blocks of 16: the coefficients in registers, then independent updates
            // (all 16 entries of a row are loaded before any is stored back: the loads then
            // issue together instead of waiting on possibly aliasing stores)
            for (int cb = j + 1; cb < nb; cb += 16) {
                const int nc = min(16, nb - cb);
                T wr[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) wr[u] = u < nc ? wcoef[cb + u - j] : T(0);
                for (int rr = rr_lo + tid; rr < nr; rr += blockDim.x) {
                    T *row = S + (size_t)cb * R + rr;
                    const T v = S[(size_t)j * R + rr] * scT;
                    T xr[16];
#pragma unroll
                    for (int u = 0; u < 16; ++u) xr[u] = u < nc ? row[(size_t)u * R] : T(0);
#pragma unroll
                    for (int u = 0; u < 16; ++u)
                        if (u < nc) row[(size_t)u * R] = xr[u] - v * wr[u];
                }
            }
            for (int rr = rr_lo + tid; rr < nr; rr += blockDim.x) S[(size_t)j * R + rr] *= scT;
            if (p == owner) {
                for (int c = j + 1 + tid; c < nb; c += blockDim.x) S[(size_t)c * R + (j - r0)] -= wcoef[c - j];
                if (tid == 0) S[(size_t)j * R + (j - r0)] = sh_beta;
            }
        }
        __syncthreads();
    }
    if (cs == 1) {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int c = idx % nb, rr = idx / nb;
            P[(long)(r0 + rr) * rs + c] = S[(size_t)c * R + rr];
        }
    } else {
        for (int idx = tid; idx < nr * nb; idx += blockDim.x) {
            int rr = idx % nr, c = idx / nr;
            P[(long)(r0 + rr) * rs + (long)c * cs] = S[(size_t)c * R + rr];
        }
    }
    if (p == 0) {
        // T(0:k, k) = -tau_k T(0:k, 0:k) G(0:k, k), T(k, k) = tau_k -- one warp, column by column
        if (warp == 0) {
            // lane i (and i + 32) forms T(i, kk) = -tau_kk sum_{i <= q < kk} T(i, q) G(q, kk); the
            // q loop is unrolled in blocks of 16 with the range as a predicate
            for (int kk = 0; kk < kmax; ++kk) {
                const T tk = taus[kk];
                for (int i = lane; i < kk; i += 32) {
                    T t = T(0);
                    for (int q0 = i & ~15; q0 < kk; q0 += 16) {
#pragma unroll
                        for (int u = 0; u < 16; ++u) {
                            const int q = q0 + u;
                            const T tv = q < nb ? Tsh[i + q * nb] : T(0), gv = q < nb ? Tsh[kk + q * nb] : T(0);
                            t = (q >= i && q < kk) ? fma(tv, gv, t) : t;  // T(i, q) G(q, kk)
                        }
                    }
                    Tsh[i + kk * nb] = -tk * t;
                }
                if (lane == 0) Tsh[kk + kk * nb] = tk;
                __syncwarp();
            }
        }
        __syncthreads();
        for (int idx = tid; idx < nb * nb; idx += blockDim.x) Tm[idx] = (idx % nb) <= (idx / nb) ? Tsh[idx] : T(0);
    }
    cluster.sync();  // no block leaves while another may still write to its shared memory
}

// Asynchronous store into another block's shared memory that completes as bytes on
// that block's mbarrier (release at cluster scope); addresses from cluster_addr.
NLA_DEV void st_async_remote(uint32_t addr, float v, uint32_t mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(addr), "f"(v),
                 "r"(mbar)
                 : "memory");
}
NLA_DEV void st_async_remote(uint32_t addr, double v, uint32_t mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(addr), "d"(v),
                 "r"(mbar)
                 : "memory");
}
// This block's arrival on its own barrier, announcing the bytes the phase waits for.
NLA_DEV void mbar_arrive_expect_tx(uint64_t *mbar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(mbar)), "r"(bytes)
                 : "memory");
}

// ------------------------------------------------------------------ register-resident cluster variant
// The same factorisation with the panel in registers, a thread owning R rows of one
// column: lane c of a warp holds column c (NB = 32), or column c % 16 of one of two row groups
// (NB = 16), so a warp holds all columns of its rows.  Column j then costs
//   - the owner lanes' x (column j below the diagonal) through the warp's own shared memory,
//     one 128-bit broadcast per four rows: no block barrier, no select;
//   - R multiply-adds for x . a_c, the whole sum over the warp's rows but for one shuffle: c ==
//     j gives ||x||^2, c > j the trailing columns, c < j the Gram matrix of the reflectors;
//   - the warps' sums through shared memory and one block barrier;
//   - with several blocks, every warp pushes the block's sums to its share of the blocks as
//     st.async stores that complete as bytes on the receiver's mbarrier, and every warp
//     waits on that mbarrier itself (no second block barrier);
//   - the reflector's scalars in every warp, and R multiply-adds for the update.
// Finished columns keep x unscaled until the panel is written: the scale of column c is one
// number in its owners' registers.  Row j leaves the registers with column j (it is final then):
// its group moves the rows below up by one, so the pivot row is always register 0.  T is formed by an extra warp of block 0, one column
// behind the others, from the Gram column that warp 0 leaves in shared memory.
//
// Bound: latency of the chain above, per column (FP32 about 0.7 us, of which one exchange
// between blocks is 0.2 us).  The variant this replaced, a thread per row with 16 products per
// thread and column, a 16-value warp reduce-scatter and selects over the columns, took 1.7 us a
// column; panel_reg_launch has the times per panel.

constexpr int kRegWarps = 15;  // row warps per block at most (with the extra one: 128 registers a thread)

// beta, tau and the scale 1 / (alpha - beta) of the reflector of [alpha; x], xn2 = ||x||^2 > 0.
NLA_DEV void panel_scalars(float alpha, float xn2, float &beta, float &tau, float &scale) {
    float r, rs;
    sqrt_and_inverse(fmaf(alpha, alpha, xn2), r, rs);
    beta = alpha >= 0.f ? -r : r;
    tau = fmaf(fabsf(alpha), rs, 1.f);
    scale = inverse(alpha - beta);
}
NLA_DEV void panel_scalars(double alpha, double xn2, double &beta, double &tau, double &scale) {
    const double q = fma(alpha, alpha, xn2);
    if (ordinary(q)) {
        house_tau(alpha, xn2, beta, tau, scale);
        return;
    }
    const double r = sqrt(q);
    beta = alpha >= 0.0 ? -r : r;
    tau = (beta - alpha) / beta;
    scale = 1.0 / (alpha - beta);
}

// Whether the scale of a short vector times an entry of the largest size overflows (above 2^480).  FP32
// does without: a vector below 2^-66 has lost its norm's digits, above 2^-63 nothing overflows
// beside coefficients of 2^62, and the test took 3 % of a panel (FP64: nothing).
NLA_DEV bool too_large(float) { return false; }
NLA_DEV bool too_large(double scale) { return ((unsigned)__double2hiint(scale) & 0x7fffffffu) > 1503u << 20; }

template <typename T, int NB, int R>
__global__ void __launch_bounds__(32 * (kRegWarps + 1), 1)
panel_reg_kernel(T *__restrict__ P, long rs, long cs, int M, int nb, int nw, T *__restrict__ tau,
                 T *__restrict__ Tm, int *info) {
    pdl_wait();
    pdl_trigger();
    static_assert(NB == 16 || NB == 32, "NB");
    constexpr int HV = 32 / NB, kMaxWarps = kRegWarps + 1, VEC = 16 / (int)sizeof(T);
    constexpr int RT = R < NB ? R : NB;  // pivot rows a group can hold
    cg::cluster_group cluster = cg::this_cluster();
    const int p = (int)cluster.block_rank(), nP = (int)cluster.num_blocks();
    __shared__ __align__(16) T xs[kMaxWarps * HV * R];  // x of the current column, per row group
    __shared__ T red[2][kMaxWarps][NB];                 // by column parity: the warps' column sums
    __shared__ T inbox[2][16][NB];                      // the blocks' column sums
    __shared__ T rowj[2][NB], rowin[2][NB];             // row j (block 0's, received)
    // block 0: T(i, k), i <= k, at Tsh[i + k*NB]; G(i, k) = v_i . v_k, i < k, at Gsh[i + k*NB]
    __shared__ T Tsh[NB * NB], Gsh[NB * NB];
    __shared__ T top[NB][NB];  // block 0: the finished rows
    __shared__ T taus[NB];
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ int sh_abort;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int c = lane % NB, group = warp * HV + lane / NB;
    const int gr0 = (p * nw * HV + group) * R;  // first of the thread's rows
    const int kmax = min(nb, M);
    if (tid == 0) {
        // one arrival per phase (this block's expect_tx); the blocks' sums and row j
        // complete it as transaction bytes
        tc::mbar_init(&mbar[0], 1);
        tc::mbar_init(&mbar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        sh_abort = 0;
    }
    if (p == 0) {
        for (int j = kmax + tid; j < nb; j += blockDim.x) tau[j] = T(0);
        for (int i = tid; i < NB * NB; i += blockDim.x) Tsh[i] = T(0);
    }
    const int bar_threads = 32 * (p == 0 ? nw + 1 : nw);
    const auto block_bar = [&] { asm volatile("bar.sync 1, %0;" ::"r"(bar_threads) : "memory"); };
    if (warp < nw) {
        T a[R];
        // a column's rows are contiguous on the QR side: 16-byte vectors where they are aligned
        T *Pc = P + (long)gr0 * rs + (long)c * cs;
        const bool vec = rs == 1 && gr0 + R <= M && c < nb && reinterpret_cast<uintptr_t>(Pc) % 16 == 0;
        if (vec) {
#pragma unroll
            for (int i = 0; i < R; i += VEC) {
                const float4 f = *reinterpret_cast<const float4 *>(Pc + i);
                const T *q = reinterpret_cast<const T *>(&f);
#pragma unroll
                for (int u = 0; u < VEC; ++u) a[i + u] = q[u];
            }
        } else {
#pragma unroll
            for (int i = 0; i < R; ++i) a[i] = gr0 + i < M && c < nb ? Pc[(long)i * rs] : T(0);
        }
        T myscale = T(1);
        if (nP > 1) {
            cluster.sync();  // every block's barriers are initialised before the first remote store
        } else {
            block_bar();
        }
        T *xw = xs + group * R;
        for (int j = 0; j < kmax; ++j) {
            const int buf = j & 1;
            const bool pivot = p == 0 && gr0 <= j && j < gr0 + RT;  // the thread holds row j, in a[0]
            T rv = a[0];
            if (c == j) {
#pragma unroll
                for (int i = 0; i < R; i += VEC) {
                    float4 f;
                    T *q = reinterpret_cast<T *>(&f);
#pragma unroll
                    for (int u = 0; u < VEC; ++u) q[u] = i + u == 0 && pivot ? T(0) : a[i + u];
                    *reinterpret_cast<float4 *>(xw + i) = f;
                }
            }
            if (pivot) rowj[buf][c] = rv;
            __syncwarp();
            T x[R];
#pragma unroll
            for (int i = 0; i < R; i += VEC) {
                const float4 f = *reinterpret_cast<const float4 *>(xw + i);
                const T *q = reinterpret_cast<const T *>(&f);
#pragma unroll
                for (int u = 0; u < VEC; ++u) x[i + u] = q[u];
            }
            T s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = x[u] * a[u];
#pragma unroll
            for (int i = 4; i < R; ++i) s[i % 4] = fma(x[i], a[i], s[i % 4]);
            T sum = (s[0] + s[1]) + (s[2] + s[3]);
            if (HV == 2) sum += __shfl_xor_sync(0xffffffffu, sum, 16);
            if (lane < NB) red[buf][warp][c] = sum;
            block_bar();
            // ---- the block's sums (in every warp, in a fixed order: HV == 2 halves add the even and odd warps)
            sum = T(0);
#pragma unroll
            for (int w = 0; w < kMaxWarps; w += HV) {
                const int v = w + (HV == 2 ? lane / NB : 0);
                sum += v < nw ? red[buf][v][c] : T(0);
            }
            if (HV == 2) sum += __shfl_xor_sync(0xffffffffu, sum, 16);
            if (nP > 1) {
                if (tid == 0) mbar_arrive_expect_tx(&mbar[buf], (uint32_t)((nP + 1) * NB * sizeof(T)));
                const T rj = p == 0 ? rowj[buf][c] : T(0);
                for (int q = warp * HV + lane / NB; q < nP; q += nw * HV) {
                    const uint32_t mb = cluster_addr(&mbar[buf], q);
                    st_async_remote(cluster_addr(&inbox[buf][p][c], q), sum, mb);
                    if (p == 0) st_async_remote(cluster_addr(&rowin[buf][c], q), rj, mb);
                }
                const uint32_t par = (uint32_t)((j >> 1) & 1);
                if (!mbar_try_wait_cluster(&mbar[buf], par)) {
                    const unsigned long long t0 = global_ns();
                    volatile int *vab = &sh_abort;
                    while (!mbar_try_wait_cluster(&mbar[buf], par)) {
                        if (*vab) break;
                        if (global_ns() - t0 > kSpinBudgetNs) {
                            if (info) atomicExch(info, kInfoTimeout);
                            *vab = 1;
                            break;
                        }
                    }
                }
                __syncwarp();
                sum = T(0);
#pragma unroll
                for (int w = 0; w < 16; w += HV) {  // (the cluster size as a predicate: the loads issue together)
                    const int q = w + (HV == 2 ? lane / NB : 0);
                    sum += q < nP ? inbox[buf][q][c] : T(0);
                }
                if (HV == 2) sum += __shfl_xor_sync(0xffffffffu, sum, 16);
                rv = rowin[buf][c];
            } else {
                rv = rowj[buf][c];
            }
            // ---- the reflector
            const T alpha = __shfl_sync(0xffffffffu, rv, j), xn2 = __shfl_sync(0xffffffffu, sum, j);
            T beta = alpha, tj = T(0), scale = T(0);
            if (xn2 > T(0)) panel_scalars(alpha, xn2, beta, tj, scale);
            const T vdot = (rv + scale * sum) * myscale;  // v . a_c (c > j) or G(c, j) = v_c . v_j (c < j)
            const T w = c > j ? tj * vdot : T(0);
            if (c == j && tj != T(0)) myscale = scale;
            if (p == 0 && warp == 0 && lane < NB) {
                if (c < j) Gsh[c + j * NB] = vdot;
                if (c == j) taus[j] = tau[j] = tj;
            }
            // ---- rows below j: a_c -= x (scale w_c); row j: a_c -= w_c, beta in column j
            if (__builtin_expect(too_large(scale), 0)) {  // scale w may overflow: v = x / (alpha - beta) first
#pragma unroll
                for (int i = 0; i < R; ++i) a[i] = fma(x[i] * scale, -w, a[i]);
            } else {
                const T m = -scale * w;
#pragma unroll
                for (int i = 0; i < R; ++i) a[i] = fma(x[i], m, a[i]);
            }
            if (p == 0 && warp * HV * R < NB) {
                if (pivot) top[j][c] = c < j ? rv * myscale : c == j ? beta : rv - w;
#pragma unroll
                for (int i = 0; i < RT; ++i) a[i] = !pivot ? a[i] : i + 1 < RT ? a[i + 1] : T(0);
            }
        }
        if (p == 0) block_bar();  // the last Gram column is there
        // ---- v = x / (alpha - beta) below the diagonal, and the panel back to memory
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] *= myscale;
        if (p == 0 && gr0 < NB) {
            // rows below the last pivot that still sit where they were moved to
            const int gone = min(max(kmax - gr0, 0), RT);
            for (int r = gone; r < RT; ++r) {
                top[gr0 + r][c] = a[0];
#pragma unroll
                for (int i = 0; i + 1 < RT; ++i) a[i] = a[i + 1];
            }
#pragma unroll
            for (int i = 0; i < RT; ++i) a[i] = top[gr0 + i][c];
        }
        if (vec) {
#pragma unroll
            for (int i = 0; i < R; i += VEC) {
                float4 f;
                T *q = reinterpret_cast<T *>(&f);
#pragma unroll
                for (int u = 0; u < VEC; ++u) q[u] = a[i + u];
                *reinterpret_cast<float4 *>(Pc + i) = f;
            }
        } else if (c < nb) {
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (gr0 + i < M) Pc[(long)i * rs] = a[i];
        }
    } else {
        // ---------------- the extra warp: T(0:k, k) = -tau_k T(0:k, 0:k) G(0:k, k), T(k, k) = tau_k
        if (nP > 1) cluster.sync();
        if (p == 0) {
            if (nP == 1) block_bar();
            for (int j = 0; j <= kmax; ++j) {
                block_bar();
                const int k = j - 1;  // its Gram column was left before this barrier
                if (k < 0) continue;
                T t = T(0);
                if (lane < k) {
#pragma unroll 4
                    for (int q = 0; q < k; ++q) t = fma(Tsh[lane + q * NB], Gsh[q + k * NB], t);
                }
                if (lane < k) Tsh[lane + k * NB] = -taus[k] * t;
                if (lane == k) Tsh[k + k * NB] = taus[k];
                __syncwarp();
            }
            for (int idx = lane; idx < nb * nb; idx += 32) {
                const int i = idx % nb, k = idx / nb;
                Tm[idx] = i <= k ? Tsh[i + k * NB] : T(0);
            }
        }
    }
    if (nP > 1) cluster.sync();  // no block leaves while another may still write to its shared memory
}

// NLA_PANEL_CLUSTER: cluster size of the shared-memory variant where it fits (0: the grid
// kernel for every panel); -1 when not set.
static int panel_cluster_forced() {
    static const int force = [] {
        const char *v = getenv("NLA_PANEL_CLUSTER");
        return v ? atoi(v) : -1;
    }();
    return force;
}

// Cluster size and rows per block for an M x nb panel, or 0 if it does not fit one cluster.
// Which cluster sizes the device can schedule (one block per SM at the largest
// dynamic shared memory) is asked once; smaller allocations schedule as well.
struct ClusterCaps {
    size_t max_dyn = 0;
    bool sched[5] = {false, false, false, false, false};  // cluster sizes 1, 2, 4, 8, 16
};

template <typename T>
static int cluster_plan(int M, int nb, int &R, size_t &dyn) {
    static PerDeviceValue<ClusterCaps> caps_dev;
    const ClusterCaps caps = caps_dev.get([] {
        ClusterCaps c;
        int optin = 0;
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, std::max(current_device(), 0));
        cudaFuncAttributes fa;
        if (cudaFuncGetAttributes(&fa, panel_cluster_kernel<T>) == cudaSuccess && (size_t)optin > fa.sharedSizeBytes)
            c.max_dyn = (size_t)optin - fa.sharedSizeBytes;
        if (cudaFuncSetAttribute(panel_cluster_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.max_dyn) !=
                cudaSuccess ||
            cudaFuncSetAttribute(panel_cluster_kernel<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
                cudaSuccess)
            c.max_dyn = 0;
        for (int k = 0; k < 5 && c.max_dyn > 0; ++k) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1u << k);
            cfg.blockDim = dim3(kClusterThreads);
            cfg.dynamicSmemBytes = c.max_dyn;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 1u << k;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int ncl = 0;
            c.sched[k] = cudaOccupancyMaxActiveClusters(&ncl, panel_cluster_kernel<T>, &cfg) == cudaSuccess && ncl >= 1;
        }
        cudaGetLastError();
        return c;
    });
    const size_t max_dyn = caps.max_dyn;
    const bool *sched = caps.sched;
    int k0 = 0;
    while (k0 < 4 && (1 << k0) * kPanelRowsTarget < M) ++k0;  // smallest size with <= 256 rows per block
    const int force = panel_cluster_forced();
    if (force == 0) return 0;
    int best = 0;
    for (int k = 0; k < 5; ++k) {
        if (!sched[k]) continue;
        if (force > 0 && (1 << k) != force) continue;
        const int C = 1 << k;
        const int r = (M + C - 1) / C;
        const size_t d = (size_t)r * nb * sizeof(T);
        if (d > max_dyn) continue;
        best = C;
        R = r;
        dyn = d;
        if (k >= k0) break;  // the smallest fitting size at or above the target, else the largest that fits
    }
    return best;
}

// Register-resident panel: nb <= 32 columns and as many rows as 16 blocks hold; otherwise
// cudaErrorNotSupported.  NLA_PANEL_REG=0 keeps the shared-memory variant.
// Blocks of four row warps (one per SM sub-partition) up to 16 blocks, taller blocks above that.
template <typename T, int NB, int R>
cudaError_t panel_reg_launch_nb(T *P, long rs, long cs, int M, int nb, int max_warps, T *tau, T *Tm, int *info,
                                cudaStream_t st) {
    constexpr int per_warp = 32 / NB * R;  // rows
    const int warps = (M + per_warp - 1) / per_warp;
    int C = 1;
    while (C < 16 && C * 4 < warps) C *= 2;
    // (block 0 holds every pivot row)
    const int nw = std::max((warps + C - 1) / C, C > 1 ? (NB + per_warp - 1) / per_warp : 1);
    if (nw > max_warps) return cudaErrorNotSupported;
    static PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(panel_reg_kernel<T, NB, R>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cudaGetLastError();
    });
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(32 * (nw + 1));
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, panel_reg_kernel<T, NB, R>, P, rs, cs, M, nb, nw, tau, Tm, info);
}

// Rows per thread.  FP32: 16 while 16 blocks of eight warps hold them (4,096 rows at 16
// columns), then 32 (us per panel at 16 columns, R = 16 / 32: 1,024 rows 15.5 / 15.9, 3,001 rows
// 17.2 / 18.2, 8,192 rows with R = 32 and 8 warps 19.4; 16 columns of 8,192 rows took 32 before).
// FP64: 16 at 16 columns (2,048 rows: 57 us against 160 before), 8 at 32 columns while they fit
// (256 rows: 104 us, 117 with 16, 355 before); its chain is the FP64 pipe's, so spreading the
// rows over more SMs matters more than the exchange.
template <typename T>
cudaError_t panel_reg_launch(T *P, long rs, long cs, int M, int nb, T *tau, T *Tm, int *info, cudaStream_t st) {
    static const bool on = [] {
        const char *v = getenv("NLA_PANEL_REG");
        return !v || atoi(v) != 0;
    }();
    if (!on || nb > 32) return cudaErrorNotSupported;
    cudaError_t e = cudaErrorNotSupported;
    if constexpr (sizeof(T) == 4) {
        e = nb <= 16 ? panel_reg_launch_nb<T, 16, 16>(P, rs, cs, M, nb, 8, tau, Tm, info, st)
                     : panel_reg_launch_nb<T, 32, 16>(P, rs, cs, M, nb, 8, tau, Tm, info, st);
        if (e == cudaErrorNotSupported)
            e = nb <= 16 ? panel_reg_launch_nb<T, 16, 32>(P, rs, cs, M, nb, kRegWarps, tau, Tm, info, st)
                         : panel_reg_launch_nb<T, 32, 32>(P, rs, cs, M, nb, kRegWarps, tau, Tm, info, st);
    } else if (nb <= 16) {
        e = panel_reg_launch_nb<T, 16, 16>(P, rs, cs, M, nb, kRegWarps, tau, Tm, info, st);
    } else {
        e = panel_reg_launch_nb<T, 32, 8>(P, rs, cs, M, nb, 4, tau, Tm, info, st);
        if (e == cudaErrorNotSupported) e = panel_reg_launch_nb<T, 32, 16>(P, rs, cs, M, nb, kRegWarps, tau, Tm, info, st);
    }
    return e;
}

template <typename T>
cudaError_t panel_factor(T *P, long rs, long cs, int M, int nb, T *tau, T *Tm, const PanelCtl &ctl,
                         cudaStream_t st) {
    if (M <= 0 || nb <= 0) return cudaSuccess;
    if (nb > kNbMax) return cudaErrorInvalidValue;
    if (panel_cluster_forced() < 0) {  // preferred: rows in registers, one thread-block cluster
        cudaError_t e = panel_reg_launch<T>(P, rs, cs, M, nb, tau, Tm, ctl.info, st);
        if (e == cudaSuccess) return e;
        cudaGetLastError();  // not available for this shape: shared-memory variant
    }
    {
        int R = 0;
        size_t dyn = 0;
        const int C = cluster_plan<T>(M, nb, R, dyn);
        if (C > 0) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(C);
            cfg.blockDim = dim3(kClusterThreads);
            cfg.dynamicSmemBytes = dyn;
            cfg.stream = st;
            cudaLaunchAttribute attr[2];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = C;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            attr[1].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = attr;
            cfg.numAttrs = pdl_enabled() ? 2 : 1;
            cudaError_t e = cudaLaunchKernelEx(&cfg, panel_cluster_kernel<T>, P, rs, cs, M, nb, R, tau, Tm, ctl.info);
            if (e == cudaSuccess) return e;
            cudaGetLastError();  // fall back to the grid-wide version
        }
    }
    static PerDeviceValue<size_t> grid_dyn;
    const size_t max_dyn = grid_dyn.get([] {
        int optin = 0;
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, std::max(current_device(), 0));
        cudaFuncAttributes fa;
        size_t md = 0;
        if (cudaFuncGetAttributes(&fa, panel_kernel<T>) == cudaSuccess)
            md = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
        cudaFuncSetAttribute(panel_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)md);
        cudaGetLastError();
        return md;
    });
    const int maxP = panel_max_ctas();
    int Pn = std::max(1, std::min(maxP, (M + kPanelRowsTarget - 1) / kPanelRowsTarget));
    const size_t gt_bytes = (size_t)2 * nb * nb * sizeof(double) + 16;
    if (max_dyn <= gt_bytes) return cudaErrorInvalidConfiguration;
    size_t rows_fit = (max_dyn - gt_bytes) / ((size_t)nb * sizeof(T));
    if (rows_fit == 0) return cudaErrorInvalidConfiguration;
    int R = (M + Pn - 1) / Pn;
    if ((size_t)R > rows_fit) {
        Pn = (int)((M + rows_fit - 1) / rows_fit);
        if (Pn > maxP) return cudaErrorInvalidConfiguration;
        R = (M + Pn - 1) / Pn;
    }
    Pn = (M + R - 1) / R;  // no empty blocks
    size_t dyn = (((size_t)R * nb * sizeof(T) + 15) & ~(size_t)15) + (size_t)2 * nb * nb * sizeof(double);

    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(Pn);
    cfg.blockDim = dim3(kPanelThreads);
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, panel_kernel<T>, P, rs, cs, M, nb, R, tau, Tm, ctl.bar, ctl.part,
                              ctl.info);
}

template cudaError_t panel_factor<double>(double *, long, long, int, int, double *, double *,
                                          const PanelCtl &, cudaStream_t);
template cudaError_t panel_factor<float>(float *, long, long, int, int, float *, float *,
                                         const PanelCtl &, cudaStream_t);

}  // namespace nla
