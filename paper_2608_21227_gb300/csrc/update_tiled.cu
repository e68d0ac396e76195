// update_tiled.cu -- register-tiled trailing update (Algorithm 2, both sides),
// the main FP64 / FP32 SIMT path.  Same three steps as update.cu
// (W = V^T X_strip, W <- T^T W, X_strip -= V W'), with the work of each step
// tiled for the FMA pipes:
//
//   threads = (w/4 column groups) x (nb/R reflector groups); thread (cg, rg)
//   owns 4 strip columns (QR side) / 4 strip rows (LQ side) and R reflectors.
//   Step 1: for every staged row (column) of X the thread does R x 4 FMAs from
//           one 128-bit shared load of X and R reflector values that the whole
//           warp shares (broadcast).
//   Step 3: the thread updates sub-blocks of A x 4 entries of the staged X
//           tile (A = 4; 2 or 1 where FP64 needs more warps); per reflector
//           one 128-bit load of W' and one broadcast load of V (128-bit for
//           A = 4; stored k-major) feed 4 A FMAs.
//
// Two launches per side keep every SM busy: step 1 runs on a grid of (strips) x
// (splits of the long dimension) and the last block of each strip -- chosen by
// an atomic ticket, so nothing waits -- reduces the partial sums and applies T (step 2); step 3 runs on a full 2-D
// grid of (tile x strip) blocks.
//
// QR side: X tiles are staged row-major with an XOR swizzle of the 4-column
// group by (row & 7), so that both the column-wise staging stores and the
// row-wise 128-bit reads are free of bank conflicts.  LQ side: X tiles are
// staged column-major (the strip rows are contiguous), which needs no swizzle.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace nla {

constexpr size_t kTiledSmemLimit = 226 * 1024;  // dynamic bytes; the kernels' static shared memory fits in the rest

template <typename T>
struct Vec4;
template <>
struct Vec4<float> {
    NLA_DEV static void ld(const float *p, float v[4]) {
        float4 q = *reinterpret_cast<const float4 *>(p);
        v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    }
    NLA_DEV static void st(float *p, const float v[4]) { *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]); }
};
template <>
struct Vec4<double> {
    NLA_DEV static void ld(const double *p, double v[4]) {
        double2 a = *reinterpret_cast<const double2 *>(p), b = *reinterpret_cast<const double2 *>(p + 2);
        v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    }
    NLA_DEV static void st(double *p, const double v[4]) {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
        *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
    }
};

// One element from global to shared memory, asynchronously.
template <typename T>
NLA_DEV void cp_async1(T *dst, const T *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(sizeof(T)) : "memory");
}
NLA_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
NLA_DEV void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Swizzled position of X(r, c) in a row-major tile with w columns.
NLA_DEV int swz(int r, int c, int w) { return r * w + ((((c >> 2) ^ (r & 7))) << 2) + (c & 3); }

constexpr int kMaxSplit = 8;

// Step 3, and what a configuration is checked by: one tile of th lines, V's rows and W.  (Step 1
// takes two tiles of th / 2 lines in the same room.)
size_t tiled_smem(int side, int elem, int nb, int th, int w) {
    (void)side;
    return (size_t)elem * ((size_t)th * w + (size_t)th * (nb + 4) + (size_t)nb * w);
}
// Step 1: elements before W (nb x w): two X and V tiles, later T.
__host__ NLA_DEV int tiled_w_offset(int nb, int th, int w) {
    const int tiles = 2 * th * (w + nb + 4), t = (nb * nb + 3) / 4 * 4;
    return tiles > t ? tiles : t;
}

// R = reflectors per thread, or 0 if (nb, threads, cpb, tile, unroll) do not tile.
int tiled_r(int nb, const UpdCfg &c) {
    if (nb < 4 || nb > 64 || nb % 4) return 0;
    if (c.threads < 32 || c.threads > 1024 || c.threads % 32) return 0;
    if (c.cpb != 1 && c.cpb != 2 && c.cpb != 4 && c.cpb != 8) return 0;  // swizzle needs 2^k column groups
    if (c.unroll != 1 && c.unroll != 2 && c.unroll != 4) return 0;
    const int w = 32 * c.cpb, ncg = w / 4;
    if (c.threads % ncg) return 0;
    const int nrg = c.threads / ncg;
    if (nb % nrg) return 0;
    const int R = nb / nrg;
    if (R != 1 && R != 2 && R != 4 && R != 8) return 0;
    if (c.tile < 4 || c.tile > 256 || c.tile % (4 * nrg)) return 0;  // step-3 rows per thread: multiple of 4
    return R;
}

// -------------------------------------------------------------------- QR side
// Step 1 (+ step 2 in the last block of each strip): block (cb, s) accumulates
// the partial W = V^T X over rows [s*Ms, (s+1)*Ms) of strip cb and stores it;
// the last block of the strip to finish (atomic ticket) sums the S partials,
// applies T^T and stores W' for step 3.
template <typename T, int R, int U>
__global__ void left_w_kernel(const T *__restrict__ X, long ldx, int M, int N, const T *__restrict__ V, long ldv,
                              int nb, const T *__restrict__ Tm, int th, int w, int Ms, T *part, T *fin,
                              unsigned int *tickets) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int sh_last;
    const int ldv_s = nb + 4;
    T *Xs = reinterpret_cast<T *>(smem_raw);  // 2 x th x w, swizzled
    T *Vs = Xs + (size_t)2 * th * w;             // 2 x th x (nb+4) row-major
    T *Ws = reinterpret_cast<T *>(smem_raw) + tiled_w_offset(nb, th, w);  // nb x w row-major
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ncg = w >> 2, cg = tid % ncg, rg = tid / ncg;
    const int c0 = blockIdx.x * w, wc = min(w, N - c0);
    const int s = blockIdx.y, S = gridDim.y;
    const int rbeg = s * Ms, rend = min(M, rbeg + Ms);

    T acc[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    // two half tiles in the room of one: the next lands while this one is multiplied (one block
    // often holds an SM; 2048 x 2048 FP64 SVD 65.6 -> 63.5 ms)
    const auto stage = [&](int r0, int buf) {
        const int rows = min(th, rend - r0);
        T *const xs = Xs + buf * th * w, *const vs = Vs + buf * th * ldv_s;
        for (int idx = tid; idx < th * w; idx += nt) {
            const int r = idx % th, c = idx / th;
            T *const d = xs + swz(r, c, w);
            if (r < rows && c < wc)
                cp_async1(d, X + (r0 + r) + (long)(c0 + c) * ldx);
            else
                *d = T(0);
        }
        for (int idx = tid; idx < th * nb; idx += nt) {
            const int r = idx % th, k = idx / th, gr = r0 + r;
            T *const d = vs + r * ldv_s + k;
            if (r < rows && gr > k)
                cp_async1(d, V + gr + (long)k * ldv);
            else
                *d = r < rows && gr == k ? T(1) : T(0);
        }
        cp_async_commit();
    };
    if (rbeg < rend) stage(rbeg, 0);
    for (int r0 = rbeg, buf = 0; r0 < rend; r0 += th, buf ^= 1) {
        const int rows = min(th, rend - r0);
        if (r0 + th < rend) {
            stage(r0 + th, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const T *const xs = Xs + buf * th * w, *const vs = Vs + buf * th * ldv_s;
#pragma unroll U
        for (int r = 0; r < rows; ++r) {
            T x[4], v[R];
            Vec4<T>::ld(xs + swz(r, 4 * cg, w), x);
            const T *vr = vs + r * ldv_s + R * rg;
            if constexpr (R % 4 == 0) {
#pragma unroll
                for (int i = 0; i < R; i += 4) Vec4<T>::ld(vr + i, v + i);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) v[i] = vr[i];
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += v[i] * x[j];
        }
        __syncthreads();
    }
    // store the partial W (nb x N slab of this split)
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = 4 * cg + j;
            if (c < wc) part[((size_t)s * nb + R * rg + i) * N + c0 + c] = acc[i][j];
        }
    __threadfence();
    __syncthreads();
    if (tid == 0) sh_last = atomicAdd(&tickets[blockIdx.x], 1u) == (unsigned)(S - 1);
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    // ---- step 2 (last block of the strip): sum of the partials, times T.  A sum's S loads are in
    // flight together and T waits in shared memory.
    T *const Ts = reinterpret_cast<T *>(smem_raw);  // nb x nb, where the tiles were
#pragma unroll 1
    for (int idx = tid; idx < nb * w; idx += nt) {
        const int c = idx % w, k = idx / w;
        T p[kMaxSplit], sum = T(0);
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q)
            p[q] = q < S && c < wc ? __ldcg(part + ((size_t)q * nb + k) * N + c0 + c) : T(0);
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q) sum += p[q];
        Ws[k * w + c] = sum;
    }
    for (int idx = tid; idx < nb * nb; idx += nt) Ts[idx] = Tm[idx];
    __syncthreads();
    const int nrg = nt / ncg;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int kk = rg + nrg * i;  // (interleaved: term counts grow with kk)
        T a[4] = {};
#pragma unroll 2
        for (int k = 0; k <= kk; ++k) {
            const T t = Ts[k + kk * nb];
            T wv[4];
            Vec4<T>::ld(Ws + k * w + 4 * cg, wv);
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] += t * wv[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * cg + j < wc) fin[(size_t)kk * N + c0 + 4 * cg + j] = a[j];
    }
    if (tid == 0) tickets[blockIdx.x] = 0u;  // ready for the next launch
}

// Step 3: block (cb, rb) updates the th x w tile X(rb, cb) -= V(rb, :) W'(:, cb).
template <typename T, int U, int A>
__global__ void left_x_kernel(T *__restrict__ X, long ldx, int M, int N, const T *__restrict__ V, long ldv, int nb,
                              int th, int w, const T *__restrict__ fin) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *Xs = reinterpret_cast<T *>(smem_raw);  // th x w, swizzled
    T *Vs = Xs + (size_t)th * w;             // nb x th, k-major
    T *Ws = Vs + (size_t)th * (nb + 4);      // nb x w
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ncg = w >> 2, cg = tid % ncg, rg = tid / ncg, nrg = nt / ncg;
    const int c0 = blockIdx.x * w, wc = min(w, N - c0);
    const int r0 = blockIdx.y * th, rows = min(th, M - r0);
    for (int idx = tid; idx < th * w; idx += nt) {
        int r = idx % th, c = idx / th;
        Xs[swz(r, c, w)] = (r < rows && c < wc) ? X[(r0 + r) + (long)(c0 + c) * ldx] : T(0);
    }
    for (int idx = tid; idx < th * nb; idx += nt) {
        int r = idx % th, k = idx / th, gr = r0 + r;
        T v = T(0);
        if (r < rows) v = gr > k ? V[gr + (long)k * ldv] : (gr == k ? T(1) : T(0));
        Vs[k * th + r] = v;
    }
    for (int idx = tid; idx < nb * w; idx += nt) {
        int c = idx % w, k = idx / w;
        Ws[k * w + c] = c < wc ? fin[(size_t)k * N + c0 + c] : T(0);
    }
    __syncthreads();
    const int rpt = th / nrg;  // rows per thread, a multiple of A
    for (int rb = rg * rpt; rb < rg * rpt + rpt; rb += A) {
        T sacc[A][4];
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int j = 0; j < 4; ++j) sacc[a][j] = T(0);
#pragma unroll U
        for (int k = 0; k < nb; ++k) {
            T v[A], wv[4];
            if constexpr (A == 4) {
                Vec4<T>::ld(Vs + k * th + rb, v);
            } else {
#pragma unroll
                for (int a = 0; a < A; ++a) v[a] = Vs[k * th + rb + a];
            }
            Vec4<T>::ld(Ws + k * w + 4 * cg, wv);
#pragma unroll
            for (int a = 0; a < A; ++a)
#pragma unroll
                for (int j = 0; j < 4; ++j) sacc[a][j] += v[a] * wv[j];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            T *p = Xs + swz(rb + a, 4 * cg, w);
            T x[4];
            Vec4<T>::ld(p, x);
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] -= sacc[a][j];
            Vec4<T>::st(p, x);
        }
    }
    __syncthreads();
    for (int idx = tid; idx < th * w; idx += nt) {
        int r = idx % th, c = idx / th;
        if (r < rows && c < wc) X[(r0 + r) + (long)(c0 + c) * ldx] = Xs[swz(r, c, w)];
    }
}

// -------------------------------------------------------------------- LQ side
// Step 1 (+2): block (rb, s) accumulates Y = X V over columns [s*Ns, (s+1)*Ns)
// of the h-row strip rb; the last block sums the partials and stores Y' = Y T.
// (bounds: 64 lines / 4 times 64 reflectors / R, the widest block that a configuration may ask for)
template <typename T, int R, int U>
__global__ void __launch_bounds__(R < 8 ? 1024 : 512)
    right_w_kernel(const T *__restrict__ X, long ldx, int M, int N, const T *__restrict__ Vt, long ldvt,
                               int nb, const T *__restrict__ Tm, int th, int h, int Ns, T *part, T *fin,
                               unsigned int *tickets) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int sh_last;
    const int ldv_s = nb + 4;
    T *Xs = reinterpret_cast<T *>(smem_raw);  // 2 x th columns x h rows, column-major
    T *Vs = Xs + (size_t)2 * th * h;             // 2 x th x (nb+4): row c = V(c, :)
    T *Ys = reinterpret_cast<T *>(smem_raw) + tiled_w_offset(nb, th, h);  // nb x h
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ncg = h >> 2, cg = tid % ncg, rg = tid / ncg;
    const int i0 = blockIdx.x * h, hr = min(h, M - i0);
    const int s = blockIdx.y, S = gridDim.y;
    const int cbeg = s * Ns, cend = min(N, cbeg + Ns);

    T acc[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    const auto stage = [&](int cb, int buf) {
        const int cols = min(th, cend - cb);
        T *const xs = Xs + buf * th * h, *const vs = Vs + buf * th * ldv_s;
        for (int idx = tid; idx < th * h; idx += nt) {
            const int i = idx % h, c = idx / h;
            if (i < hr && c < cols)
                cp_async1(xs + c * h + i, X + (i0 + i) + (long)(cb + c) * ldx);
            else
                xs[c * h + i] = T(0);
        }
        for (int idx = tid; idx < th * nb; idx += nt) {
            const int k = idx % nb, c = idx / nb, gc = cb + c;
            T *const d = vs + c * ldv_s + k;
            if (c < cols && gc > k)
                cp_async1(d, Vt + k + (long)gc * ldvt);
            else
                *d = c < cols && gc == k ? T(1) : T(0);
        }
        cp_async_commit();
    };
    if (cbeg < cend) stage(cbeg, 0);
    for (int cb = cbeg, buf = 0; cb < cend; cb += th, buf ^= 1) {
        const int cols = min(th, cend - cb);
        if (cb + th < cend) {
            stage(cb + th, buf ^ 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        __syncthreads();
        const T *const xs = Xs + buf * th * h, *const vs = Vs + buf * th * ldv_s;
#pragma unroll U
        for (int c = 0; c < cols; ++c) {
            T x[4], v[R];
            Vec4<T>::ld(xs + c * h + 4 * cg, x);
            const T *vc = vs + c * ldv_s + R * rg;
            if constexpr (R % 4 == 0) {
#pragma unroll
                for (int i = 0; i < R; i += 4) Vec4<T>::ld(vc + i, v + i);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) v[i] = vc[i];
            }
#pragma unroll
            for (int i = 0; i < R; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] += v[i] * x[j];
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int r = 4 * cg + j;
            if (r < hr) part[((size_t)s * nb + R * rg + i) * M + i0 + r] = acc[i][j];
        }
    __threadfence();
    __syncthreads();
    if (tid == 0) sh_last = atomicAdd(&tickets[blockIdx.x], 1u) == (unsigned)(S - 1);
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    // ---- step 2 (last block of the strip): sum of the partials, times T.  A sum's S loads are in
    // flight together and T waits in shared memory.
    T *const Ts = reinterpret_cast<T *>(smem_raw);  // nb x nb, where the tiles were
#pragma unroll 1
    for (int idx = tid; idx < nb * h; idx += nt) {
        const int c = idx % h, k = idx / h;
        T p[kMaxSplit], sum = T(0);
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q)
            p[q] = q < S && c < hr ? __ldcg(part + ((size_t)q * nb + k) * M + i0 + c) : T(0);
#pragma unroll
        for (int q = 0; q < kMaxSplit; ++q) sum += p[q];
        Ys[k * h + c] = sum;
    }
    for (int idx = tid; idx < nb * nb; idx += nt) Ts[idx] = Tm[idx];
    __syncthreads();
    const int nrg = nt / ncg;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int kk = rg + nrg * i;  // (interleaved: term counts grow with kk)
        T a[4] = {};
#pragma unroll 2
        for (int k = 0; k <= kk; ++k) {
            const T t = Ts[k + kk * nb];
            T yv[4];
            Vec4<T>::ld(Ys + k * h + 4 * cg, yv);
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] += t * yv[j];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (4 * cg + j < hr) fin[(size_t)kk * M + i0 + 4 * cg + j] = a[j];
    }
    if (tid == 0) tickets[blockIdx.x] = 0u;
}

// Step 3: block (rb, cbk) updates the h x th tile X(rb, cbk) -= Y'(rb, :) V(cbk, :)^T.
template <typename T, int U, int A>
__global__ void right_x_kernel(T *__restrict__ X, long ldx, int M, int N, const T *__restrict__ Vt, long ldvt, int nb,
                               int th, int h, const T *__restrict__ fin) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *Xs = reinterpret_cast<T *>(smem_raw);  // th columns x h rows
    T *Vs = Xs + (size_t)th * h;             // nb x th, k-major
    T *Ys = Vs + (size_t)th * (nb + 4);      // nb x h
    const int tid = threadIdx.x, nt = blockDim.x;
    const int ncg = h >> 2, cg = tid % ncg, rg = tid / ncg, nrg = nt / ncg;
    const int i0 = blockIdx.x * h, hr = min(h, M - i0);
    const int cb = blockIdx.y * th, cols = min(th, N - cb);
    for (int idx = tid; idx < th * h; idx += nt) {
        int i = idx % h, c = idx / h;
        Xs[c * h + i] = (i < hr && c < cols) ? X[(i0 + i) + (long)(cb + c) * ldx] : T(0);
    }
    for (int idx = tid; idx < th * nb; idx += nt) {
        int k = idx % nb, c = idx / nb, gc = cb + c;
        T v = T(0);
        if (c < cols) v = gc > k ? Vt[k + (long)gc * ldvt] : (gc == k ? T(1) : T(0));
        Vs[k * th + c] = v;
    }
    for (int idx = tid; idx < nb * h; idx += nt) {
        int i = idx % h, k = idx / h;
        Ys[k * h + i] = i < hr ? fin[(size_t)k * M + i0 + i] : T(0);
    }
    __syncthreads();
    const int cpt = th / nrg;
    for (int cbl = rg * cpt; cbl < rg * cpt + cpt; cbl += A) {
        T sacc[A][4];  // [column a][row j]
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
            for (int j = 0; j < 4; ++j) sacc[a][j] = T(0);
#pragma unroll U
        for (int k = 0; k < nb; ++k) {
            T v[A], yv[4];
            if constexpr (A == 4) {
                Vec4<T>::ld(Vs + k * th + cbl, v);
            } else {
#pragma unroll
                for (int a = 0; a < A; ++a) v[a] = Vs[k * th + cbl + a];
            }
            Vec4<T>::ld(Ys + k * h + 4 * cg, yv);
#pragma unroll
            for (int a = 0; a < A; ++a)
#pragma unroll
                for (int j = 0; j < 4; ++j) sacc[a][j] += v[a] * yv[j];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            T *p = Xs + (cbl + a) * h + 4 * cg;
            T x[4];
            Vec4<T>::ld(p, x);
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] -= sacc[a][j];
            Vec4<T>::st(p, x);
        }
    }
    __syncthreads();
    for (int idx = tid; idx < th * h; idx += nt) {
        int i = idx % h, c = idx / h;
        if (i < hr && c < cols) X[(i0 + i) + (long)(cb + c) * ldx] = Xs[c * h + i];
    }
}

// -------------------------------------------------------------------- dispatch
// partial slabs, the projection's W' / Y', and room for the mixed path's line exponents
size_t tiled_scratch_elems(int M, int N) { return (size_t)(kMaxSplit + 2) * 64 * (size_t)std::max(std::max(M, N), 1); }
size_t tiled_tickets(int M, int N) { return (size_t)std::max(M, N) / 32 + 2; }

// number of splits of the long dimension L for `nblk` strips: about three waves
static int split_count(int L, int th, int nblk) {
    int S = (3 * device_sm_count() + nblk - 1) / std::max(nblk, 1);
    S = std::max(1, std::min({S, kMaxSplit, (L + th - 1) / th}));
    return S;
}

// The blocks of one launch: strips of w lines and tiles of th; step 1: R reflectors a thread and
// S splits of Ms entries; step 3: A lines of the tile at a time a thread.
struct Shape {
    int threads, w, th, R, S, Ms, A;
};

// FP64: an SM's pipe (a warp's FMA holds a quarter of it for 64 cycles) is the bound, not memory,
// so a launch lasts as long as the quarter with the most warps: ceil(blocks / SMs) blocks, their
// warps over four quarters, and a warp's FMAs.  The configuration's block is the largest one; it is
// halved along the strip (and, in step 3, along the tile), with all or half of its threads, where
// this count says that more SMs or quarters work.  Step 1 takes the number of splits and their
// length (whole 64-byte lines) by it too.  A halving has to win 2 %: smaller blocks stage V more
// often.  FP32 is bound by memory and keeps its tuned blocks and splits.  Updates of a whole
// reduction, 64 x 64 blocks with three waves of splits before: 2048 x 2048, band 16, 35.9 -> 28.3 ms
// (21.6 at the pipe's rate); 256 x 256, band 32, 1.60 -> 0.70 ms.
static double quarter_warps(long blocks, int threads) {
    const long sm = device_sm_count();
    return (double)(((blocks + sm - 1) / sm * (threads / 32) + 3) / 4);
}

template <typename T>
static Shape step1_shape(int side, int nb, int R, const UpdCfg &c, int strip, int len) {
    Shape best{c.threads, 32 * c.cpb, c.tile, R, 1, 0, 4};
    if constexpr (sizeof(T) == 4) {
        best.S = split_count(len, c.tile, (strip + best.w - 1) / best.w);
        best.Ms = ((len + best.S - 1) / best.S + c.tile - 1) / c.tile * c.tile;
        best.S = (len + best.Ms - 1) / best.Ms;
        return best;
    }
    double least = 0;
    for (int h = 1; h <= 2; ++h)
        for (int ht = 1; ht <= 2; ++ht) {
            const int w = 32 * c.cpb / h, threads = c.threads / ht;
            if (w < 32 || threads % 32 || threads % (w / 4) || nb % (threads / (w / 4))) continue;
            const int r = nb / (threads / (w / 4));
            if ((r != 1 && r != 2 && r != 4 && r != 8) || r > R || threads > tiled_max_threads(side, 8, r, c.unroll)) continue;
            for (int S = 1; S <= kMaxSplit; ++S) {
                const int Ms = ((len + S - 1) / S + 7) / 8 * 8, used = (len + Ms - 1) / Ms;
                const double cost = quarter_warps((long)((strip + w - 1) / w) * used, threads) * Ms * r *
                                    (1 + 0.02 * (h * ht - 1));
                if (best.Ms == 0 || cost < least)
                    best = Shape{threads, w, std::min(c.tile, Ms), r, used, Ms, 4}, least = cost;
            }
        }
    return best;
}

template <typename T>
static Shape step3_shape(const UpdCfg &c, int strip, int len) {
    Shape best{c.threads, 32 * c.cpb, c.tile, 0, 0, 0, 4};
    if constexpr (sizeof(T) == 4) return best;
    double least = 0;
    for (int hw = 1; hw <= 2; ++hw)
        for (int ht = 1; ht <= 2; ++ht)
            for (int hn = 1; hn <= hw * ht; hn *= 2) {
                const int w = 32 * c.cpb / hw, th = c.tile / ht, threads = c.threads / hn;
                if (w < 32 || c.tile % ht || threads % 32 || threads % (w / 4)) continue;
                const int nrg = threads / (w / 4);
                if (th % nrg || th / nrg > c.tile * 8 * c.cpb / c.threads) continue;
                const int rpt = th / nrg, A = rpt % 4 == 0 ? 4 : rpt % 2 == 0 ? 2 : 1;
                const long blocks = (long)((strip + w - 1) / w) * ((len + th - 1) / th);
                const double cost = quarter_warps(blocks, threads) * rpt * (1 + 0.02 * (hw * ht - 1));
                if (least == 0 || cost < least) best = Shape{threads, w, th, 0, 0, 0, A}, least = cost;
            }
    return best;
}

template <typename T, int U, int R>
static cudaError_t run_step1(int side, const T *X, long ldx, int M, int N, const T *V, long ldv, int nb, const T *Tm,
                             const Shape &a, T *part, T *fin, unsigned int *tickets, cudaStream_t st) {
    const int th = a.th / 2;  // (two tiles in the room of one; a tile is a multiple of 4 lines)
    const size_t smem = sizeof(T) * ((size_t)tiled_w_offset(nb, th, a.w) + (size_t)nb * a.w);
    const dim3 grid(((side == 0 ? N : M) + a.w - 1) / a.w, a.S);
    static PerDeviceOnce once[2];
    const auto kern = side == 0 ? left_w_kernel<T, R, U> : right_w_kernel<T, R, U>;
    allow_max_smem(kern, once[side]);
    kern<<<grid, a.threads, smem, st>>>(X, ldx, M, N, V, ldv, nb, Tm, th, a.w, a.Ms, part, fin, tickets);
    return cudaGetLastError();
}

template <typename T, int U, int A>
static cudaError_t run_step3(int side, T *X, long ldx, int M, int N, const T *V, long ldv, int nb, const Shape &b,
                             const T *fin, cudaStream_t st) {
    const int strip = side == 0 ? N : M, len = side == 0 ? M : N;
    const dim3 grid((strip + b.w - 1) / b.w, (len + b.th - 1) / b.th);
    static PerDeviceOnce once[2];
    const auto kern = side == 0 ? left_x_kernel<T, U, A> : right_x_kernel<T, U, A>;
    allow_max_smem(kern, once[side]);
    kern<<<grid, b.threads, tiled_smem(side, (int)sizeof(T), nb, b.th, b.w), st>>>(X, ldx, M, N, V, ldv, nb, b.th, b.w,
                                                                                   fin);
    return cudaGetLastError();
}

template <typename T, int U>
static cudaError_t run_tiled(int side, T *X, long ldx, int M, int N, const T *V, long ldv, int nb, const T *Tm, int R,
                             const UpdCfg &c, const UpdScratch &sc, cudaStream_t st) {
    T *part = reinterpret_cast<T *>(sc.work);
    T *fin = part + (size_t)kMaxSplit * 64 * std::max(M, N);
    const int strip = side == 0 ? N : M, len = side == 0 ? M : N;
    const Shape a = step1_shape<T>(side, nb, R, c, strip, len), b = step3_shape<T>(c, strip, len);
    if (a.Ms <= 0) return cudaErrorInvalidConfiguration;  // no block shape fits: a zero W otherwise
    const auto step1 = a.R == 1   ? run_step1<T, U, 1>
                       : a.R == 2 ? run_step1<T, U, 2>
                       : a.R == 4 ? run_step1<T, U, 4>
                                  : run_step1<T, U, 8>;
    cudaError_t e = step1(side, X, ldx, M, N, V, ldv, nb, Tm, a, part, fin, sc.tickets, st);
    if (e != cudaSuccess) return e;
    if constexpr (sizeof(T) == 8) {
        if (b.A == 1) return run_step3<T, U, 1>(side, X, ldx, M, N, V, ldv, nb, b, fin, st);
        if (b.A == 2) return run_step3<T, U, 2>(side, X, ldx, M, N, V, ldv, nb, b, fin, st);
    }
    return run_step3<T, U, 4>(side, X, ldx, M, N, V, ldv, nb, b, fin, st);
}

template <typename T>
cudaError_t trail_tiled(int side, T *X, long ldx, int M, int N, const T *V, long ldv, int nb, const T *Tm,
                        const UpdCfg &c, const UpdScratch &sc, cudaStream_t st) {
    const int R = tiled_r(nb, c);
    if (!R || !sc.work || !sc.tickets) return cudaErrorInvalidConfiguration;
    const size_t smem = tiled_smem(side, (int)sizeof(T), nb, c.tile, 32 * c.cpb);
    if (smem > kTiledSmemLimit) return cudaErrorInvalidConfiguration;
    switch (c.unroll) {
        case 1: return run_tiled<T, 1>(side, X, ldx, M, N, V, ldv, nb, Tm, R, c, sc, st);
        case 2: return run_tiled<T, 2>(side, X, ldx, M, N, V, ldv, nb, Tm, R, c, sc, st);
        default: return run_tiled<T, 4>(side, X, ldx, M, N, V, ldv, nb, Tm, R, c, sc, st);
    }
}

// Largest block the compiled kernel can launch; 1024 (not cached) when it cannot be
// asked because this process has no CUDA device.
template <typename K>
static int kernel_max_threads(K kernel, bool &known) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) {
        cudaGetLastError();
        known = false;
        return 1024;
    }
    return fa.maxThreadsPerBlock;
}

template <typename T, int R, int U>
static int max_threads_one(int side, bool &known) {
    const auto w = side == 0 ? left_w_kernel<T, R, U> : right_w_kernel<T, R, U>;
    int n = std::min(kernel_max_threads(w, known),
                     kernel_max_threads(side == 0 ? left_x_kernel<T, U, 4> : right_x_kernel<T, U, 4>, known));
    if constexpr (sizeof(T) == 8) {
        n = std::min(n, kernel_max_threads(side == 0 ? left_x_kernel<T, U, 2> : right_x_kernel<T, U, 2>, known));
        n = std::min(n, kernel_max_threads(side == 0 ? left_x_kernel<T, U, 1> : right_x_kernel<T, U, 1>, known));
    }
    return n;
}

template <typename T, int R>
static int max_threads_r(int side, int u, bool &known) {
    return u == 1 ? max_threads_one<T, R, 1>(side, known)
           : u == 2 ? max_threads_one<T, R, 2>(side, known) : max_threads_one<T, R, 4>(side, known);
}

int tiled_max_threads(int side, int elem, int R, int unroll) {
    // a kernel's thread limit (from its register count) is the same on every device of
    // this architecture: cached once, under a lock
    static std::mutex mu;
    static int cache[2][2][4][3];
    static bool init = false;
    std::lock_guard<std::mutex> lk(mu);
    if (!init) {
        for (auto &a : cache)
            for (auto &b : a)
                for (auto &c : b)
                    for (int &d : c) d = -1;
        init = true;
    }
    const int ri = R == 1 ? 0 : R == 2 ? 1 : R == 4 ? 2 : 3, ui = unroll == 1 ? 0 : unroll == 2 ? 1 : 2;
    int &v = cache[side][elem == 8 ? 0 : 1][ri][ui];
    if (v < 0) {
        bool known = true;
        int q;
        if (elem == 8)
            q = R == 1 ? max_threads_r<double, 1>(side, unroll, known) : R == 2 ? max_threads_r<double, 2>(side, unroll, known)
              : R == 4 ? max_threads_r<double, 4>(side, unroll, known) : max_threads_r<double, 8>(side, unroll, known);
        else
            q = R == 1 ? max_threads_r<float, 1>(side, unroll, known) : R == 2 ? max_threads_r<float, 2>(side, unroll, known)
              : R == 4 ? max_threads_r<float, 4>(side, unroll, known) : max_threads_r<float, 8>(side, unroll, known);
        if (!known) return q;
        v = q;
    }
    return v;
}

template cudaError_t trail_tiled<double>(int, double *, long, int, int, const double *, long, int, const double *,
                                         const UpdCfg &, const UpdScratch &, cudaStream_t);
template cudaError_t trail_tiled<float>(int, float *, long, int, int, const float *, long, int, const float *,
                                        const UpdCfg &, const UpdScratch &, cudaStream_t);

}  // namespace nla
