// chase.cu -- stage 2 (band -> bidiagonal) for band widths 8, 16, 32 and 64: the
// grouped bulge chase of band.cu's header with every block step shortened.
//
// The chase is a chain: sweep s + 1 may do step k once sweep s has done step k + 1, so
// n sweeps take about 2n block steps one after another, whatever the number of SMs.
// What counts is the time of one step and of one hand-off between groups, not
// throughput.  A block runs a group of G sweeps on a shared-memory window of band
// columns; at wavefront step tau team i (NW warps) does block step tau - 2i of its
// sweep as a right half, a barrier, a left half, a barrier.
//
// A half step applies H = I - g u u^T (u = x - beta e1) to 2B vectors of length B: on the
// right the rows tr .. tr + 2B - 1 (the first one is x itself), on the left the columns
// c0 .. c0 + 2B - 1 (likewise).  LPR lanes share a vector.
//   - the norm is the dot product of the first vector, so it costs nothing extra, and all dot
//     products (u^T row = u_0 row_0 + the rest, which is x's) start before it is known.
//   - x arrives through a small buffer that the previous half filled from registers (one
//     128-bit broadcast per four entries instead of a strided read).
//   - nothing is normalised: v = u / u_0 never exists, only g.
//
// What bounds it, and the layout that follows:
//   FP32: shared-memory cycles.  A half reads and writes every entry once, 36 cycles of
//   the SM's one port per team at B = 16, so a group of 8 teams keeps a half near its
//   latency (about 300 cycles) and more teams stretch it.
//   FP64: the FP64 pipe.  An SM issues one FP64 warp instruction per 19 cycles, and one
//   warp alone gets one per 64 whatever its active lanes (measured), so a sweep is
//   spread over four warps (one per sub-partition) with LPR = 4 lanes a row: 12
//   instructions a half in each plus 12 for the scalars in one.
// Columns move between global memory and the window as bulk copies (16-byte aligned
// columns: the packed leading dimension chase_ld), issued by one thread each way.
//
// Measured on GB300 (one warp per sweep, 16 sweeps a block, element copies -> this kernel):
// FP32 B = 16 n = 1024 4.43 -> 2.4 ms, n = 8192 38.1 -> 21.6 ms; FP32 B = 32 n = 3000 47.8 ->
// 12.8 ms; FP64 B = 16 n = 2048 35.4 -> 16.5 ms, B = 32 n = 256 9.1 -> 3.6 ms.  A block step is
// 1,370 cycles with one FP32 team and 1,900 with eight (B = 16), 5,080 in FP64; the hand-off
// between groups costs another 10,000 cycles a group.  Hence the group sizes below: FP32 8 to 12
// sweeps measured within 1 %, 4 gave 26 % and 16 8 % more; FP64 B = 16 two sweeps 8.4 against 9.6 ms
// for one (n = 1024), B = 32 one.
#include <algorithm>
#include <climits>
#include <cstdlib>

#include "common.cuh"
#include "house.cuh"
#include "kernels.cuh"
#include "tma.cuh"

namespace nla {

constexpr int kLag = 2;  // block steps between consecutive sweeps of a group

// Leading dimension of the packed band: the 3b+1 storage rows rounded up to 16 bytes.  The
// stride of a matrix row through the window, ld - 1, is odd, so lanes on neighbouring columns
// hit distinct banks.  0 for band widths this file does not cover.
int chase_ld(int b, int elem) {
    if (b != 8 && b != 16 && b != 32 && b != 64) return 0;
    const int per = 16 / elem;
    return (3 * b + 1 + per - 1) / per * per;
}

namespace {

NLA_DEV void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }
NLA_DEV void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *mbar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     tc::smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(tc::smem_u32(mbar))
                 : "memory");
}
NLA_DEV void bulk_store(void *dst, const void *src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(tc::smem_u32(src)),
                 "r"(bytes)
                 : "memory");
}

NLA_DEV unsigned magnitude_bits(float v) { return __float_as_uint(v) << 1; }
NLA_DEV unsigned magnitude_bits(double v) {
    return (unsigned)__double2loint(v) | (unsigned)__double2hiint(v) << 1;
}

// Teams of NW warps, LPR lanes per vector of B entries (lane p of them holds entries p + LPR i),
// RPT vectors per thread.
template <typename T, int B_, int NW_, int LPR_>
struct Shape {
    using Elem = T;
    static constexpr int B = B_, NW = NW_, LPR = LPR_;
    static constexpr int kLd = (3 * B + 1 + 16 / (int)sizeof(T) - 1) / (16 / (int)sizeof(T)) * (16 / (int)sizeof(T));
    static constexpr int CPT = B / LPR, GPP = 32 * NW / LPR, RPT = 2 * B / GPP;
    static constexpr int kMaxWarps = sizeof(T) == 8 ? 8 : 16;  // of all teams of a block (registers)
    static constexpr int kTeamElems = 2 * B + 16 / (int)sizeof(T) * 2;  // x and y buffers, four scalars
    static_assert(RPT * GPP == 2 * B && CPT * LPR == B && 32 % LPR == 0, "shape");
};

template <class S>
struct Half {
    using T = typename S::Elem;
    static constexpr int B = S::B, LD = S::kLd, LPR = S::LPR, CPT = S::CPT, RPT = S::RPT, GPP = S::GPP, NW = S::NW;

    // The half step where the vector's square leaves the normal range: H = I - m1 m2 u u^T does not
    // depend on the length of u, so x becomes x 2^-ex with its largest entry in [0.5, 1).  Rare, so
    // plain: a thread per vector, straight from shared memory, and out of line (inside the step
    // it took registers and 1 to 2 % of every step).
    template <bool RIGHT>
    __device__ __noinline__ static void scaled(T *win, int wc, int sl0, int n, int s, int k, int c0, int L, T *team,
                                               int ttid, int barid) {
        const auto sync = [&] {
            if (NW == 1)
                __syncwarp();
            else
                asm volatile("bar.sync %0, %1;" ::"r"(barid), "n"(32 * NW) : "memory");
        };
        const int tr = k == 0 ? s : c0 - B;
        const int nvec = RIGHT ? c0 + L - tr : min(c0 + 2 * B, n) - c0;
        const auto at = [&](int g, int c) -> T & {  // entry c of vector g
            const int w = RIGHT ? c : g;
            const int sl = sl0 + w - (sl0 + w >= wc ? wc : 0);
            return win[sl * LD + 2 * B + (RIGHT ? tr + g - c0 - c : c - g)];
        };
        const T *const buf = RIGHT ? team : team + B;
        const bool first = RIGHT && k == 0;  // the sweep starts: x is still in the window
        const auto x = [&](int i) { return first ? at(0, i) : buf[i]; };
        // a zero vector, not rare in a matrix with zero blocks: H = I, and nothing has changed (in
        // integers: an FP64 maximum holds the pipe for 64 cycles an entry)
        unsigned bits = 0u;
        for (int i = 0; i < L; ++i) bits |= magnitude_bits(x(i));
        if (bits == 0u) return;
        T mx = T(0);
        for (int i = 0; i < L; ++i) mx = fmax(mx, fabs(x(i)));
        sync();  // what the team left in the buffer for the next half is written again below
        int ex;
        frexp(mx, &ex);
        const T f1 = ldexp(T(1), -(ex / 2)), f2 = ldexp(T(1), -(ex - ex / 2));  // normal numbers both
        T beta, u0, m1, m2, qt = T(0);
        for (int i = 1; i < L; ++i) qt = fma(x(i) * f1 * f2, x(i) * f1 * f2, qt);
        house(x(0) * f1 * f2, qt, beta, u0, m1, m2);
        beta = beta / f1 / f2;
        for (int g = ttid; g < nvec; g += 32 * NW) {
            if (g > 0) {
                T d = u0 * at(g, 0);
                for (int i = 1; i < L; ++i) d = fma(x(i) * f1 * f2, at(g, i), d);
                const T w = d * m1 * m2;
                at(g, 0) = fma(-w, u0, at(g, 0));
                for (int i = 1; i < L; ++i) at(g, i) = fma(-w, x(i) * f1 * f2, at(g, i));
            }
            const int o = RIGHT ? g - (c0 - tr) : g - B;
            if (o >= 0) (RIGHT ? team + B : team)[o] = at(g, 0);
        }
        sync();
        if (ttid == 0)  // (x may have been vector 0 itself until here)
            for (int i = 0; i < L; ++i) at(0, i) = i == 0 ? beta : T(0);
    }

    // One half step of a team at position k of sweep s: c0 = s + k B + 1 is its first column, sl0 that
    // column's slot in the window (wc slots), L its reflector length.  FAST: every vector and
    // entry exists and, on the right, the B columns do not wrap in the window.
    template <bool RIGHT, bool FAST>
    NLA_DEV static void run(T *win, int wc, int sl0, int n, int s, int k, int c0, int L, T *team, int ttid, int barid) {
        const int lane = threadIdx.x & 31, p = ttid % LPR, g0 = ttid / LPR;
        T *const xbuf = team, *const ybuf = team + B, *const sc = team + 2 * B;
        const int tr = k == 0 ? s : c0 - B;
        const int c1 = c0 + L - 1;
        const int nvec = FAST ? 2 * B : RIGHT ? c1 - tr + 1 : min(c0 + 2 * B, n) - c0;
        const int wrap_c = wc - sl0;  // columns from c0 on before the window wraps
        T *base[RPT];
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const int gi = g0 + v * GPP;
            if (RIGHT) {
                base[v] = win + sl0 * LD + 2 * B - c0 + tr + gi + p * (LD - 1);
            } else {
                int sl = sl0 + gi;
                sl -= sl >= wc ? wc : 0;
                base[v] = win + sl * LD + 2 * B - gi + p;
            }
        }
        auto at = [&](int v, int i) -> T & {
            if (!RIGHT) return base[v][LPR * i];
            int off = LPR * i * (LD - 1);
            if (!FAST && p + LPR * i >= wrap_c) off -= wc * LD;
            return base[v][off];
        };
        T x[CPT], e[RPT][CPT], alpha;
#pragma unroll
        for (int v = 0; v < RPT; ++v)
#pragma unroll
            for (int i = 0; i < CPT; ++i)
                e[v][i] = (FAST || (g0 + v * GPP < nvec && p + LPR * i < L)) ? at(v, i) : T(0);
        if (!FAST && RIGHT && k == 0) {  // the sweep starts: x is row s of the window
            const T *row = win + sl0 * LD + 2 * B - c0 + s;
            alpha = row[0];
#pragma unroll
            for (int i = 0; i < CPT; ++i) {
                const int c = p + LPR * i;
                x[i] = c < L ? row[c * (LD - 1) - (c >= wrap_c ? wc * LD : 0)] : T(0);
            }
        } else {
            const T *buf = RIGHT ? xbuf : ybuf;
            alpha = buf[0];
            if constexpr (LPR == 1) {
                constexpr int per = 16 / (int)sizeof(T);
#pragma unroll
                for (int i = 0; i < CPT; i += per) {
                    const float4 f = *reinterpret_cast<const float4 *>(buf + i);
                    const T *q = reinterpret_cast<const T *>(&f);
#pragma unroll
                    for (int u = 0; u < per; ++u) x[i + u] = q[u];
                }
            } else {
#pragma unroll
                for (int i = 0; i < CPT; ++i) x[i] = buf[p + LPR * i];
            }
            if (!FAST) {
#pragma unroll
                for (int i = 0; i < CPT; ++i) x[i] = p + LPR * i < L ? x[i] : T(0);
            }
        }
        // ---- dot products without entry 0 (u^T row = u_0 row_0 + the rest); vector 0 is x itself
        if (p == 0) x[0] = T(0);
        T d[RPT], first[RPT];
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            constexpr int CH = CPT >= 8 && sizeof(T) == 4 ? 4 : 1;  // (an FP64 warp issues no faster than its latency)
            constexpr int I0 = LPR == 1 ? 1 : 0;
            T a[CH];
#pragma unroll
            for (int u = 0; u < CH; ++u) a[u] = e[v][u + I0] * x[u + I0];
#pragma unroll
            for (int i = CH + I0; i < CPT; ++i) a[(i - I0) % CH] = fma(e[v][i], x[i], a[(i - I0) % CH]);
            d[v] = CH == 4 ? (a[0] + a[CH / 4]) + (a[CH / 2] + a[CH - 1]) : a[0];
#pragma unroll
            for (int o = 1; o < LPR; o <<= 1) d[v] += __shfl_xor_sync(0xffffffffu, d[v], o);
            first[v] = LPR == 1 ? e[v][0] : __shfl_sync(0xffffffffu, e[v][0], lane & ~(LPR - 1));
        }
        // ---- scalars (by the warp that holds vector 0)
        T beta, u0, m1, m2;
        if (NW == 1 || ttid < 32) {
            const T qt = __shfl_sync(0xffffffffu, d[0], 0);
            house(alpha, qt, beta, u0, m1, m2);
            // a zero tail: H = I; m2 without m1: the vector has to be scaled first (by selects: a branch
            // would lengthen the chain)
            const bool fits = ordinary(fma(alpha, alpha, qt));
            if (magnitude_bits(qt) == 0u || !fits) beta = alpha, u0 = T(0), m1 = T(0), m2 = fits ? T(0) : T(1);
        }
        if constexpr (NW > 1) {
            if (ttid == 0) sc[0] = beta, sc[1] = u0, sc[2] = m1, sc[3] = m2;
            asm volatile("bar.sync %0, %1;" ::"r"(barid), "n"(32 * NW) : "memory");
            beta = sc[0], u0 = sc[1], m1 = sc[2], m2 = sc[3];
        }
        const bool reflect = magnitude_bits(m1) != 0u, rescale = !reflect && magnitude_bits(m2) != 0u;
        if (p == 0) x[0] = u0;
#pragma unroll
        for (int v = 0; v < RPT; ++v) {
            const int gi = g0 + v * GPP;
            T w = fma(u0, first[v], d[v]) * m1;
            if constexpr (sizeof(T) == 4) w *= m2;
#pragma unroll
            for (int i = 0; i < CPT; ++i) e[v][i] = fma(-w, x[i], e[v][i]);
            // (vector 0 becomes beta e1 below)
            const bool own = (v > 0 || g0 > 0 || !reflect) && (FAST || gi < nvec) && !rescale;
#pragma unroll
            for (int i = 0; i < CPT; ++i)
                if (own && (FAST || p + LPR * i < L)) at(v, i) = e[v][i];
            // the next half's x: column c0 of rows c0.. after the right half, row c0 of the
            // columns beyond the reflector's after the left half
            const int o = RIGHT ? gi - (c0 - tr) : gi - B;
            if (p == 0 && o >= 0 && (FAST || gi < nvec)) (RIGHT ? ybuf : xbuf)[o] = e[v][0];
        }
#pragma unroll
        for (int q = 0; q < B; q += 32) {
            const int c = ttid + q;
            if ((NW == 1 || ttid < 32) && (B % 32 == 0 || c < B) && reflect && (FAST || c < L)) {
                T *at0 = RIGHT ? win + sl0 * LD + 2 * B - c0 + tr + c * (LD - 1) - (!FAST && c >= wrap_c ? wc * LD : 0)
                               : win + sl0 * LD + 2 * B + c;
                *at0 = c == 0 ? beta : T(0);
            }
        }
        if (__builtin_expect(rescale, 0)) scaled<RIGHT>(win, wc, sl0, n, s, k, c0, L, team, ttid, barid);
    }
};

// Mover warp, element by element (a band whose leading dimension is not the packed one): columns
// j0 .. j0 + cnt - 1, 3B+1 storage rows each, of which only those inside the matrix are touched.
// Loads are asynchronous copies; stores are read four columns at a time before the first is stored.
// (Waiting for each chunk's loads and a division per column bound the chase before: n = 4096, B = 16,
// FP32, with a counters-only workspace 19.4 -> 12.3 ms; B = 32, n = 3000 29.5 -> 20.9.)
template <class S, bool LOAD>
NLA_DEV void copy_columns(typename S::Elem *win, int wc, typename S::Elem *AB, long ldab, int n, int j0, int cnt, int lane) {
    using T = typename S::Elem;
    constexpr int B = S::B, H = 3 * B + 1, QI = (H + 31) / 32, CU = LOAD ? 1 : 4;
    const int sl0 = j0 % wc;
    const auto inside = [&](int c, int q) { return q < H && (unsigned)(j0 + c + q - 2 * B) < (unsigned)n; };
    const auto slot = [&](int c) { return win + (size_t)(sl0 + c - (sl0 + c >= wc ? wc : 0)) * S::kLd; };
    T *const src = AB + (long)j0 * ldab;
    for (int c0 = 0; c0 < cnt; c0 += CU) {
        T r[CU][QI];
#pragma unroll
        for (int u = 0; u < CU; ++u)
#pragma unroll
            for (int i = 0; i < QI; ++i) {
                const int c = c0 + u, q = 32 * i + lane;
                if (c >= cnt || !inside(c, q)) continue;
                if (LOAD)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(tc::smem_u32(slot(c) + q)),
                                 "l"(src + (long)c * ldab + q), "n"((int)sizeof(T))
                                 : "memory");
                else
                    r[u][i] = slot(c)[q];
            }
        if (!LOAD) {
#pragma unroll
            for (int u = 0; u < CU; ++u)
#pragma unroll
                for (int i = 0; i < QI; ++i) {
                    const int c = c0 + u, q = 32 * i + lane;
                    if (c < cnt && inside(c, q)) __stcg(src + (long)c * ldab + q, r[u][i]);
                }
        }
    }
}

// Block = G teams, then a clerk, a flusher and a loader warp.  The teams run the group's sweeps
// in lockstep and never touch global memory.  The loader brings the group's columns in by
// chunks of B, each completing on its own mbarrier, as soon as the previous group has released
// them and the window has room.  The flusher writes back columns the group will not touch again
// and announces them in done[group].  The clerk takes part in the barriers on the movers'
// behalf, so that the teams' chain holds nothing but the two halves: it waits for the chunk that
// the coming left half needs (team 0 is always ahead of the others) before it arrives, and
// publishes the step count, whose memory fence takes a third of a half step, after it left.
// The window holds wc >= (2G - 1) B + G + 1 + B circular column slots.  Every wait is bounded; a
// timeout raises sh_abort, which the teams act on together.
constexpr int kChunkBars = 64;  // > chunks a window can hold

template <class S, bool BULK>
__global__ void __launch_bounds__(32 * (S::kMaxWarps + 3))
chase_kernel(typename S::Elem *AB, long ldab, int n, int G, int wc, int *done, int *info) {
    using T = typename S::Elem;
    constexpr int B = S::B, NW = S::NW, LD = S::kLd;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int sh_tau, sh_fl, sh_abort, sh_stop;  // steps complete, flushed-up-to column, abort, stop
    __shared__ __align__(8) uint64_t cbar[kChunkBars];
    T *win = reinterpret_cast<T *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nsweeps = n - 2;
    const int ngroups = (nsweeps + G - 1) / G;
    volatile int *vtau = &sh_tau, *vfl = &sh_fl, *vabort = &sh_abort, *vstop = &sh_stop;
    const auto bounded = [&](unsigned long long t0) {  // false when the budget has run out
        if (global_ns() - t0 <= kSpinBudgetNs) return true;
        if (info) atomicExch(info, kInfoTimeout);
        *vabort = 1;
        return false;
    };
    // A mover's view of a shared word.  With bulk copies one lane moves the columns; without them the
    // whole warp does and meets in warp-wide operations, so all lanes act on lane 0's value, and on
    // what was written before it (fence, then the warp barrier).
    const auto seen = [&](volatile int *word) {
        int v = *word;
        if (!BULK) {
            __threadfence_block();
            __syncwarp();
            v = __shfl_sync(0xffffffffu, v, 0);
        }
        return v;
    };
    uint32_t chunk0 = 0;  // chunks of this block's earlier groups: chunk m uses barrier (chunk0 + m) % kChunkBars
    if (tid == 0) {
        sh_abort = 0;
        sh_stop = 0;
        // (a chunk completes with the one lane that issued it, or with every lane's own copies)
        for (int i = 0; i < kChunkBars; ++i) tc::mbar_init(&cbar[i], BULK ? 1 : 32);
        tma::fence_init();
    }
    __syncthreads();
    for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
        const int s0 = grp * G, g = min(G, nsweeps - s0);
        const int lo0 = s0 + 1;                    // first column of the group
        const int nch = (n - lo0 + B - 1) / B;     // its chunks
        // steps of the group: its last sweep ends last (a sweep starts two steps later and
        // is at most one step shorter than the one before it)
        const int ntau = kLag * (g - 1) + (n - 2 - (s0 + g - 1)) / B + 1;
        if (tid == 0) {
            sh_tau = 0;
            sh_fl = lo0 - 1;
        }
        if (__syncthreads_or(*vabort)) break;  // (the same way for every thread)
        if (warp < G * NW) {
            // ---------------- teams
            const int it = warp / NW, ttid = tid - it * 32 * NW, s = s0 + it;
            T *team = win + (size_t)wc * LD + it * S::kTeamElems;
            int sl = (s + 1) % wc;  // window slot of this team's current c0
            int c0 = s + 1;
            const int kn = it < g ? (n - 3 - s) / B + 1 : 0;  // its steps (reflectors of two entries or more)
            const int kfull = it < g ? (n - 1 - s) / B : 0;   // the first kfull of them have B entries
            asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");  // chunk 0 is there
            for (int tau = 0, k = -kLag * it; tau < ntau; ++tau, ++k) {
                const bool go = (unsigned)k < (unsigned)kn;
                const int L = min(B, n - c0);
                if (go) {
                    if (k > 0 && k < kfull && sl + B <= wc)
                        Half<S>::template run<true, true>(win, wc, sl, n, s, k, c0, B, team, ttid, 2 + it);
                    else
                        Half<S>::template run<true, false>(win, wc, sl, n, s, k, c0, L, team, ttid, 2 + it);
                }
                // the right reflectors of this step all precede every left reflector:
                // with sweeps two steps apart that is the order the sequential chase needs
                asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");
                const int stop = *vstop;
                if (go) {
                    if (k < kfull - 1)
                        Half<S>::template run<false, true>(win, wc, sl, n, s, k, c0, B, team, ttid, 2 + it);
                    else
                        Half<S>::template run<false, false>(win, wc, sl, n, s, k, c0, L, team, ttid, 2 + it);
                }
                asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");
                if (k >= 0) {
                    c0 += B;
                    sl += B;
                    sl -= sl >= wc ? wc : 0;
                }
                if (stop) break;
            }
        } else if (warp == G * NW) {
            // ---------------- clerk
            const auto wait_chunk = [&](int m) {
                const uint32_t c = chunk0 + m, par = c / kChunkBars & 1;
                uint64_t *bar = &cbar[c % kChunkBars];
                if (tc::mbar_try_wait(bar, par)) return;
                const unsigned long long t0 = global_ns();
                // (after giving up the step still runs, on whatever the window holds: the teams
                // stay together until they stop at the closing barrier)
                while (!tc::mbar_try_wait(bar, par))
                    if (*vabort || !bounded(t0)) return;
            };
            wait_chunk(0);
            __syncwarp();
            asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");
            for (int tau = 0; tau < ntau; ++tau) {
                // the left half of team 0's step k, the first to use them, reads columns up to
                // lo0 - 1 + (k + 2) B: chunk k + 1 (the last chunk may be a step short)
                if (tau + 1 < nch) wait_chunk(tau + 1);
                if (lane == 0) *vstop = *vabort;
                __syncwarp();
                asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");
                const int stop = *vstop;
                asm volatile("bar.sync 1, %0;" ::"r"(32 * (NW * G + 1)) : "memory");
                if (stop) break;
                if (lane == 0) {
                    __threadfence_block();
                    *vtau = tau + 1;
                }
                __syncwarp();
            }
        } else if (warp == G * NW + 1) {
            // ---------------- flusher (one lane with bulk copies, the whole warp without)
            if (!BULK || lane == 0) {
                int flushed = lo0 - 1;
                for (;;) {
                    if (seen(vabort)) break;
                    const int t = seen(vtau);  // steps < t are complete
                    __threadfence_block();
                    // columns <= fin are final: the last started sweep is the lowest, and a sweep that
                    // has not started will start one column further on
                    int fin = n - 1;
                    if (t < ntau) {
                        const int ils = min(g - 1, t / kLag);
                        fin = min(s0 + ils + (t - kLag * ils) * B, n - 1);
                        if (ils + 1 < g) fin = min(fin, s0 + ils + 1);
                    }
                    if (fin > flushed) {
                        const int j0 = flushed + 1;
                        if (BULK) {
                            fence_async_all();  // the teams' writes precede the copies' reads
                            const int sl = j0 % wc, k1 = min(fin - flushed, wc - sl), k2 = fin - flushed - k1;
                            bulk_store(AB + (long)j0 * LD, win + (size_t)sl * LD, (uint32_t)(k1 * LD * sizeof(T)));
                            if (k2 > 0) bulk_store(AB + (long)(j0 + k1) * LD, win, (uint32_t)(k2 * LD * sizeof(T)));
                            tma::commit();
                            tma::wait_all();
                            fence_async_all();  // the copies' writes precede the release
                        } else {
                            copy_columns<S, false>(win, wc, AB, ldab, n, j0, fin - flushed, lane);
                            __threadfence();
                            __syncwarp();
                        }
                        flushed = fin;
                        if (lane == 0) {
                            st_release(&done[grp], t < ntau ? flushed + 1 : INT_MAX);
                            *vfl = flushed;  // the loader may reuse these slots now
                        }
                        if (!BULK) __syncwarp();
                    }
                    if (t >= ntau) break;
                }
            }
            __syncwarp();
        } else {
            // ---------------- loader
            if (!BULK || lane == 0) {
                int have = grp > 0 ? 0 : INT_MAX;  // columns < have are final in the previous group
                int m = 0;
                for (; m < nch && !seen(vabort);) {
                    const int j0 = lo0 + m * B, cnt = min(B, n - j0);
                    if (j0 + cnt > have) {
                        // every lane acquires, so that its own copies see what the previous group
                        // wrote; the smallest value seen is final for all of them
                        have = ld_acquire(&done[grp - 1]);
                        if (!BULK) have = __reduce_min_sync(0xffffffffu, have);
                        fence_async_all();  // what was acquired precedes the copies' reads
                        continue;
                    }
                    if (j0 + cnt - 1 > seen(vfl) + wc) continue;  // no room in the window yet
                    __threadfence_block();
                    const uint32_t c = chunk0 + m;
                    uint64_t *bar = &cbar[c % kChunkBars];
                    if (BULK) {
                        fence_async_all();  // the slots' earlier reads and writes precede the copies
                        const int sl = j0 % wc, k1 = min(cnt, wc - sl), k2 = cnt - k1;
                        tma::expect_tx(bar, (uint32_t)(cnt * LD * sizeof(T)));
                        bulk_load(win + (size_t)sl * LD, AB + (long)j0 * LD, (uint32_t)(k1 * LD * sizeof(T)), bar);
                        if (k2 > 0) bulk_load(win, AB + (long)(j0 + k1) * LD, (uint32_t)(k2 * LD * sizeof(T)), bar);
                    } else {
                        copy_columns<S, true>(win, wc, AB, ldab, n, j0, cnt, lane);
                        asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
                    }
                    ++m;
                }
                // let the copies in flight land before the block may leave
                if (!BULK) asm volatile("cp.async.wait_all;" ::: "memory");
                for (int i = max(0, m - kChunkBars); BULK && i < m && *vabort; ++i) {
                    const uint32_t c = chunk0 + i;
                    tc::mbar_wait(&cbar[c % kChunkBars], c / kChunkBars & 1, info);
                }
            }
            __syncwarp();
        }
        chunk0 += nch;
        __syncthreads();
    }
}

// AB (leading dimension ldab) <-> packed band, storage rows 0 .. 3b of every column.
template <typename T>
__global__ void repack_kernel(const T *__restrict__ src, long lds, T *__restrict__ dst, long ldd, int n, int h) {
    const long total = (long)n * h;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const long j = i / h, q = i % h;
        dst[j * ldd + q] = src[j * lds + q];
    }
}

template <class S>
cudaError_t launch(typename S::Elem *AB, long ldab, int n, int gmax, int *done, int *info, cudaStream_t st) {
    using T = typename S::Elem;
    constexpr size_t kBudget = 220 * 1024;
    const bool bulk = ldab == S::kLd && reinterpret_cast<uintptr_t>(AB) % 16 == 0;
    const auto kern = bulk ? chase_kernel<S, true> : chase_kernel<S, false>;
    static PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(chase_kernel<S, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBudget);
        cudaFuncSetAttribute(chase_kernel<S, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBudget);
        cudaGetLastError();
    });
    const size_t col = (size_t)S::kLd * sizeof(T);
    const auto smem_of = [&](int G, int pf) {
        const size_t wc = (size_t)(kLag * G - 1) * S::B + G + 1 + (size_t)pf * S::B;
        return wc * col + (size_t)G * S::kTeamElems * sizeof(T);
    };
    // the largest group up to gmax whose window leaves two chunks of prefetch (or one, for one
    // sweep); then as much prefetch as fits, up to 16 chunks: a column's way out of one window
    // and into the next takes several steps' time
    int G = std::max(1, std::min(gmax, S::kMaxWarps / S::NW));
    while (G > 1 && smem_of(G, 2) > kBudget) --G;
    int pf = 16;
    while (pf > 1 && smem_of(G, pf) > kBudget) --pf;
    if (smem_of(G, pf) > kBudget) return cudaErrorInvalidConfiguration;
    const int ngroups = (n - 2 + G - 1) / G;
    cudaError_t err = cudaMemsetAsync(done, 0, sizeof(int) * (size_t)ngroups, st);
    if (err != cudaSuccess) return err;
    const int wc = (kLag * G - 1) * S::B + G + 1 + pf * S::B;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::min(ngroups, device_sm_count()));
    cfg.blockDim = dim3(32 * (G * S::NW + 3));
    cfg.dynamicSmemBytes = smem_of(G, pf);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;  // groups wait on one another: all blocks resident
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, AB, ldab, n, G, wc, done, info);
}

}  // namespace

// Repack n columns of 3b+1 storage rows.
template <typename T>
cudaError_t band_repack(const T *src, long lds, T *dst, long ldd, int n, int b, cudaStream_t st) {
    const long total = (long)n * (3 * b + 1);
    const int blocks = (int)std::min<long>((total + 255) / 256, 8L * device_sm_count());
    repack_kernel<T><<<blocks, 256, 0, st>>>(src, lds, dst, ldd, n, 3 * b + 1);
    return cudaGetLastError();
}

// Chase the n x n band in place; gmax = most sweeps per block (0: the width's default).
// cudaErrorNotSupported for band widths other than 8, 16, 32, 64.  done: n ints of scratch.
template <typename T>
cudaError_t chase_fixed(T *AB, long ldab, int n, int b, int gmax, int *done, int *info, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        switch (b) {
            case 8: return launch<Shape<T, 8, 1, 2>>(AB, ldab, n, gmax ? gmax : 12, done, info, st);
            case 16: return launch<Shape<T, 16, 1, 1>>(AB, ldab, n, gmax ? gmax : 10, done, info, st);
            case 32: return launch<Shape<T, 32, 2, 1>>(AB, ldab, n, gmax ? gmax : 4, done, info, st);
            case 64: return launch<Shape<T, 64, 8, 2>>(AB, ldab, n, gmax ? gmax : 2, done, info, st);
        }
    } else {
        switch (b) {
            case 8: return launch<Shape<T, 8, 2, 4>>(AB, ldab, n, gmax ? gmax : 2, done, info, st);
            case 16: return launch<Shape<T, 16, 4, 4>>(AB, ldab, n, gmax ? gmax : 2, done, info, st);
            case 32: return launch<Shape<T, 32, 4, 4>>(AB, ldab, n, gmax ? gmax : 1, done, info, st);
            case 64: return launch<Shape<T, 64, 8, 4>>(AB, ldab, n, gmax ? gmax : 1, done, info, st);
        }
    }
    return cudaErrorNotSupported;
}

#define NLA_INST(T)                                                                                  \
    template cudaError_t band_repack<T>(const T *, long, T *, long, int, int, cudaStream_t);         \
    template cudaError_t chase_fixed<T>(T *, long, int, int, int, int *, int *, cudaStream_t);
NLA_INST(double)
NLA_INST(float)
#undef NLA_INST

}  // namespace nla
