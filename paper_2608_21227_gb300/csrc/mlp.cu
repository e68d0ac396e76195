// mlp.cu -- the tuner's learned cost model: a 15 -> 128 -> 128 -> 128 -> 1 ReLU
// MLP in FP32 that predicts the log runtime of a configuration, trained and
// evaluated on the GPU by the kernels below (forward, backward, Adam).
//
// Layer l: Z_l = H_{l-1} W_l^T + b_l (W_l: out x in, row-major), H_l = relu(Z_l)
// for the hidden layers; loss = mean squared error.  Backward: G_L = 2/B (p - y),
// dW_l = G_l^T H_{l-1}, db_l = sum_rows G_l, G_{l-1} = (G_l W_l) .* [Z_{l-1} > 0].
// Adam (Kingma & Ba 2015): m <- b1 m + (1-b1) g, v <- b2 v + (1-b2) g^2,
// w <- w - lr (m / (1-b1^t)) / (sqrt(v / (1-b2^t)) + eps).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/kt.h"
#include "common.cuh"
#include "kernels.cuh"
#include "tuned.h"

namespace {

constexpr int kIn = KT_MLP_FEATURES;
constexpr int kH = 128;
constexpr int kLayers = 4;
const int kDims[kLayers + 1] = {kIn, kH, kH, kH, 1};

size_t w_off(int l) {  // offset of W_l (0-based layer) in the packed parameter vector
    size_t o = 0;
    for (int i = 0; i < l; ++i) o += (size_t)kDims[i + 1] * kDims[i] + kDims[i + 1];
    return o;
}
constexpr size_t kParams = (size_t)kH * kIn + kH + 2 * ((size_t)kH * kH + kH) + kH + 1;

// One block takes tiles of R rows through the whole network: forward, loss gradient and
// backward, with every activation in shared memory and one layer's weights staged at a time.
// The weights' gradients of a block's rows are 35,201 partial sums; each block writes its own
// (grad_sum_kernel adds them in block order, so results do not depend on timing).
//
// Why fused: as separate matrix products the step was 17 launches whose weight gradients had
// K = rows on 16 blocks (4096 rows: 101 us per product, 90 us per bias sum).  What bounds it
// now is shared-memory reads (a thread's 4 x 4 outputs read 8 values per 16 FMAs).
// One training step of 4096 rows: 1501 -> 57 us.
//
// Shared memory (floats): Ws kH x kLd (one layer's weights, transposed for the forward pass),
// X R x 16, H1..H3 and two gradient buffers R x kLd.
constexpr int kLd = kH + 4;  // rows stay 16-byte aligned, neighbouring rows shift by four banks
constexpr int kMlpThreads = 256;

constexpr size_t mlp_smem_floats(int R) { return (size_t)kH * kLd + (size_t)R * 16 + (size_t)5 * R * kLd + R + 8; }

// Rows per tile: small batches are spread over more blocks (8 rows: two blocks per SM fit).
int mlp_small_rows() { return 16 * nla::device_sm_count(); }
int mlp_tile(int rows) { return rows <= mlp_small_rows() ? 8 : 32; }
int mlp_blocks(int rows) {
    const int tile = mlp_tile(rows), sms = nla::device_sm_count();
    return std::min((rows + tile - 1) / tile, tile == 8 ? 2 * sms : sms);
}

// Ws(k, o) = W[o * K + k] (TRANS) or Ws(o, k) = W[o * K + k], K = kH.
template <bool TRANS>
__device__ void stage_weights(float *Ws, const float *__restrict__ W, int tid, bool vec) {
    if (vec) {
        for (int i = tid; i < kH * kH / 4; i += kMlpThreads) {
            if (TRANS) {
                const int o = i % kH, k = i / kH * 4;  // lanes along o: conflict-free stores
                const float4 w = *reinterpret_cast<const float4 *>(W + o * kH + k);
                Ws[k * kLd + o] = w.x, Ws[(k + 1) * kLd + o] = w.y;
                Ws[(k + 2) * kLd + o] = w.z, Ws[(k + 3) * kLd + o] = w.w;
            } else {
                const int k = i % (kH / 4) * 4, o = i / (kH / 4);
                *reinterpret_cast<float4 *>(Ws + o * kLd + k) = *reinterpret_cast<const float4 *>(W + o * kH + k);
            }
        }
    } else {
        for (int i = tid; i < kH * kH; i += kMlpThreads) {
            const int o = i / kH, k = i % kH;
            Ws[TRANS ? k * kLd + o : o * kLd + k] = W[i];
        }
    }
}

// acc(r, q) += sum_k In(r0 + r, k) Ws(k, 4 c + q) over the first K columns of In (leading dimension ld).
template <int RT>
__device__ void tile_product(float (&acc)[RT][4], const float *In, int ld, const float *Ws, int K, int r0, int c) {
#pragma unroll 2
    for (int k = 0; k < K; k += 4) {
        float4 h[RT], w[4];
#pragma unroll
        for (int r = 0; r < RT; ++r) h[r] = *reinterpret_cast<const float4 *>(In + (r0 + r) * ld + k);
#pragma unroll
        for (int u = 0; u < 4; ++u) w[u] = *reinterpret_cast<const float4 *>(Ws + (k + u) * kLd + 4 * c);
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const float hv[4] = {h[r].x, h[r].y, h[r].z, h[r].w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                acc[r][0] += hv[u] * w[u].x, acc[r][1] += hv[u] * w[u].y;
                acc[r][2] += hv[u] * w[u].z, acc[r][3] += hv[u] * w[u].w;
            }
        }
    }
}

// dW(o, k) (+)= sum_r G(r, o) H(r, k): thread t owns outputs o = 8 (t / 16) .., k = 4 (t % 16) .. and
// 64 + 4 (t % 16) ..; db(o) likewise.
template <int R>
__device__ void weight_grads(const float *G, const float *H, float *dW, float *db, bool first, int tid) {
    const int o0 = 8 * (tid / 16), k0 = 4 * (tid % 16);
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 2
    for (int r = 0; r < R; ++r) {
        float g[8], h[8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const float4 gv = *reinterpret_cast<const float4 *>(G + r * kLd + o0 + 4 * u);
            const float4 hv = *reinterpret_cast<const float4 *>(H + r * kLd + k0 + 64 * u);
            g[4 * u] = gv.x, g[4 * u + 1] = gv.y, g[4 * u + 2] = gv.z, g[4 * u + 3] = gv.w;
            h[4 * u] = hv.x, h[4 * u + 1] = hv.y, h[4 * u + 2] = hv.z, h[4 * u + 3] = hv.w;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] += g[i] * h[j];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float *d = dW + (o0 + i) * kH + k0 + (j & 3) + 64 * (j >> 2);
            *d = first ? acc[i][j] : *d + acc[i][j];
        }
    if (tid < kH) {
        float s = 0.f;
        for (int r = 0; r < R; ++r) s += G[r * kLd + tid];
        db[tid] = first ? s : db[tid] + s;
    }
}

template <int R>
__global__ void __launch_bounds__(kMlpThreads)
mlp_kernel(const float *__restrict__ P, const float *__restrict__ X, const float *__restrict__ y, int rows,
           float *pred, float *part, float *loss_acc, int train) {
    extern __shared__ __align__(16) float smem[];
    constexpr int RT = R / 8;  // rows per thread: 8 row groups x 32 output groups
    float *Ws = smem, *Xs = Ws + kH * kLd, *H[3], *Ga, *Gb, *gout;
    H[0] = Xs + R * 16;
    H[1] = H[0] + R * kLd, H[2] = H[1] + R * kLd;
    Ga = H[2] + R * kLd, Gb = Ga + R * kLd, gout = Gb + R * kLd;
    const int tid = threadIdx.x, c = tid % 32, r0 = tid / 32 * RT;
    const bool vec = (reinterpret_cast<uintptr_t>(P) & 15) == 0;  // (every layer starts on a multiple of four)
    constexpr size_t oW[kLayers] = {0, (size_t)kH * kIn + kH, (size_t)kH * kIn + kH + kH * kH + kH,
                                    (size_t)kH * kIn + kH + 2 * (kH * kH + kH)};
    constexpr size_t oB[kLayers] = {(size_t)kH * kIn, oW[1] + kH * kH, oW[2] + kH * kH, oW[3] + kH};
    float *dP = part + (size_t)blockIdx.x * kParams;
    bool first = true;
    float loss = 0.f;  // of this warp's rows
    for (int row0 = blockIdx.x * R; row0 < rows; row0 += gridDim.x * R, first = false) {
        __syncthreads();
        for (int i = tid; i < R * 16; i += kMlpThreads) {
            const int r = i / 16, k = i % 16;
            Xs[i] = (row0 + r < rows && k < kIn) ? X[(size_t)(row0 + r) * kIn + k] : 0.f;
        }
        // ---- forward
        for (int l = 0; l < 3; ++l) {
            if (l == 0) {
                for (int i = tid; i < kH * 16; i += kMlpThreads) {
                    const int o = i % kH, k = i / kH;
                    Ws[k * kLd + o] = k < kIn ? P[o * kIn + k] : 0.f;
                }
            } else {
                stage_weights<true>(Ws, P + oW[l], tid, vec);
            }
            __syncthreads();
            float acc[RT][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float bq = P[oB[l] + 4 * c + q];
#pragma unroll
                for (int r = 0; r < RT; ++r) acc[r][q] = bq;
            }
            if (l == 0)
                tile_product<RT>(acc, Xs, 16, Ws, 16, r0, c);
            else
                tile_product<RT>(acc, H[l - 1], kLd, Ws, kH, r0, c);
#pragma unroll
            for (int r = 0; r < RT; ++r)
                *reinterpret_cast<float4 *>(H[l] + (r0 + r) * kLd + 4 * c) =
                    make_float4(fmaxf(acc[r][0], 0.f), fmaxf(acc[r][1], 0.f), fmaxf(acc[r][2], 0.f), fmaxf(acc[r][3], 0.f));
            __syncthreads();
        }
        // ---- output layer: a warp per row (R / 8 rows each)
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < kH; k += 32) s += H[2][(r0 + r) * kLd + k + c] * P[oW[3] + k + c];
            s = nla::warp_sum(s) + P[oB[3]];
            const int row = row0 + r0 + r;
            float d = 0.f;
            if (row < rows) {
                if (c == 0) pred[row] = s;
                if (train) d = s - y[row];
            }
            if (c == 0) {
                gout[r0 + r] = 2.f * d / (float)rows;
                loss += d * d / (float)rows;
            }
        }
        if (!train) continue;
        __syncthreads();
        // ---- backward: output layer
        if (tid < kH) {
            float s = 0.f;
            const float w4 = P[oW[3] + tid];
            for (int r = 0; r < R; ++r) {
                const float h = H[2][r * kLd + tid], g = gout[r];
                s += g * h;
                Ga[r * kLd + tid] = h > 0.f ? g * w4 : 0.f;
            }
            dP[oW[3] + tid] = first ? s : dP[oW[3] + tid] + s;
        } else if (tid == kH) {
            float s = 0.f;
            for (int r = 0; r < R; ++r) s += gout[r];
            dP[oB[3]] = first ? s : dP[oB[3]] + s;
        }
        // ---- hidden layers 3 and 2: dW = G^T H, G' = (G W) .* [H > 0]
        float *G = Ga, *Gn = Gb;
        for (int l = 2; l >= 1; --l) {
            stage_weights<false>(Ws, P + oW[l], tid, vec);
            __syncthreads();
            weight_grads<R>(G, H[l - 1], dP + oW[l], dP + oB[l], first, tid);
            float acc[RT][4];
#pragma unroll
            for (int r = 0; r < RT; ++r)
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = 0.f;
            tile_product<RT>(acc, G, kLd, Ws, kH, r0, c);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                const float4 h = *reinterpret_cast<const float4 *>(H[l - 1] + (r0 + r) * kLd + 4 * c);
                *reinterpret_cast<float4 *>(Gn + (r0 + r) * kLd + 4 * c) =
                    make_float4(h.x > 0.f ? acc[r][0] : 0.f, h.y > 0.f ? acc[r][1] : 0.f, h.z > 0.f ? acc[r][2] : 0.f,
                                h.w > 0.f ? acc[r][3] : 0.f);
            }
            __syncthreads();
            float *t = G;
            G = Gn;
            Gn = t;
        }
        // ---- first layer: dW1 (kH x kIn), db1
        for (int i = tid; i < kH * 16; i += kMlpThreads) {
            const int o = i % kH, k = i / kH;  // k == kIn: the bias
            float s = 0.f;
            for (int r = 0; r < R; ++r) s += G[r * kLd + o] * (k < kIn ? Xs[r * 16 + k] : 1.f);
            float *d = k < kIn ? dP + o * kIn + k : dP + oB[0] + o;
            *d = first ? s : *d + s;
        }
    }
    if (train && loss_acc && c == 0) atomicAdd(loss_acc, loss);
}

// grads[i] = sum over the blocks' partial sums, in block order.  32 parameters x 8 slices of
// the blocks per thread block: enough loads in flight to read the partials at L2 speed.
__global__ void grad_sum_kernel(const float *__restrict__ part, int nblk, float *__restrict__ grads) {
    __shared__ float sh[8][33];
    const size_t i = (size_t)blockIdx.x * 32 + threadIdx.x;
    const int per = (nblk + 7) / 8, b0 = threadIdx.y * per, b1 = min(nblk, b0 + per);
    float s = 0.f;
    if (i < kParams) {
#pragma unroll 8
        for (int b = b0; b < b1; ++b) s += part[(size_t)b * kParams + i];
    }
    sh[threadIdx.y][threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.y == 0 && i < kParams) {
#pragma unroll
        for (int q = 1; q < 8; ++q) s += sh[q][threadIdx.x];
        grads[i] = s;
    }
}

// Floats of work for a batch of `rows`: the predictions and, to train, the blocks' partial gradients.
size_t pred_floats(int rows) { return ((size_t)rows + 63) & ~(size_t)63; }
size_t work_floats(int rows) { return pred_floats(rows) + (size_t)mlp_blocks(rows) * kParams; }
// The same for any batch of up to `rows` (the number of blocks halves above mlp_small_rows).
size_t work_floats_up_to(int rows) {
    const int small = mlp_small_rows();
    return rows > small ? std::max(work_floats(rows), work_floats(small)) : work_floats(rows);
}

// Predictions (into pred) and, when grads is given, the gradients of the mean squared error.
cudaError_t mlp_pass(cudaStream_t st, const float *P, const float *X, const float *y, int rows, float *work,
                     float *pred, float *grads, float *loss_acc) {
    const int R = mlp_tile(rows), nblk = mlp_blocks(rows);
    const size_t smem = mlp_smem_floats(R) * sizeof(float);
    float *part = work + pred_floats(rows);
    auto kern = R == 8 ? mlp_kernel<8> : mlp_kernel<32>;
    static nla::PerDeviceOnce attr;
    attr.run([] {
        cudaFuncSetAttribute(mlp_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(mlp_smem_floats(8) * 4));
        cudaFuncSetAttribute(mlp_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(mlp_smem_floats(32) * 4));
        cudaGetLastError();
    });
    kern<<<nblk, kMlpThreads, smem, st>>>(P, X, y, rows, pred ? pred : work, part, loss_acc, grads ? 1 : 0);
    if (grads) grad_sum_kernel<<<(int)((kParams + 31) / 32), dim3(32, 8), 0, st>>>(part, nblk, grads);
    return cudaGetLastError();
}

__global__ void adam_kernel(float *w, const float *g, float *m, float *v, size_t count, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        float gi = g[i];
        float mi = b1 * m[i] + (1.f - b1) * gi;
        float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

__global__ void gather_rows_kernel(const float *X, const float *y, const int *idx, int rows, float *Xb, float *yb) {
    int i = blockIdx.x;
    if (i >= rows) return;
    int src = idx[i];
    for (int k = threadIdx.x; k < kIn; k += blockDim.x) Xb[i * kIn + k] = X[(long)src * kIn + k];
    if (threadIdx.x == 0) yb[i] = y[src];
}

struct Model {
    std::vector<float> mean, sd, params;
    float ymean = 0.f, ysd = 1.f;
};

bool save_model(const char *path, const Model &m) {
    FILE *f = fopen(path, "wb");
    if (!f) return false;
    const char magic[8] = {'K', 'T', 'M', 'L', 'P', '1', 0, 0};
    int hdr[3] = {kIn, kH, (int)kParams};
    bool ok = fwrite(magic, 1, 8, f) == 8 && fwrite(hdr, sizeof(int), 3, f) == 3 &&
              fwrite(m.mean.data(), sizeof(float), kIn, f) == (size_t)kIn &&
              fwrite(m.sd.data(), sizeof(float), kIn, f) == (size_t)kIn && fwrite(&m.ymean, sizeof(float), 1, f) == 1 &&
              fwrite(&m.ysd, sizeof(float), 1, f) == 1 &&
              fwrite(m.params.data(), sizeof(float), kParams, f) == kParams;
    fclose(f);
    return ok;
}

bool load_model(const char *path, Model &m) {
    FILE *f = fopen(path, "rb");
    if (!f) return false;
    char magic[8];
    int hdr[3];
    m.mean.resize(kIn);
    m.sd.resize(kIn);
    m.params.resize(kParams);
    bool ok = fread(magic, 1, 8, f) == 8 && memcmp(magic, "KTMLP1", 6) == 0 && fread(hdr, sizeof(int), 3, f) == 3 &&
              hdr[0] == kIn && hdr[1] == kH && hdr[2] == (int)kParams &&
              fread(m.mean.data(), sizeof(float), kIn, f) == (size_t)kIn &&
              fread(m.sd.data(), sizeof(float), kIn, f) == (size_t)kIn && fread(&m.ymean, sizeof(float), 1, f) == 1 &&
              fread(&m.ysd, sizeof(float), 1, f) == 1 && fread(m.params.data(), sizeof(float), kParams, f) == kParams;
    fclose(f);
    return ok;
}

struct SplitMix {
    unsigned long long s;
    unsigned long long next() {
        s += 0x9E3779B97F4A7C15ull;
        unsigned long long z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    }
    double uniform() { return (double)(next() >> 11) * 0x1p-53; }
};

nla_status merr(nla_status s, const char *msg) {
    nla_set_last_error(msg);
    return s;
}

}  // namespace

namespace nla {

nla_status mlp_predict_host(const char *model_path, const float *X, int rows, float *y) {
    Model m;
    if (!model_path || !load_model(model_path, m)) return merr(NLA_ERR_ARG, "cannot read the MLP model file");
    if (rows <= 0) return NLA_OK;
    std::vector<float> Xs((size_t)rows * kIn);
    for (int i = 0; i < rows; ++i)
        for (int k = 0; k < kIn; ++k) Xs[(size_t)i * kIn + k] = (X[(size_t)i * kIn + k] - m.mean[k]) / m.sd[k];
    float *dP = nullptr, *dX = nullptr, *dW = nullptr;
    cudaStream_t st;
    cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    nla_status s = NLA_OK;
    if (cudaMalloc(&dP, kParams * sizeof(float)) || cudaMalloc(&dX, Xs.size() * sizeof(float)) ||
        cudaMalloc(&dW, pred_floats(rows) * sizeof(float))) {
        cudaGetLastError();
        s = merr(NLA_ERR_CUDA, "MLP inference: allocation failed");
    } else {
        cudaMemcpyAsync(dP, m.params.data(), kParams * sizeof(float), cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dX, Xs.data(), Xs.size() * sizeof(float), cudaMemcpyHostToDevice, st);
        mlp_pass(st, dP, dX, nullptr, rows, dW, dW, nullptr, nullptr);
        cudaMemcpyAsync(y, dW, rows * sizeof(float), cudaMemcpyDeviceToHost, st);
        if (cudaStreamSynchronize(st) != cudaSuccess) s = merr(NLA_ERR_CUDA, "MLP inference failed");
        for (int i = 0; i < rows; ++i) y[i] = y[i] * m.ysd + m.ymean;
    }
    cudaFree(dP);
    cudaFree(dX);
    cudaFree(dW);
    cudaStreamDestroy(st);
    return s;
}

}  // namespace nla

extern "C" {

size_t kt_mlp_param_count(void) { return kParams; }

size_t kt_mlp_work_bytes(int rows) { return work_floats_up_to(std::max(rows, 1)) * sizeof(float); }

nla_status kt_mlp_forward_backward(const float *dParams, const float *dX, const float *dY, int rows, float *dPred,
                                   float *dGrads, void *dWork, size_t work_bytes, nla_stream_t stream) {
    if (rows <= 0 || !dParams || !dX || !dY || !dGrads || !dWork) return merr(NLA_ERR_ARG, "bad arguments");
    if (work_bytes < work_floats(rows) * sizeof(float)) return merr(NLA_ERR_WORKSPACE, "MLP workspace too small");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = mlp_pass(st, dParams, dX, dY, rows, reinterpret_cast<float *>(dWork), dPred, dGrads, nullptr);
    return e == cudaSuccess ? NLA_OK : merr(NLA_ERR_CUDA, cudaGetErrorString(e));
}

nla_status kt_mlp_adam_step(float *dParams, const float *dGrads, float *dM, float *dV, size_t count, int t, float lr,
                            nla_stream_t stream) {
    if (t < 1 || !dParams || !dGrads || !dM || !dV) return merr(NLA_ERR_ARG, "bad arguments");
    const float b1 = 0.9f, b2 = 0.999f;
    float c1 = 1.f - (float)std::pow(0.9, t), c2 = 1.f - (float)std::pow(0.999, t);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    adam_kernel<<<256, 256, 0, st>>>(dParams, dGrads, dM, dV, count, lr, b1, b2, 1e-8f, c1, c2);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NLA_OK : merr(NLA_ERR_CUDA, cudaGetErrorString(e));
}

nla_status kt_mlp_train(const float *X, const float *y, int rows, int epochs, int batch, float lr,
                        unsigned long long seed, const char *model_path, float *final_loss) {
    if (!X || !y || rows <= 0 || epochs <= 0 || batch <= 0 || !model_path) return merr(NLA_ERR_ARG, "bad arguments");
    batch = std::min(batch, rows);
    Model m;
    m.mean.assign(kIn, 0.f);
    m.sd.assign(kIn, 1.f);
    // standardisation of inputs and target
    for (int k = 0; k < kIn; ++k) {
        double s = 0, s2 = 0;
        for (int i = 0; i < rows; ++i) {
            double v = X[(size_t)i * kIn + k];
            s += v;
            s2 += v * v;
        }
        double mu = s / rows, var = std::max(0.0, s2 / rows - mu * mu);
        m.mean[k] = (float)mu;
        m.sd[k] = var > 1e-12 ? (float)std::sqrt(var) : 1.f;
    }
    {
        double s = 0, s2 = 0;
        for (int i = 0; i < rows; ++i) {
            s += y[i];
            s2 += (double)y[i] * y[i];
        }
        double mu = s / rows, var = std::max(0.0, s2 / rows - mu * mu);
        m.ymean = (float)mu;
        m.ysd = var > 1e-12 ? (float)std::sqrt(var) : 1.f;
    }
    std::vector<float> Xs((size_t)rows * kIn), ys(rows);
    for (int i = 0; i < rows; ++i) {
        for (int k = 0; k < kIn; ++k) Xs[(size_t)i * kIn + k] = (X[(size_t)i * kIn + k] - m.mean[k]) / m.sd[k];
        ys[i] = (y[i] - m.ymean) / m.ysd;
    }
    // He-uniform initialisation from SplitMix64, zero biases
    SplitMix g{seed};
    m.params.assign(kParams, 0.f);
    for (int l = 0; l < kLayers; ++l) {
        double lim = std::sqrt(6.0 / kDims[l]);
        for (size_t i = 0; i < (size_t)kDims[l + 1] * kDims[l]; ++i)
            m.params[w_off(l) + i] = (float)((2.0 * g.uniform() - 1.0) * lim);
    }
    float *dX = nullptr, *dY = nullptr, *dP = nullptr, *dG = nullptr, *dM = nullptr, *dV = nullptr, *dXb = nullptr,
          *dYb = nullptr, *dW = nullptr, *dLoss = nullptr;
    int *dIdx = nullptr;
    cudaStream_t st;
    cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    nla_status s = NLA_OK;
    if (cudaMalloc(&dX, Xs.size() * 4) || cudaMalloc(&dY, rows * 4) || cudaMalloc(&dP, kParams * 4) ||
        cudaMalloc(&dG, kParams * 4) || cudaMalloc(&dM, kParams * 4) || cudaMalloc(&dV, kParams * 4) ||
        cudaMalloc(&dXb, (size_t)batch * kIn * 4) || cudaMalloc(&dYb, batch * 4) ||
        cudaMalloc(&dW, kt_mlp_work_bytes(batch)) || cudaMalloc(&dLoss, 4) || cudaMalloc(&dIdx, rows * 4)) {
        cudaGetLastError();
        s = merr(NLA_ERR_CUDA, "MLP training: allocation failed");
    }
    float last = NAN;
    if (s == NLA_OK) {
        cudaMemcpyAsync(dX, Xs.data(), Xs.size() * 4, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dY, ys.data(), rows * 4, cudaMemcpyHostToDevice, st);
        cudaMemcpyAsync(dP, m.params.data(), kParams * 4, cudaMemcpyHostToDevice, st);
        cudaMemsetAsync(dM, 0, kParams * 4, st);
        cudaMemsetAsync(dV, 0, kParams * 4, st);
        std::vector<int> idx(rows);
        int t = 0;
        for (int ep = 0; ep < epochs; ++ep) {
            for (int i = 0; i < rows; ++i) idx[i] = i;
            for (int i = rows - 1; i > 0; --i) std::swap(idx[i], idx[g.next() % (unsigned long long)(i + 1)]);
            cudaMemcpyAsync(dIdx, idx.data(), rows * 4, cudaMemcpyHostToDevice, st);
            cudaMemsetAsync(dLoss, 0, 4, st);
            int nb = 0;
            for (int b0 = 0; b0 + batch <= rows; b0 += batch, ++nb) {
                gather_rows_kernel<<<batch, 32, 0, st>>>(dX, dY, dIdx + b0, batch, dXb, dYb);
                mlp_pass(st, dP, dXb, dYb, batch, dW, nullptr, dG, dLoss);
                kt_mlp_adam_step(dP, dG, dM, dV, kParams, ++t, lr, st);
            }
            float h = 0.f;
            cudaMemcpyAsync(&h, dLoss, 4, cudaMemcpyDeviceToHost, st);
            if (cudaStreamSynchronize(st) != cudaSuccess) {
                s = merr(NLA_ERR_CUDA, "MLP training failed");
                break;
            }
            last = nb ? h / nb : NAN;
        }
        if (s == NLA_OK) {
            cudaMemcpyAsync(m.params.data(), dP, kParams * 4, cudaMemcpyDeviceToHost, st);
            cudaStreamSynchronize(st);
            if (!save_model(model_path, m)) s = merr(NLA_ERR_ARG, "cannot write the MLP model file");
        }
    }
    cudaFree(dX);
    cudaFree(dY);
    cudaFree(dP);
    cudaFree(dG);
    cudaFree(dM);
    cudaFree(dV);
    cudaFree(dXb);
    cudaFree(dYb);
    cudaFree(dW);
    cudaFree(dLoss);
    cudaFree(dIdx);
    cudaStreamDestroy(st);
    if (final_loss) *final_loss = last * m.ysd * m.ysd;  // in units of (log ms)^2
    return s;
}

nla_status kt_mlp_predict(const char *model_path, const float *X, int rows, float *y_out) {
    if (!X || !y_out || rows < 0) return merr(NLA_ERR_ARG, "bad arguments");
    return nla::mlp_predict_host(model_path, X, rows, y_out);
}

}  // extern "C"
