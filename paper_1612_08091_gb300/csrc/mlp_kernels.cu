// mlp_kernels.cu -- the cost model behind the learned fusion planner:
// a 3-layer perceptron  x (16) -> relu(W1 x + b1) (H) -> relu(W2 h1 + b2) (H)
// -> w3 . h2 + b3 (1),  trained on the GPU with these kernels.
//
// Not a method of the paper.  Its inputs are the features of one unit of
// planned device work (a fused block or a plain gate launch; see planner.cpp)
// and its output is the predicted log of that launch's duration in ms.  The
// training targets are durations the simulator measured itself with CUDA
// events (sim_get_item_times).
//
// Everything is FP32 and deterministic: weight gradients are sums over the
// batch in sample order, no atomics.  The kernels are small dense loops on
// the CUDA cores; the matrices are far too small for the tensor cores to
// matter.  Training a network of up to 64 hidden units runs in one launch
// for many steps (k_train); the per-layer kernels serve inference, single
// gradients and wider networks.
//
// Parameter vector layout (P = H*16 + H + H*H + H + H + 1 floats):
//   W1 [H][16], b1 [H], W2 [H][H], b2 [H], w3 [H], b3.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "../../include/qsim.h"

namespace {

constexpr int kIn = 16;

struct Dims {
    int H;
    size_t oW1, ob1, oW2, ob2, ow3, ob3, P;
};

Dims dims(int H) {
    Dims d;
    d.H = H;
    d.oW1 = 0;
    d.ob1 = d.oW1 + (size_t)H * kIn;
    d.oW2 = d.ob1 + H;
    d.ob2 = d.oW2 + (size_t)H * H;
    d.ow3 = d.ob2 + H;
    d.ob3 = d.ow3 + H;
    d.P = d.ob3 + 1;
    return d;
}

// Y[b][j] = act( sum_i X[b][i] W[j][i] + bias[j] ),  one thread per (b, j)
__global__ void k_linear_fwd(const float *__restrict__ X, const float *__restrict__ W, const float *__restrict__ bias,
                             float *__restrict__ Y, int B, int in, int out, int relu) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= B * out) return;
    const int b = idx / out, j = idx % out;
    float acc = bias[j];
    for (int i = 0; i < in; ++i) acc = fmaf(X[(size_t)b * in + i], W[(size_t)j * in + i], acc);
    Y[idx] = relu ? fmaxf(acc, 0.f) : acc;
}

// dY[b] = 2 (Y[b] - T[b]) / B  and the per-sample squared error
__global__ void k_mse_grad(const float *__restrict__ Y, const float *__restrict__ T, float *__restrict__ dY,
                           float *__restrict__ sq, int B) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const float d = Y[b] - T[b];
    dY[b] = 2.f * d / (float)B;
    sq[b] = d * d;
}

// dX[b][i] = (sum_j dY[b][j] W[j][i]) * (Xact[b][i] > 0 if mask)
__global__ void k_linear_bwd_data(const float *__restrict__ dY, const float *__restrict__ W,
                                  const float *__restrict__ Xact, float *__restrict__ dX, int B, int in, int out,
                                  int mask) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= B * in) return;
    const int b = idx / in, i = idx % in;
    float acc = 0.f;
    for (int j = 0; j < out; ++j) acc = fmaf(dY[(size_t)b * out + j], W[(size_t)j * in + i], acc);
    if (mask && !(Xact[idx] > 0.f)) acc = 0.f;
    dX[idx] = acc;
}

// dW[j][i] = sum_b dY[b][j] X[b][i];  db[j] = sum_b dY[b][j]  (batch order)
__global__ void k_linear_bwd_weight(const float *__restrict__ dY, const float *__restrict__ X, float *__restrict__ dW,
                                    float *__restrict__ db, int B, int in, int out) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < out * in) {
        const int j = idx / in, i = idx % in;
        float acc = 0.f;
        for (int b = 0; b < B; ++b) acc = fmaf(dY[(size_t)b * out + j], X[(size_t)b * in + i], acc);
        dW[idx] = acc;
    } else if (idx < out * in + out) {
        const int j = idx - out * in;
        float acc = 0.f;
        for (int b = 0; b < B; ++b) acc += dY[(size_t)b * out + j];
        db[j] = acc;
    }
}

// Adam (bias-corrected): one parameter's step; returns its new value
__device__ __forceinline__ float adam_step(float p, float g, float &m, float &v, float lr, float b1, float b2,
                                           float eps, float c1, float c2) {
    const float mi = b1 * m + (1.f - b1) * g;
    const float vi = b2 * v + (1.f - b2) * g * g;
    m = mi;
    v = vi;
    return p - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    p[i] = adam_step(p[i], g[i], m[i], v[i], lr, b1, b2, eps, c1, c2);
}

// ---------------------------------------------------------------------------
// training: many steps in one launch
// ---------------------------------------------------------------------------
// A step of the 16-64-64-1 network on 256 samples is 8 MFLOP in twelve
// dependent layers; as twelve launches of one thread per output it took
// 146 us, nearly all of it launch gaps and loads waited for one at a time.
// Here one cluster of eight CTAs runs the steps.  The parameters sit in each
// CTA's shared memory.  Rows: CTA r takes an eighth of the batch forward and
// back (8 rows x 1 column a thread, so a weight read serves 8 FMAs) and
// writes its activations and deltas out (they stay in L2).  Weights: CTA r
// owns an eighth of the rows j of W1, W2 and their biases and of w3; it reads
// all samples' values and forms its gradients, a thread 4 rows j of one
// column, then the Adam step on moments held in registers, and writes the new
// parameters for all CTAs to read.  Two cluster barriers a step.  Every
// output's sum runs over the same terms in the same order as in the
// per-layer kernels, so both give the same numbers.
// 11,646 samples in batches of 256, 64 hidden units: 16.6 us a step against
// 146 us (clock64: 4.6 us parameters out, barrier and in again, 6.2 us rows,
// 2.1 us staging, 3.2 us gradients; the sums are bound by 16-byte broadcast
// reads of shared memory).
constexpr int kClusterCtas = 8;
constexpr int kTrainThreads = 256;
constexpr int kTrainMaxH = 64;      // one gradient task a thread (task_count(64) = 256)
constexpr int kTrainRows = 32;      // rows a CTA takes forward and back at a time
constexpr int kTrainChunk = 256;    // samples staged at a time for the weight gradients
constexpr int kTrainSteps = 4096;   // steps per launch

struct TrainArgs {
    const float *X, *T;        // all n samples
    const float2 *corr;        // Adam's bias corrections (c1, c2) of each step
    float *params, *m, *v;
    float *H1, *H2, *dY, *dH2, *dH1;  // one batch
    float *sq;                 // n squared errors of the last epoch
    int n, batch, H;
    long long step0, step1;    // steps of this launch (of epochs * steps per epoch)
    long long record_from;     // first step of the last epoch
    float lr, b1, b2, eps;
};

__host__ __device__ constexpr int train_slice(int H) { return (H + kClusterCtas - 1) / kClusterCtas; }
__host__ __device__ constexpr int train_groups(int H) { return (train_slice(H) + 3) / 4; }
// gradient tasks of a CTA: W2 columns, W1 columns (by groups of 4 rows j),
// then each in a warp of its own b2 and b1, w3, b3: their loops differ, and
// in one warp they would run one after the other
__host__ __device__ constexpr int train_bias_task(int H) { return ((H + kIn) * train_groups(H) + 31) & ~31; }
__host__ __device__ constexpr int task_count(int H) { return train_bias_task(H) + 96; }
static_assert(task_count(kTrainMaxH) <= kTrainThreads, "one gradient task a thread");
// 16-byte units of the parameters a thread loads
constexpr int kParamUnits = ((kTrainMaxH * (kTrainMaxH + kIn + 3)) / 4 + kTrainThreads - 1) / kTrainThreads;

// shared memory, in floats
__host__ __device__ constexpr int train_param_floats(int H) {
    return (kIn + H) * (H + 1) + H * H + 3 * H + 4;
}
__host__ __device__ constexpr int train_row_floats(int H) { return kTrainRows * (kIn + 3 * (H + 4) + 1); }
__host__ __device__ constexpr int train_chunk_floats(int H) {
    return kTrainChunk * (H + kIn + 8 * train_groups(H) + train_slice(H) + 1);
}
size_t train_smem(int H) {
    const int pf = (train_param_floats(H) + 3) & ~3;
    return sizeof(float) * (size_t)(pf + std::max(train_row_floats(H), train_chunk_floats(H)));
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// acc[r] += sum_k in[r][k] * w(k) in the order of k, for 8 rows
template <class W>
__device__ __forceinline__ void rows8(float (&acc)[8], const float *in, int pitch, int K, W w) {
#pragma unroll 4
    for (int k = 0; k < K; k += 4) {
        const float w0 = w(k), w1 = w(k + 1), w2 = w(k + 2), w3 = w(k + 3);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float4 x = *(const float4 *)(in + r * pitch + k);
            acc[r] = fmaf(x.x, w0, acc[r]);
            acc[r] = fmaf(x.y, w1, acc[r]);
            acc[r] = fmaf(x.z, w2, acc[r]);
            acc[r] = fmaf(x.w, w3, acc[r]);
        }
    }
}

__global__ void __cluster_dims__(kClusterCtas, 1, 1) __launch_bounds__(kTrainThreads, 1) k_train(const TrainArgs A) {
    extern __shared__ __align__(16) float tsm[];
    const int H = A.H, tid = threadIdx.x, rank = blockIdx.x, HP = H + 1, HR = H + 4;
    const int SL = train_slice(H), G = train_groups(H), SP = 4 * G;
    // parameters: W1 and W2 transposed (lanes over j), W2 as it is (lanes over i)
    float *W1T = tsm, *W2T = W1T + kIn * HP, *W2 = W2T + H * HP, *b1 = W2 + H * H, *b2 = b1 + H, *w3 = b2 + H,
          *b3 = w3 + H;
    float *u = tsm + ((train_param_floats(H) + 3) & ~3);  // the two phases' buffers share this
    float *xs = u, *h1 = xs + kTrainRows * kIn, *h2 = h1 + kTrainRows * HR, *d2 = h2 + kTrainRows * HR,
          *dy = d2 + kTrainRows * HR;
    float *cH1 = u, *cX = cH1 + kTrainChunk * H, *cD2 = cX + kTrainChunk * kIn, *cD1 = cD2 + kTrainChunk * SP,
          *cH2 = cD1 + kTrainChunk * SP, *cDy = cH2 + kTrainChunk * SL;
    const int oW1 = 0, ob1 = H * kIn, oW2 = ob1 + H, ob2 = oW2 + H * H, ow3 = ob2 + H, ob3 = ow3 + H, P = ob3 + 1;

    // this thread's gradient task: up to 4 parameters at base + k * stride
    const int j0 = rank * SL;
    int kind = -1, base = 0, stride = 0, cnt = 0, ti = 0, tg = 0;
    {
        int t = tid;
        const int tb = train_bias_task(H);
        auto rows = [&](int g) { return max(0, min(min(4, SL - 4 * g), H - j0 - 4 * g)); };
        if (t < H * G) {
            kind = 0, ti = t % H, tg = t / H, cnt = rows(tg), base = oW2 + (j0 + 4 * tg) * H + ti, stride = H;
        } else if (t < (H + kIn) * G) {
            t -= H * G;
            kind = 1, ti = t % kIn, tg = t / kIn, cnt = rows(tg), base = oW1 + (j0 + 4 * tg) * kIn + ti, stride = kIn;
        } else if (t >= tb && t < tb + 2 * G) {
            t -= tb;
            kind = t < G ? 2 : 3, tg = t % G, cnt = rows(tg), base = (t < G ? ob2 : ob1) + j0 + 4 * tg, stride = 1;
        } else if (t >= tb + 32 && t < tb + 32 + SL) {
            t -= tb + 32;
            kind = 4, ti = t, cnt = j0 + t < H ? 1 : 0, base = ow3 + j0 + t;
        } else if (t == tb + 64 && rank == 0) {
            kind = 5, cnt = 1, base = ob3;
        }
    }
    float pv[4], mv[4], vv[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < cnt) {
            pv[k] = A.params[base + k * stride];
            mv[k] = A.m[base + k * stride];
            vv[k] = A.v[base + k * stride];
        }
    const int per_epoch = (A.n + A.batch - 1) / A.batch;
    const unsigned invH = (1u << 20) / (unsigned)H + 1u;
    for (long long st = A.step0; st < A.step1; ++st) {
        const int s0 = (int)(st % per_epoch) * A.batch, B = min(A.batch, A.n - s0);
        const float *X = A.X + (size_t)s0 * kIn, *T = A.T + s0;
        // the parameters the previous step left: 16-byte units (every
        // section is a multiple of 4 floats), all loads in flight at once
        {
            const int U = (P - 1) / 4;
            float4 r[kParamUnits];
#pragma unroll
            for (int k = 0; k < kParamUnits; ++k)
                if (tid + k * kTrainThreads < U) r[k] = __ldcg((const float4 *)A.params + tid + k * kTrainThreads);
            if (tid == 0) b3[0] = __ldcg(A.params + ob3);
#pragma unroll
            for (int k = 0; k < kParamUnits; ++k) {
                const int i = 4 * (tid + k * kTrainThreads);
                if (i >= 4 * U) continue;
                if (i < ob1) {
                    float *w = W1T + (i % kIn) * HP + i / kIn;
                    w[0] = r[k].x;
                    w[HP] = r[k].y;
                    w[2 * HP] = r[k].z;
                    w[3 * HP] = r[k].w;
                } else if (i >= oW2 && i < ob2) {
                    // x / H by a reciprocal: exact for x <= 2^12 and H <= 64
                    const int x = i - oW2, j = (int)(((unsigned)x * invH) >> 20), c = x - j * H;
                    *(float4 *)(W2 + x) = r[k];
                    float *w = W2T + c * HP + j;
                    w[0] = r[k].x;
                    w[HP] = r[k].y;
                    w[2 * HP] = r[k].z;
                    w[3 * HP] = r[k].w;
                } else {
                    float *w = i < oW2 ? b1 + (i - ob1) : i < ow3 ? b2 + (i - ob2) : w3 + (i - ow3);
                    *(float4 *)w = r[k];
                }
            }
        }
        // ---- this CTA's rows, forward and back
        const int per = (B + kClusterCtas - 1) / kClusterCtas, r1 = min(B, (rank + 1) * per);
        for (int r0 = rank * per; r0 < r1; r0 += kTrainRows) {
            const int R = min(kTrainRows, r1 - r0);
            for (int i = tid; i < kTrainRows * kIn; i += kTrainThreads)
                xs[i] = i < R * kIn ? X[(size_t)r0 * kIn + i] : 0.f;
            __syncthreads();
            for (int t = tid; t < H * (kTrainRows / 8); t += kTrainThreads) {
                const int j = t % H, b = t / H * 8;
                float acc[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) acc[r] = b1[j];
                rows8(acc, xs + b * kIn, kIn, kIn, [&](int k) { return W1T[k * HP + j]; });
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float y = fmaxf(acc[r], 0.f);
                    h1[(b + r) * HR + j] = y;
                    if (b + r < R) A.H1[(size_t)(r0 + b + r) * H + j] = y;
                }
            }
            __syncthreads();
            for (int t = tid; t < H * (kTrainRows / 8); t += kTrainThreads) {
                const int j = t % H, b = t / H * 8;
                float acc[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) acc[r] = b2[j];
                rows8(acc, h1 + b * HR, HR, H, [&](int k) { return W2T[k * HP + j]; });
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float y = fmaxf(acc[r], 0.f);
                    h2[(b + r) * HR + j] = y;
                    if (b + r < R) A.H2[(size_t)(r0 + b + r) * H + j] = y;
                }
            }
            __syncthreads();
            if (tid < R) {
                float acc = b3[0];
#pragma unroll 8
                for (int i = 0; i < H; ++i) acc = fmaf(h2[tid * HR + i], w3[i], acc);
                const float d = acc - T[r0 + tid];
                const float g = 2.f * d / (float)B;
                dy[tid] = g;
                A.dY[r0 + tid] = g;
                if (st >= A.record_from) A.sq[s0 + r0 + tid] = d * d;
            }
            __syncthreads();
#pragma unroll 4
            for (int t = tid; t < R * H; t += kTrainThreads) {
                const int b = (int)(((unsigned)t * invH) >> 20), i = t - b * H;
                const float g = h2[b * HR + i] > 0.f ? fmaf(dy[b], w3[i], 0.f) : 0.f;
                d2[b * HR + i] = g;
                A.dH2[(size_t)(r0 + b) * H + i] = g;
            }
            __syncthreads();
            for (int t = tid; t < H * (kTrainRows / 8); t += kTrainThreads) {
                const int i = t % H, b = t / H * 8;
                float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                rows8(acc, d2 + b * HR, HR, H, [&](int k) { return W2[k * H + i]; });
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    if (b + r < R) A.dH1[(size_t)(r0 + b + r) * H + i] = h1[(b + r) * HR + i] > 0.f ? acc[r] : 0.f;
            }
            __syncthreads();
        }
        cluster_barrier();
        // ---- this CTA's weights: gradients over the whole batch
        float g[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c0 = 0; c0 < B; c0 += kTrainChunk) {
            const int C = min(kTrainChunk, B - c0);
            if (c0) __syncthreads();
            {
                const float4 *h = (const float4 *)(A.H1 + (size_t)c0 * H), *x4 = (const float4 *)(X + (size_t)c0 * kIn);
                const int nh = C * H / 4, nx = C * kIn / 4;
                float4 r[8];
                for (int i0 = tid; i0 < nh; i0 += 8 * kTrainThreads) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (i0 + k * kTrainThreads < nh) r[k] = __ldcg(h + i0 + k * kTrainThreads);
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (i0 + k * kTrainThreads < nh) ((float4 *)cH1)[i0 + k * kTrainThreads] = r[k];
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (tid + k * kTrainThreads < nx) r[k] = x4[tid + k * kTrainThreads];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (tid + k * kTrainThreads < nx) ((float4 *)cX)[tid + k * kTrainThreads] = r[k];
            }
            if (SL % 4 == 0) {  // whole 16-byte units of this CTA's rows j (SL = SP; G is 1 or 2)
                float4 r2[2], r1[2], rh[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i = tid + k * kTrainThreads, b = i / G, q = i % G;
                    const size_t at = (size_t)(c0 + b) * H + j0 + 4 * q;
                    if (i < C * G && j0 + 4 * q < H) {
                        r2[k] = __ldcg((const float4 *)(A.dH2 + at));
                        r1[k] = __ldcg((const float4 *)(A.dH1 + at));
                        rh[k] = __ldcg((const float4 *)(A.H2 + at));
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int i = tid + k * kTrainThreads;
                    if (i < C * G && j0 + 4 * (i % G) < H) {
                        ((float4 *)cD2)[i] = r2[k];
                        ((float4 *)cD1)[i] = r1[k];
                        ((float4 *)cH2)[i] = rh[k];
                    }
                }
            } else {
                for (int i = tid; i < C * SP; i += kTrainThreads) {
                    const int b = i / SP, k = i % SP;
                    const bool on = k < SL && j0 + k < H;
                    cD2[i] = on ? __ldcg(A.dH2 + (size_t)(c0 + b) * H + j0 + k) : 0.f;
                    cD1[i] = on ? __ldcg(A.dH1 + (size_t)(c0 + b) * H + j0 + k) : 0.f;
                    if (on) cH2[b * SL + k] = __ldcg(A.H2 + (size_t)(c0 + b) * H + j0 + k);
                }
            }
            for (int i = tid; i < C; i += kTrainThreads) cDy[i] = __ldcg(A.dY + c0 + i);
            __syncthreads();
            if (kind == 0 || kind == 1) {
                const float *d = (kind == 0 ? cD2 : cD1) + 4 * tg, *x = (kind == 0 ? cH1 : cX) + ti;
                const int px = kind == 0 ? H : kIn;
#pragma unroll 8
                for (int b = 0; b < C; ++b) {
                    const float4 dv = *(const float4 *)(d + b * SP);
                    const float xv = x[b * px];
                    g[0] = fmaf(dv.x, xv, g[0]);
                    g[1] = fmaf(dv.y, xv, g[1]);
                    g[2] = fmaf(dv.z, xv, g[2]);
                    g[3] = fmaf(dv.w, xv, g[3]);
                }
            } else if (kind == 2 || kind == 3) {
                const float *d = (kind == 2 ? cD2 : cD1) + 4 * tg;
#pragma unroll 8
                for (int b = 0; b < C; ++b) {
                    const float4 dv = *(const float4 *)(d + b * SP);
                    g[0] += dv.x;
                    g[1] += dv.y;
                    g[2] += dv.z;
                    g[3] += dv.w;
                }
            } else if (kind == 4 && cnt) {
#pragma unroll 8
                for (int b = 0; b < C; ++b) g[0] = fmaf(cDy[b], cH2[b * SL + ti], g[0]);
            } else if (kind == 5) {
#pragma unroll 8
                for (int b = 0; b < C; ++b) g[0] += cDy[b];
            }
        }
        const float2 c = A.corr[st - A.step0];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < cnt) {
                pv[k] = adam_step(pv[k], g[k], mv[k], vv[k], A.lr, A.b1, A.b2, A.eps, c.x, c.y);
                A.params[base + k * stride] = pv[k];
            }
        cluster_barrier();
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (k < cnt) {
            A.m[base + k * stride] = mv[k];
            A.v[base + k * stride] = vv[k];
        }
}

unsigned blocks(size_t work, int t = 256) { return (unsigned)((work + t - 1) / t); }

}  // namespace

struct qsim_mlp {
    Dims d;
    int cap = 0;  // batch capacity of the activation buffers
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    float *X = nullptr, *T = nullptr, *H1 = nullptr, *H2 = nullptr, *Y = nullptr;
    float *dY = nullptr, *dH2 = nullptr, *dH1 = nullptr, *sq = nullptr;
    // the training set and its squared errors, kept from one call to the next
    float *Xall = nullptr, *Tall = nullptr, *sq_all = nullptr;
    float2 *corr = nullptr;  // kTrainSteps bias corrections
    int cap_all = 0;
    long long step = 0;
    cudaStream_t stream = nullptr;
    std::string err;
};

namespace {

int mlp_err(qsim_mlp *m, int code, const char *msg) {
    if (m) m->err = msg;
    return code;
}

int ensure_capacity(qsim_mlp *m, int B) {
    if (B <= m->cap) return QSIM_OK;
    const int H = m->d.H;
    float **bufs[] = {&m->X, &m->T, &m->H1, &m->H2, &m->Y, &m->dY, &m->dH2, &m->dH1, &m->sq};
    const size_t sizes[] = {(size_t)B * kIn, (size_t)B, (size_t)B * H, (size_t)B * H, (size_t)B,
                            (size_t)B, (size_t)B * H, (size_t)B * H, (size_t)B};
    for (int i = 0; i < 9; ++i) {
        if (*bufs[i]) cudaFree(*bufs[i]);
        *bufs[i] = nullptr;
        if (cudaMalloc((void **)bufs[i], sizeof(float) * sizes[i]) != cudaSuccess) {
            cudaGetLastError();
            m->cap = 0;
            return mlp_err(m, QSIM_ENOMEM, "activation buffers");
        }
    }
    m->cap = B;
    return QSIM_OK;
}

int ensure_training_set(qsim_mlp *m, int n) {
    if (!m->corr && cudaMalloc((void **)&m->corr, sizeof(float2) * kTrainSteps) != cudaSuccess) {
        cudaGetLastError();
        m->corr = nullptr;
        return mlp_err(m, QSIM_ENOMEM, "training set");
    }
    if (n <= m->cap_all) return QSIM_OK;
    m->cap_all = 0;
    float **bufs[] = {&m->Xall, &m->Tall, &m->sq_all};
    const size_t sizes[] = {(size_t)n * kIn, (size_t)n, (size_t)n};
    for (int i = 0; i < 3; ++i) {
        if (*bufs[i]) cudaFree(*bufs[i]);
        *bufs[i] = nullptr;
        if (cudaMalloc((void **)bufs[i], sizeof(float) * sizes[i]) != cudaSuccess) {
            cudaGetLastError();
            return mlp_err(m, QSIM_ENOMEM, "training set");
        }
    }
    m->cap_all = n;
    return QSIM_OK;
}

// forward on m->X (B samples) into H1, H2, Y
void forward(qsim_mlp *m, int B) {
    const Dims &d = m->d;
    const int H = d.H;
    k_linear_fwd<<<blocks((size_t)B * H), 256, 0, m->stream>>>(m->X, m->params + d.oW1, m->params + d.ob1, m->H1, B,
                                                                 kIn, H, 1);
    k_linear_fwd<<<blocks((size_t)B * H), 256, 0, m->stream>>>(m->H1, m->params + d.oW2, m->params + d.ob2, m->H2, B,
                                                                 H, H, 1);
    k_linear_fwd<<<blocks((size_t)B), 256, 0, m->stream>>>(m->H2, m->params + d.ow3, m->params + d.ob3, m->Y, B, H, 1,
                                                             0);
}

// gradients of the mean squared error into m->grads (after forward)
void backward(qsim_mlp *m, int B) {
    const Dims &d = m->d;
    const int H = d.H;
    k_mse_grad<<<blocks(B), 256, 0, m->stream>>>(m->Y, m->T, m->dY, m->sq, B);
    k_linear_bwd_weight<<<blocks((size_t)H + 1), 256, 0, m->stream>>>(m->dY, m->H2, m->grads + d.ow3,
                                                                        m->grads + d.ob3, B, H, 1);
    k_linear_bwd_data<<<blocks((size_t)B * H), 256, 0, m->stream>>>(m->dY, m->params + d.ow3, m->H2, m->dH2, B, H, 1,
                                                                      1);
    k_linear_bwd_weight<<<blocks((size_t)H * H + H), 256, 0, m->stream>>>(m->dH2, m->H1, m->grads + d.oW2,
                                                                            m->grads + d.ob2, B, H, H);
    k_linear_bwd_data<<<blocks((size_t)B * H), 256, 0, m->stream>>>(m->dH2, m->params + d.oW2, m->H1, m->dH1, B, H,
                                                                      H, 1);
    k_linear_bwd_weight<<<blocks((size_t)H * kIn + H), 256, 0, m->stream>>>(m->dH1, m->X, m->grads + d.oW1,
                                                                              m->grads + d.ob1, B, kIn, H);
}

// splitmix64 -> uniform in [-1, 1)
double mix_uniform(unsigned long long &state) {
    unsigned long long z = (state += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    return (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

}  // namespace

extern "C" {

int sim_mlp_param_count(int hidden) { return hidden >= 1 && hidden <= 1024 ? (int)dims(hidden).P : -1; }

int sim_mlp_create(int hidden, unsigned long long seed, void *stream, qsim_mlp **out) {
    if (!out || hidden < 1 || hidden > 1024) return QSIM_EINVAL;
    *out = nullptr;
    qsim_mlp *m = new (std::nothrow) qsim_mlp();
    if (!m) return QSIM_ENOMEM;
    m->d = dims(hidden);
    m->stream = (cudaStream_t)stream;
    const size_t P = m->d.P;
    float **bufs[] = {&m->params, &m->grads, &m->m, &m->v};
    for (float **b : bufs) {
        if (cudaMalloc((void **)b, sizeof(float) * P) != cudaSuccess) {
            cudaGetLastError();
            sim_mlp_destroy(m);
            return QSIM_ENOMEM;
        }
    }
    // He-uniform weights, zero biases, from a seeded splitmix64 stream
    std::vector<float> p(P, 0.f);
    unsigned long long st = seed;
    const int H = hidden;
    const double a1 = std::sqrt(6.0 / kIn), a2 = std::sqrt(6.0 / H);
    for (size_t i = 0; i < (size_t)H * kIn; ++i) p[m->d.oW1 + i] = (float)(a1 * mix_uniform(st));
    for (size_t i = 0; i < (size_t)H * H; ++i) p[m->d.oW2 + i] = (float)(a2 * mix_uniform(st));
    for (int i = 0; i < H; ++i) p[m->d.ow3 + i] = (float)(a2 * mix_uniform(st));
    cudaMemcpyAsync(m->params, p.data(), sizeof(float) * P, cudaMemcpyHostToDevice, m->stream);
    cudaMemsetAsync(m->m, 0, sizeof(float) * P, m->stream);
    cudaMemsetAsync(m->v, 0, sizeof(float) * P, m->stream);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) {
        sim_mlp_destroy(m);
        return QSIM_ECUDA;
    }
    *out = m;
    return QSIM_OK;
}

int sim_mlp_destroy(qsim_mlp *m) {
    if (!m) return QSIM_OK;
    if (m->stream) cudaStreamSynchronize(m->stream);
    float *bufs[] = {m->params, m->grads, m->m, m->v, m->X, m->T, m->H1, m->H2, m->Y, m->dY, m->dH2, m->dH1, m->sq, m->Xall, m->Tall, m->sq_all};
    for (float *b : bufs)
        if (b) cudaFree(b);
    if (m->corr) cudaFree(m->corr);
    delete m;
    return QSIM_OK;
}

int sim_mlp_get_params(qsim_mlp *m, float *out, int count) {
    if (!m || !out || count != (int)m->d.P) return QSIM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(out, m->params, sizeof(float) * count, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? QSIM_OK : QSIM_ECUDA;
}

int sim_mlp_set_params(qsim_mlp *m, const float *in, int count) {
    if (!m || !in || count != (int)m->d.P) return QSIM_EINVAL;
    cudaError_t e = cudaMemcpyAsync(m->params, in, sizeof(float) * count, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    return e == cudaSuccess ? QSIM_OK : QSIM_ECUDA;
}

int sim_mlp_forward(qsim_mlp *m, const float *X, int n, float *Y) {
    if (!m || n < 1 || !X || !Y) return QSIM_EINVAL;
    int rc = ensure_capacity(m, n);
    if (rc) return rc;
    cudaMemcpyAsync(m->X, X, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, m->stream);
    forward(m, n);
    cudaMemcpyAsync(Y, m->Y, sizeof(float) * n, cudaMemcpyDeviceToHost, m->stream);
    return cudaStreamSynchronize(m->stream) == cudaSuccess ? QSIM_OK : QSIM_ECUDA;
}

// Gradient of the mean squared error over the n samples (for checking).
int sim_mlp_gradient(qsim_mlp *m, const float *X, const float *T, int n, float *grads, float *loss) {
    if (!m || n < 1 || !X || !T || !grads) return QSIM_EINVAL;
    int rc = ensure_capacity(m, n);
    if (rc) return rc;
    cudaMemcpyAsync(m->X, X, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, m->stream);
    cudaMemcpyAsync(m->T, T, sizeof(float) * n, cudaMemcpyHostToDevice, m->stream);
    forward(m, n);
    backward(m, n);
    std::vector<float> sq(n);
    cudaMemcpyAsync(grads, m->grads, sizeof(float) * m->d.P, cudaMemcpyDeviceToHost, m->stream);
    cudaMemcpyAsync(sq.data(), m->sq, sizeof(float) * n, cudaMemcpyDeviceToHost, m->stream);
    if (cudaStreamSynchronize(m->stream) != cudaSuccess) return QSIM_ECUDA;
    if (loss) {
        double s = 0.0;
        for (float v : sq) s += v;
        *loss = (float)(s / n);
    }
    return QSIM_OK;
}

// Adam on the mean squared error: `epochs` passes over the n samples in
// minibatches of `batch` (in order, last one partial).  *loss receives the
// mean squared error of the final epoch.
int sim_mlp_train(qsim_mlp *m, const float *X, const float *T, int n, int epochs, int batch, float lr, float *loss) {
    if (!m || n < 1 || !X || !T || epochs < 1 || batch < 1 || !(lr > 0.f)) return QSIM_EINVAL;
    if (batch > n) batch = n;
    int rc = ensure_capacity(m, n);
    if (rc) return rc;
    // all samples resident on the device; minibatches are views
    if ((rc = ensure_training_set(m, n))) return rc;
    cudaMemcpyAsync(m->Xall, X, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, m->stream);
    cudaMemcpyAsync(m->Tall, T, sizeof(float) * n, cudaMemcpyHostToDevice, m->stream);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const long long per_epoch = ((long long)n + batch - 1) / batch, steps = per_epoch * epochs;
    auto corrections = [&](long long step) {
        return make_float2(1.f - std::pow(b1, (float)step), 1.f - std::pow(b2, (float)step));
    };
    // one launch for many steps where a thread holds one gradient task and
    // rows are whole 16-byte units; the per-layer kernels for other widths
    // (256-sample batches, 64 units: 16.6 us a step against 146 us)
    const bool fused = m->d.H <= kTrainMaxH && m->d.H % 4 == 0;
    // the copies from host memory are waited for before every return, and the
    // corrections live as long: the runtime may read them as late as that
    std::vector<float2> corr;
    if (fused) {
        const size_t smem = train_smem(m->d.H);
        if (cudaFuncSetAttribute(k_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
            cudaGetLastError();
            cudaStreamSynchronize(m->stream);
            return mlp_err(m, QSIM_ECUDA, "training kernel attribute");
        }
        for (long long s0 = 0; s0 < steps; s0 += kTrainSteps) {
            const long long s1 = std::min<long long>(steps, s0 + kTrainSteps);
            if (s0) cudaStreamSynchronize(m->stream);  // `corr` is still being copied from
            corr.clear();
            for (long long st = s0; st < s1; ++st) corr.push_back(corrections(++m->step));
            cudaMemcpyAsync(m->corr, corr.data(), sizeof(float2) * corr.size(), cudaMemcpyHostToDevice, m->stream);
            TrainArgs a{};
            a.X = m->Xall;
            a.T = m->Tall;
            a.corr = m->corr;
            a.params = m->params;
            a.m = m->m;
            a.v = m->v;
            a.H1 = m->H1;
            a.H2 = m->H2;
            a.dY = m->dY;
            a.dH2 = m->dH2;
            a.dH1 = m->dH1;
            a.sq = m->sq_all;
            a.n = n;
            a.batch = batch;
            a.H = m->d.H;
            a.step0 = s0;
            a.step1 = s1;
            a.record_from = steps - per_epoch;
            a.lr = lr;
            a.b1 = b1;
            a.b2 = b2;
            a.eps = eps;
            k_train<<<kClusterCtas, kTrainThreads, smem, m->stream>>>(a);
            const cudaError_t e = cudaGetLastError();
            if (e != cudaSuccess) {
                cudaStreamSynchronize(m->stream);
                return mlp_err(m, QSIM_ECUDA, cudaGetErrorString(e));
            }
        }
    } else {
        float *keepX = m->X, *keepT = m->T;
        for (long long st = 0; st < steps; ++st) {
            const int s0 = (int)(st % per_epoch) * batch, B = std::min(batch, n - s0);
            m->X = m->Xall + (size_t)s0 * kIn;
            m->T = m->Tall + s0;
            forward(m, B);
            backward(m, B);
            const float2 c = corrections(++m->step);
            k_adam<<<blocks(m->d.P), 256, 0, m->stream>>>(m->params, m->grads, m->m, m->v, (int)m->d.P, lr, b1, b2,
                                                          eps, c.x, c.y);
            if (st >= steps - per_epoch)
                cudaMemcpyAsync(m->sq_all + s0, m->sq, sizeof(float) * B, cudaMemcpyDeviceToDevice, m->stream);
        }
        m->X = keepX;
        m->T = keepT;
    }
    std::vector<float> sq(n);
    cudaMemcpyAsync(sq.data(), m->sq_all, sizeof(float) * n, cudaMemcpyDeviceToHost, m->stream);
    const cudaError_t e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return mlp_err(m, QSIM_ECUDA, cudaGetErrorString(e));
    double sum = 0.0;
    for (float v : sq) sum += v;
    if (loss) *loss = (float)(sum / n);
    return QSIM_OK;
}

}  // extern "C"
