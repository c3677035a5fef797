// k_cost.cu -- learned cost model of a tick: a multilayer perceptron
// 5 -> 64 -> 64 -> 1 (ReLU hidden layers) mapping tick features to the
// logarithm of the tick's time, trained by full-batch Adam on logged ticks.
// The paper models the cost of its phases analytically (Sec. 5.4 filtering
// complexity, the subquery-count estimate of Sec. 6); this learns it from
// measurements instead, to choose the index configuration of the next tick.
// Choices never change results (every index configuration answers exactly).
//
// Parameter layout (P floats): W1[64][5], b1[64], W2[64][64], b2[64],
// W3[64], b3.  Training runs a block per chunk of 32 samples.  A block keeps
// the parameters (W2 in both orders) and its chunk's activations in shared
// memory and computes 4 x 2 and 4 x 4 register tiles of every product; the
// chunks' gradients go to global memory, every parameter is owned by one
// thread, which adds its chunk gradients in chunk order and takes the Adam
// step, and the blocks meet twice an epoch: at a cluster barrier (up to 8
// chunks) or at a barrier of a cooperative grid.  Every sum runs over the same
// terms in the same order whatever the number of blocks.  An epoch is a chain
// of short phases, bound by latency and barriers: 400 epochs of 80 samples take
// 3.9 ms, 100 epochs of 4,096 take 1.5 (40.4 and 393 with one block for all
// chunks, two shared-memory loads to a multiplication).
#include <algorithm>
#include <cstddef>

#include "mqr_internal.cuh"

namespace mqr {

constexpr int kCostIn = 5, kCostH = 64, kCostChunk = 32, kCostThreads = 256;
constexpr int kOW1 = 0, kOB1 = kOW1 + kCostH * kCostIn, kOW2 = kOB1 + kCostH, kOB2 = kOW2 + kCostH * kCostH,
              kOW3 = kOB2 + kCostH, kOB3 = kOW3 + kCostH, kCostP = kOB3 + 1;

size_t cost_param_count() { return kCostP; }

constexpr uint32_t kCostDirect = 64;                 // chunks of a round that an owner adds straight from memory
constexpr int kCostClusterMax = 8;                   // blocks that meet at a cluster barrier (the portable size)
constexpr int kUS = kCostH + 4;                      // row stride of 64 units (16-byte rows, shifted banks)
constexpr int kStage = 32 + 1;                       // row stride of staged chunk gradients
constexpr int kSqErr = (kCostP + 31) / 32 * 32;      // a chunk's gradients, then its 32 squared errors
constexpr int kPart = kSqErr + kCostChunk;
constexpr int kOwn = 3;                              // parameters of a thread at most
constexpr int kCostBlocksMin = (kSqErr / 32 + kOwn * kCostThreads / 32 - 1) / (kOwn * kCostThreads / 32);

struct CostSmem {
    float w2[kCostH * kUS];                          // W2[j][k]
    float w2t[kCostH * kUS];                         // W2[j][k] at [k][j]
    float w1[kCostH * kCostIn], b1[kCostH], b2[kCostH], w3[kCostH];
    float h1[kCostChunk * kUS], h2[kCostChunk * kUS], d2[kCostChunk * kUS], d1[kCostChunk * kUS];   // [sample][unit]
    float x[kCostChunk * kCostIn], dout[kCostChunk];
    float b3;
    int stop;
};
static_assert(offsetof(CostSmem, w2t) % 16 == 0 && offsetof(CostSmem, b2) % 16 == 0 && offsetof(CostSmem, h1) % 16 == 0 &&
                  offsetof(CostSmem, d1) % 16 == 0, "rows are read 16 bytes at a time");

// The parameters from global memory (written by other blocks: not through
// L1), all of a thread's loads in flight together.
__device__ __forceinline__ void cost_load_params(CostSmem &sm, const float *params, int tid) {
    constexpr int kRest = kCostP - kCostH * kCostH, kR = (kRest + kCostThreads - 1) / kCostThreads;
    static_assert(kOW2 % 4 == 0 && kCostH * kCostH == 16 * kCostThreads, "four 16-byte loads of W2 a thread");
    float4 w[4];
    float r[kR];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = __ldcg(reinterpret_cast<const float4 *>(params + kOW2) + q * kCostThreads + tid);
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int i = q * kCostThreads + tid;
        r[q] = i < kRest ? __ldcg(params + (i < kOW2 ? i : i + kCostH * kCostH)) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int i = (q * kCostThreads + tid) * 4, j = i / kCostH, k = i % kCostH;
        *reinterpret_cast<float4 *>(sm.w2 + j * kUS + k) = w[q];
        sm.w2t[k * kUS + j] = w[q].x;
        sm.w2t[(k + 1) * kUS + j] = w[q].y;
        sm.w2t[(k + 2) * kUS + j] = w[q].z;
        sm.w2t[(k + 3) * kUS + j] = w[q].w;
    }
#pragma unroll
    for (int q = 0; q < kR; ++q) {
        const int i = q * kCostThreads + tid;
        if (i < kOB1) sm.w1[i] = r[q];
        else if (i < kOW2) sm.b1[i - kOB1] = r[q];
        else if (i < kOW2 + kCostH) sm.b2[i - kOW2] = r[q];
        else if (i < kOW2 + 2 * kCostH) sm.w3[i - kOW2 - kCostH] = r[q];
        else if (i < kRest) sm.b3 = r[q];
    }
}

// out[s][u] = init[u] + sum over v = 0 .. 63 of w[v][u] * act[s][v], in order,
// for the thread's 4 units (tid & 15) and 2 samples (tid >> 4).
__device__ __forceinline__ void cost_product(const float *w, const float *act, float4 init, int tid, float (&o)[2][4]) {
    const int u = (tid & 15) * 4, s = (tid >> 4) * 2;
    for (int r = 0; r < 2; ++r) { o[r][0] = init.x; o[r][1] = init.y; o[r][2] = init.z; o[r][3] = init.w; }
#pragma unroll 4
    for (int v = 0; v < kCostH; v += 4) {
        float a[2][4];
        *reinterpret_cast<float4 *>(a[0]) = *reinterpret_cast<const float4 *>(act + s * kUS + v);
        *reinterpret_cast<float4 *>(a[1]) = *reinterpret_cast<const float4 *>(act + (s + 1) * kUS + v);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 wv = *reinterpret_cast<const float4 *>(w + (v + q) * kUS + u);
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                o[r][0] = fmaf(wv.x, a[r][q], o[r][0]);
                o[r][1] = fmaf(wv.y, a[r][q], o[r][1]);
                o[r][2] = fmaf(wv.z, a[r][q], o[r][2]);
                o[r][3] = fmaf(wv.w, a[r][q], o[r][3]);
            }
        }
    }
}

// Forward pass of the chunk's samples in sm.x: h1, h2 (rectified) and, in the
// first 32 threads, the sample's output.  Contains __syncthreads.
__device__ __forceinline__ float cost_forward(CostSmem &sm, int tid) {
    const int u = (tid & 15) * 4, s = (tid >> 4) * 2;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float a = sm.b1[u + c];
#pragma unroll
            for (int k = 0; k < kCostIn; ++k) a = fmaf(sm.w1[(u + c) * kCostIn + k], sm.x[(s + r) * kCostIn + k], a);
            sm.h1[(s + r) * kUS + u + c] = a > 0.f ? a : 0.f;
        }
    __syncthreads();
    float o[2][4];
    cost_product(sm.w2t, sm.h1, *reinterpret_cast<const float4 *>(sm.b2 + u), tid, o);
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) sm.h2[(s + r) * kUS + u + c] = o[r][c] > 0.f ? o[r][c] : 0.f;
    __syncthreads();
    float out = 0.f;
    if (tid < kCostChunk) {
        out = sm.b3;
#pragma unroll 4
        for (int j = 0; j < kCostH; j += 4) {
            const float4 h = *reinterpret_cast<const float4 *>(sm.h2 + tid * kUS + j);
            const float4 w = *reinterpret_cast<const float4 *>(sm.w3 + j);
            out = fmaf(w.x, h.x, out);
            out = fmaf(w.y, h.y, out);
            out = fmaf(w.z, h.z, out);
            out = fmaf(w.w, h.w, out);
        }
    }
    return out;
}

__device__ __forceinline__ void cost_load_x(CostSmem &sm, const float *__restrict__ X, uint32_t c0, int cn, int tid) {
    for (int i = tid; i < kCostChunk * kCostIn; i += kCostThreads)
        sm.x[i] = i < cn * kCostIn ? X[(size_t)c0 * kCostIn + i] : 0.f;
}

// The gradients of one chunk (cn of 32 samples) and its squared errors to part[kPart].
__device__ void cost_chunk(CostSmem &sm, const float *__restrict__ X, const float *__restrict__ y, uint32_t n,
                           uint32_t c0, float *part, int tid) {
    const int cn = (int)min((uint32_t)kCostChunk, n - c0);
    cost_load_x(sm, X, c0, cn, tid);
    __syncthreads();
    const float out = cost_forward(sm, tid);
    if (tid < kCostChunk) {
        const float e = tid < cn ? out - y[c0 + tid] : 0.f;
        sm.dout[tid] = 2.f * e / (float)n;                       // d(mean squared error)/d(out)
        __stcg(part + kSqErr + tid, e * e);
    }
    __syncthreads();
    for (int i = tid; i < kCostH * kCostChunk; i += kCostThreads) {
        const int s = i / kCostH, j = i % kCostH;
        sm.d2[s * kUS + j] = sm.h2[s * kUS + j] > 0.f ? sm.dout[s] * sm.w3[j] : 0.f;
    }
    __syncthreads();
    {
        const int u = (tid & 15) * 4, s = (tid >> 4) * 2;
        float o[2][4];
        cost_product(sm.w2, sm.d2, make_float4(0.f, 0.f, 0.f, 0.f), tid, o);
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                sm.d1[(s + r) * kUS + u + c] = sm.h1[(s + r) * kUS + u + c] > 0.f ? o[r][c] : 0.f;
    }
    {
        // W2: a 4 x 4 tile of (j, k) summed over the samples
        const int j = (tid >> 4) * 4, k = (tid & 15) * 4;
        float g[4][4] = {};
#pragma unroll 4
        for (int s = 0; s < kCostChunk; ++s) {
            float dv[4], hv[4];
            *reinterpret_cast<float4 *>(dv) = *reinterpret_cast<const float4 *>(sm.d2 + s * kUS + j);
            *reinterpret_cast<float4 *>(hv) = *reinterpret_cast<const float4 *>(sm.h1 + s * kUS + k);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) g[r][c] = fmaf(dv[r], hv[c], g[r][c]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
            __stcg(reinterpret_cast<float4 *>(part + kOW2 + (j + r) * kCostH + k),
                   make_float4(g[r][0], g[r][1], g[r][2], g[r][3]));
    }
    __syncthreads();                                             // d1 is complete
    for (int i = tid; i < kCostH * kCostIn + 3 * kCostH + 1; i += kCostThreads) {
        float a = 0.f;
        int o;
        if (i < kCostH * kCostIn) {                              // W1
            const int j = i / kCostIn, k = i % kCostIn;
#pragma unroll 8
            for (int s = 0; s < kCostChunk; ++s) a = fmaf(sm.d1[s * kUS + j], sm.x[s * kCostIn + k], a);
            o = kOW1 + i;
        } else if (i < kCostH * (kCostIn + 1)) {                 // W3
            const int j = i - kCostH * kCostIn;
#pragma unroll 8
            for (int s = 0; s < kCostChunk; ++s) a = fmaf(sm.dout[s], sm.h2[s * kUS + j], a);
            o = kOW3 + j;
        } else if (i < kCostH * (kCostIn + 2)) {                 // b1
            const int j = i - kCostH * (kCostIn + 1);
#pragma unroll 8
            for (int s = 0; s < kCostChunk; ++s) a += sm.d1[s * kUS + j];
            o = kOB1 + j;
        } else if (i < kCostH * (kCostIn + 3)) {                 // b2
            const int j = i - kCostH * (kCostIn + 2);
#pragma unroll 8
            for (int s = 0; s < kCostChunk; ++s) a += sm.d2[s * kUS + j];
            o = kOB2 + j;
        } else {
#pragma unroll 8
            for (int s = 0; s < kCostChunk; ++s) a += sm.dout[s];
            o = kOB3;
        }
        __stcg(part + o, a);
    }
}

// All blocks of the launch: a cluster barrier, or a counter that every block
// of a cooperative grid raises (the wait gives up after kWaitNs).  Returns
// false after a wait that ran out.  stall_test: block 0 withholds its arrival
// and the wait is kStallWaitNs.
template <bool CLUSTER>
__device__ __forceinline__ bool cost_barrier(CostSmem &sm, uint32_t *sync, uint32_t &target, int stall_test) {
    if (CLUSTER) {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        return true;
    }
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (!stall_test || blockIdx.x) atomicAdd(sync, 1u);
        const unsigned long long t0 = global_ns(), limit = stall_test ? kStallWaitNs : kWaitNs;
        uint32_t v;
        int stop = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(sync) : "memory");
            if ((int)(v - target) >= 0) break;
            if (global_ns() - t0 > limit) {
                atomicExch(sync + 1, 1u);
                stop = 1;
                break;
            }
        }
        __threadfence();
        sm.stop = stop;
    }
    __syncthreads();
    return sm.stop == 0;
}

// Block b takes chunk r * gridDim + b in round r of an epoch (blocks without
// one only own parameters) and owns the parameters [b * per, (b + 1) * per),
// at most kOwn to a thread, whose moments stay in registers.  The new
// parameters and moments go to arrays of their own, so a launch whose wait ran
// out leaves the model as it was.  part: gridDim x kPart floats; grad_acc: the
// gradients carried from round to round; sync: the barrier's counter and its
// time-out flag, zeroed before the launch.
template <bool CLUSTER>
__global__ void __launch_bounds__(kCostThreads, 1)
cost_train_kernel(CostState from, CostState to, uint32_t step0,
                  const float *__restrict__ X, const float *__restrict__ y, uint32_t n, uint32_t epochs, float lr,
                  float *__restrict__ loss_out, float *__restrict__ grad_out, float *part, float *__restrict__ grad_acc,
                  uint32_t *sync, int stall_test) {
    extern __shared__ __align__(16) unsigned char cost_smem[];
    CostSmem &sm = *reinterpret_cast<CostSmem *>(cost_smem);
    float *stage = reinterpret_cast<float *>(cost_smem + sizeof(CostSmem));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t blocks = gridDim.x, b = blockIdx.x;
    const uint32_t chunks = (n + kCostChunk - 1) / kCostChunk, rounds = (chunks + blocks - 1) / blocks;
    const uint32_t per = ((uint32_t)kSqErr / 32u + blocks - 1) / blocks * 32u;
    const uint32_t i0 = min(b * per, (uint32_t)kCostP), i1 = min(i0 + per, (uint32_t)kCostP);
    const float b1m = 0.9f, b2m = 0.999f, eps = 1e-8f;
    uint32_t target = 0;
    float mo[kOwn], vo[kOwn], po[kOwn];
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
        const uint32_t i = i0 + q * kCostThreads + tid;
        mo[q] = i < i1 ? from.m[i] : 0.f;
        vo[q] = i < i1 ? from.v[i] : 0.f;
        po[q] = i < i1 ? from.params[i] : 0.f;
    }
    cost_load_params(sm, from.params, tid);
    __syncthreads();
    float loss = 0.f;                                                           // warp 0 of block 0
    for (uint32_t ep = 0; ep < epochs; ++ep) {
        const bool report = ep + 1 == epochs;
        for (uint32_t r = 0; r < rounds; ++r) {
            const uint32_t here = min(blocks, chunks - r * blocks);             // chunks of this round
            if (b < here) cost_chunk(sm, X, y, n, (r * blocks + b) * kCostChunk, part + (size_t)b * kPart, tid);
            if (!cost_barrier<CLUSTER>(sm, sync, target, stall_test)) return;
            // the owned parameters' gradients: their chunks added in order
            float g[kOwn];
#pragma unroll
            for (int q = 0; q < kOwn; ++q) {
                const uint32_t i = i0 + q * kCostThreads + tid;
                g[q] = r && i < i1 ? grad_acc[i] : 0.f;
            }
            if (here <= kCostDirect) {
#pragma unroll 8
                for (uint32_t c = 0; c < here; ++c) {
#pragma unroll
                    for (int q = 0; q < kOwn; ++q) {
                        const uint32_t i = i0 + q * kCostThreads + tid;
                        if (i < i1) g[q] += __ldcg(part + (size_t)c * kPart + i);
                    }
                }
            } else {
                // many chunks, few parameters a block (at most kCostThreads, so in g[0]):
                // all warps fetch, 32 parameters at a time; the owning warp adds
                for (uint32_t w = 0; w * 32 < i1 - i0; ++w) {
                    const uint32_t i = i0 + w * 32 + lane;
#pragma unroll 8
                    for (uint32_t c = warp; c < here; c += kCostThreads / 32)
                        stage[c * kStage + lane] = i < i1 ? __ldcg(part + (size_t)c * kPart + i) : 0.f;
                    __syncthreads();
                    if ((uint32_t)warp == w) {
#pragma unroll 8
                        for (uint32_t c = 0; c < here; ++c) g[0] += stage[c * kStage + lane];
                    }
                    __syncthreads();
                }
            }
            if (report && b == 0 && warp == 0) {
                // the loss before the last step: the squared errors in sample order
#pragma unroll 4
                for (uint32_t c = 0; c < here; ++c) {
                    const float sq = __ldcg(part + (size_t)c * kPart + kSqErr + lane);
#pragma unroll
                    for (int l = 0; l < kCostChunk; ++l) loss += __shfl_sync(0xffffffffu, sq, l);
                }
                if (lane == 0 && r + 1 == rounds) *loss_out = loss / (float)n;
            }
            if (r + 1 < rounds) {
#pragma unroll
                for (int q = 0; q < kOwn; ++q) {
                    const uint32_t i = i0 + q * kCostThreads + tid;
                    if (i < i1) grad_acc[i] = g[q];
                }
            } else if (grad_out) {                                              // gradient only
#pragma unroll
                for (int q = 0; q < kOwn; ++q) {
                    const uint32_t i = i0 + q * kCostThreads + tid;
                    if (i < i1) grad_out[i] = g[q];
                }
            } else {
                // Adam (Kingma & Ba), bias-corrected
                const float t = (float)(step0 + ep + 1);
                const float c1 = 1.f - powf(b1m, t), c2 = 1.f - powf(b2m, t);
#pragma unroll
                for (int q = 0; q < kOwn; ++q) {
                    const uint32_t i = i0 + q * kCostThreads + tid;
                    if (i < i1) {
                        const float gi = g[q];
                        const float m = b1m * mo[q] + (1.f - b1m) * gi;
                        const float v = b2m * vo[q] + (1.f - b2m) * gi * gi;
                        mo[q] = m;
                        vo[q] = v;
                        po[q] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
                        __stcg(to.params + i, po[q]);
                    }
                }
            }
            if (grad_out && r + 1 == rounds) return;
            if (!cost_barrier<CLUSTER>(sm, sync, target, stall_test)) return;
        }
        if (!report) {
            cost_load_params(sm, to.params, tid);
            __syncthreads();
        }
    }
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
        const uint32_t i = i0 + q * kCostThreads + tid;
        if (i < i1) {
            to.m[i] = mo[q];
            to.v[i] = vo[q];
        }
    }
}

// A block per 32 samples: the training kernel's forward pass.
__global__ void __launch_bounds__(kCostThreads)
cost_predict_kernel(const float *__restrict__ p, const float *__restrict__ X, uint32_t n, float *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char cost_smem[];
    CostSmem &sm = *reinterpret_cast<CostSmem *>(cost_smem);
    const int tid = threadIdx.x;
    const uint32_t c0 = blockIdx.x * kCostChunk;
    const int cn = (int)min((uint32_t)kCostChunk, n - c0);
    cost_load_x(sm, X, c0, cn, tid);
    cost_load_params(sm, p, tid);
    __syncthreads();
    const float o = cost_forward(sm, tid);
    if (tid < cn) out[c0 + tid] = o;
}

bool cost_train_grid(uint32_t n) { return n > (uint32_t)(kCostClusterMax * kCostChunk); }

// Blocks of a training launch: one per chunk, at least what the owned
// parameters need; in a grid, as many rounds as the SMs make necessary.
static uint32_t cost_blocks(uint32_t n, int num_sms, bool grid) {
    static_assert(kCostBlocksMin <= kCostClusterMax, "a cluster holds every parameter");
    if (!grid) return kCostClusterMax;
    const uint32_t chunks = n / kCostChunk + (n % kCostChunk ? 1u : 0u);
    const uint32_t rounds = (chunks + num_sms - 1) / num_sms;
    return (chunks + rounds - 1) / rounds;
}

size_t cost_train_scratch_floats(uint32_t n, int num_sms) {
    return (size_t)(std::max<uint32_t>(cost_blocks(n, num_sms, cost_train_grid(n)), kCostClusterMax) + 1) * kPart + 64;
}

// scratch: cost_train_scratch_floats(n, num_sms) floats: the chunks' gradients,
// the gradients carried between rounds, the barrier.  *sync_out: the barrier's
// words ([1] is set if a wait ran out: only a grid's can).
cudaError_t launch_cost_train(cudaStream_t st, int num_sms, bool grid, const CostState &from, const CostState &to,
                              uint32_t step0, const float *X, const float *y, uint32_t n, uint32_t epochs, float lr,
                              float *loss, float *grad, float *scratch, uint32_t **sync_out, bool stall_test) {
    const bool cluster = !grid;
    const uint32_t blocks = cost_blocks(n, num_sms, grid);
    float *part = scratch, *acc = scratch + (size_t)blocks * kPart;
    uint32_t *sync = reinterpret_cast<uint32_t *>(acc + kPart);
    *sync_out = sync;
    const size_t smem = sizeof(CostSmem) + (blocks > kCostDirect ? (size_t)blocks * kStage * sizeof(float) : 0);
    const void *f = cluster ? (const void *)cost_train_kernel<true> : (const void *)cost_train_kernel<false>;
    // the limit is the kernel's, shared by all threads: always the largest any of its launches needs
    const size_t most = sizeof(CostSmem) + (cluster ? 0 : (size_t)num_sms * kStage * sizeof(float));
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e == cudaSuccess) e = cudaMemsetAsync(sync, 0, 2 * sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr{};
    if (cluster) {
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = blocks;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    } else {                                         // every block resident: at most one per SM
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(kCostThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cluster)
        return cudaLaunchKernelEx(&cfg, cost_train_kernel<true>, from, to, step0, X, y, n, epochs, lr, loss, grad,
                                  part, acc, sync, 0);
    return cudaLaunchKernelEx(&cfg, cost_train_kernel<false>, from, to, step0, X, y, n, epochs, lr, loss, grad,
                              part, acc, sync, stall_test ? 1 : 0);
}

cudaError_t launch_cost_predict(cudaStream_t st, const float *params, const float *X, uint32_t n, float *out) {
    if (n == 0) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(cost_predict_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(CostSmem));
    if (e != cudaSuccess) return e;
    const uint32_t blocks = n / kCostChunk + (n % kCostChunk ? 1u : 0u);
    cost_predict_kernel<<<blocks, kCostThreads, sizeof(CostSmem), st>>>(params, X, n, out);
    return cudaGetLastError();
}

}  // namespace mqr
