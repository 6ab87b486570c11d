// mlp.cu -- the skin network's inference, gradient and training on the GPU
// (include/lvb_mlp.h).  bfloat16 weights and activations, binary32
// accumulation; no tensor cores: the whole network is 1,377 parameters and
// ~2.6 kFLOP per sample, far below what a contraction would need to pay.
//
// Training: a block takes kTB samples; a warp computes four units of a layer
// for 32 of them, one to a lane (forward: the exact inference formula; backward:
// straight-through the bfloat16 roundings), and then rows of the weight
// gradients, every sum in index order, into the block's own
// row of partial sums; the rows are then added in block order (no atomics), so
// training is bitwise repeatable.  Adam updates the binary32 master parameters.
// An epoch is one cooperative launch (k_mlp_epoch) for batches of up to
// kMaxTeam * kTB samples.
#include "lvb_internal.cuh"
#include "lvb_mlp.h"

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <new>
#include <random>
#include <vector>

using namespace lvb;

namespace {

constexpr int NI = LVB_MLP_IN, NH = LVB_MLP_HIDDEN, NP = LVB_MLP_PARAMS;
constexpr int OFF_W1 = 0, OFF_B1 = NH * NI, OFF_W2 = OFF_B1 + NH, OFF_B2 = OFF_W2 + NH * NH,
              OFF_W3 = OFF_B2 + NH, OFF_B3 = OFF_W3 + NH;
constexpr int kTB = 64;   // samples per training block
constexpr int kSamp = NI + 1;

__host__ __device__ inline float bf16_host_rn(float x)
{
    unsigned u;
    memcpy(&u, &x, 4);
    if ((u & 0x7f800000u) == 0x7f800000u && (u & 0x7fffffu)) return x;   // NaN
    u = (u + 0x7fffu + ((u >> 16) & 1u)) & 0xffff0000u;
    float r;
    memcpy(&r, &u, 4);
    return r;
}

__global__ void k_mlp_infer(const float *__restrict__ feats, const float *__restrict__ diam,
                            int64_t n, const lvb_mlp_weights *__restrict__ W, float *skin,
                            float *yout)
{
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = wid; i < n; i += nw) {
        float f[NI];
#pragma unroll
        for (int k = 0; k < NI; ++k) f[k] = feats[i * NI + k];
        const float y = mlp_y_warp(W, f);
        if ((threadIdx.x & 31) == 0) {
            skin[i] = mlp_skin(W, y, diam[i], f[0]);
            if (yout) yout[i] = y;
        }
    }
}

// Per-column sum and sum of squares (binary64) of the samples: the eight
// features (normalisation) and the label (output range).
// Per-warp sums of every column and of its squares (binary64), written to
// the warp's row of part (2 x kSamp values); the host adds the rows in warp
// order, so the statistics do not depend on scheduling.
constexpr int kStatBlocks = 152 * 4, kStatThreads = 256;
constexpr int kStatWarps = kStatBlocks * kStatThreads / 32;

__global__ void k_feature_stats(const float *__restrict__ samples, int64_t n, double *part)
{
    double s[kSamp] = {0}, q[kSamp] = {0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int k = 0; k < kSamp; ++k) {
            const double v = samples[i * kSamp + k];
            s[k] += v;
            q[k] += v * v;
        }
    }
#pragma unroll
    for (int k = 0; k < kSamp; ++k) {
        for (int o = 16; o; o >>= 1) {
            s[k] += __shfl_xor_sync(FULL, s[k], o);
            q[k] += __shfl_xor_sync(FULL, q[k], o);
        }
        if ((threadIdx.x & 31) == 0) {
            const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
            part[(size_t)w * 2 * kSamp + k] = s[k];
            part[(size_t)w * 2 * kSamp + kSamp + k] = q[k];
        }
    }
}

// What a block keeps in shared memory: the weights as the formulas read them
// (bfloat16 values) and, for its kTB samples, every layer's values -- unit by
// unit (suffix T: lanes take samples) and, where a gradient's lanes take units,
// also sample by sample, a column of padding apart.
constexpr int kMlpThreads = 1024, kPad = NH + 1;

struct __align__(16) MlpTile {
    // read four at a time: on 16 bytes
    float W1[NH * NI], W2[NH * NH], z[kTB][NI], d2T[NH][kTB];
    // read one at a time
    float zT[NI][kTB], h1T[NH][kTB], h1[kTB][kPad], h2T[NH][kTB], h2[kTB][kPad], d2[kTB][kPad],
        d1[kTB][kPad];
    float b1[NH], b2[NH], w3[NH], label[kTB], dy[kTB];
    double loss[2];
    float b3;
};
static_assert(offsetof(MlpTile, W1) % 16 == 0 && offsetof(MlpTile, W2) % 16 == 0 &&
                  offsetof(MlpTile, z) % 16 == 0 && offsetof(MlpTile, d2T) % 16 == 0 &&
                  NI % 4 == 0 && NH % 4 == 0 && kTB % 4 == 0,
              "rows that are read four values at a time start on 16 bytes");

// Master parameter k into the tile, as the formulas read it.
__device__ __forceinline__ void mlp_weight(MlpTile &m, int k, float v)
{
    if (k < OFF_B1) m.W1[k] = bf16_host_rn(v);
    else if (k < OFF_W2) m.b1[k - OFF_B1] = v;
    else if (k < OFF_B2) m.W2[k - OFF_W2] = bf16_host_rn(v);
    else if (k < OFF_W3) m.b2[k - OFF_B2] = v;
    else if (k < OFF_B3) m.w3[k - OFF_W3] = bf16_host_rn(v);
    else m.b3 = v;
}

// One value of a sample into the tile, normalised (thread t of the first kTB *
// kSamp: value t % kSamp of sample t / kSamp; not live: the sample is none).
__device__ __forceinline__ void mlp_sample(MlpTile &m, int t, bool live, float v, const float *mu,
                                           const float *isd)
{
    const int q = t / kSamp, k = t % kSamp;
    if (k == NI) {
        m.label[q] = v;
    } else {
        const float z = live ? bf16_rn(__fmul_rn(__fsub_rn(v, mu[k]), isd[k])) : 0.0f;
        m.zT[k][q] = z;
        m.z[q][k] = z;
    }
}

// Forward and backward pass of the tile's samples (the first `live` of them;
// the others count as nothing) and the tile's share of every parameter's
// gradient, to part[0 .. NP).  dy_scale = 2 / batch size; rel_floor > 0:
// relative error, (y - t) / max(t, rel_floor).  Returns, in thread 0, the
// tile's sum of (weighted) squared errors.  Every thread of the block; weights
// and samples in place, a block barrier behind them.
__device__ __forceinline__ double mlp_tile(MlpTile &m, int live, float dy_scale, float rel_floor,
                                           float *part)
{
    // What bounds a phase is shared memory, 128 bytes a cycle: a warp that
    // takes four units reads each value of the layer below once for four
    // sums (one unit to a warp and 64 samples: 14,400 cycles a tile, 10,600
    // this way), and the weights four to a load.
    const int lane = threadIdx.x & 31, u = threadIdx.x >> 5;
    const int g4 = (u >> 1) * 4, q = (u & 1) * 32 + lane;   // first unit, sample
    const bool layers = u < NH / 4 * 2, on = q < live;
    auto four = [](const float *p) { return *reinterpret_cast<const float4 *>(p); };
    if (layers) {
        float a[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = m.b1[g4 + j];
#pragma unroll
        for (int k = 0; k < NI; k += 4) {
            const float x[4] = {m.zT[k][q], m.zT[k + 1][q], m.zT[k + 2][q], m.zT[k + 3][q]};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 w = four(&m.W1[(g4 + j) * NI + k]);
                a[j] = fmaf(w.x, x[0], a[j]);
                a[j] = fmaf(w.y, x[1], a[j]);
                a[j] = fmaf(w.z, x[2], a[j]);
                a[j] = fmaf(w.w, x[3], a[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {   // > 0 marks the active units
            const float h = on && a[j] > 0.0f ? bf16_rn(a[j]) : 0.0f;
            m.h1T[g4 + j][q] = m.h1[q][g4 + j] = h;
        }
    }
    __syncthreads();
    if (layers) {
        float a[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = m.b2[g4 + j];
#pragma unroll
        for (int k = 0; k < NH; k += 4) {
            const float x[4] = {m.h1T[k][q], m.h1T[k + 1][q], m.h1T[k + 2][q], m.h1T[k + 3][q]};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 w = four(&m.W2[(g4 + j) * NH + k]);
                a[j] = fmaf(w.x, x[0], a[j]);
                a[j] = fmaf(w.y, x[1], a[j]);
                a[j] = fmaf(w.z, x[2], a[j]);
                a[j] = fmaf(w.w, x[3], a[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float h = on && a[j] > 0.0f ? bf16_rn(a[j]) : 0.0f;
            m.h2T[g4 + j][q] = m.h2[q][g4 + j] = h;
        }
    }
    __syncthreads();
    // the output, one sample to a lane, by two warps without units, which sum
    // the errors in binary64 while the others go back through the layers
    const int ou = u - NH / 4 * 2;
    double e = 0.0;
    if (ou >= 0 && ou < kTB / 32) {
        float y = m.b3;
#pragma unroll
        for (int k = 0; k < NH; ++k) y = fmaf(m.w3[k], m.h2T[k][ou * 32 + lane], y);
        float dy = 0.0f;
        if (ou * 32 + lane < live) {
            const float lab = m.label[ou * 32 + lane];
            const float r = y - lab;
            float w = 1.0f;   // d(loss)/d(r^2)
            if (rel_floor > 0.0f) {
                const float den = fmaxf(lab, rel_floor);
                w = 1.0f / (den * den);
            }
            dy = dy_scale * w * r;
            e = (double)w * (double)r * (double)r;
        }
        m.dy[ou * 32 + lane] = dy;
    }
    __syncthreads();
    if (layers) {
        const float dy = m.dy[q];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float d = m.h2T[g4 + j][q] > 0.0f ? dy * m.w3[g4 + j] : 0.0f;
            m.d2T[g4 + j][q] = m.d2[q][g4 + j] = d;
        }
    }
    __syncthreads();
    if (layers) {
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int o = 0; o < NH; ++o) {
            const float4 w = four(&m.W2[o * NH + g4]);
            const float d = m.d2T[o][q];
            g[0] = fmaf(d, w.x, g[0]);
            g[1] = fmaf(d, w.y, g[1]);
            g[2] = fmaf(d, w.z, g[2]);
            g[3] = fmaf(d, w.w, g[3]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) m.d1[q][g4 + j] = m.h1T[g4 + j][q] > 0.0f ? g[j] : 0.0f;
    } else if (ou < kTB / 32) {
#pragma unroll
        for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(FULL, e, o);
        if (lane == 0) m.loss[ou] = e;
    }
    __syncthreads();
    const double loss = m.loss[0] + m.loss[1];
    // The gradients, every sum over the samples in order: warps 0 .. 7 four
    // rows of W2 each, 8 and 9 four columns of W1 each, then b1, b2, w3, b3.
    if (u < 8) {
        const int o = u * 4;
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int t = 0; t < kTB; t += 4) {
            const float h[4] = {m.h1[t][lane], m.h1[t + 1][lane], m.h1[t + 2][lane],
                                m.h1[t + 3][lane]};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 d = four(&m.d2T[o + j][t]);
                g[j] = fmaf(d.x, h[0], g[j]);
                g[j] = fmaf(d.y, h[1], g[j]);
                g[j] = fmaf(d.z, h[2], g[j]);
                g[j] = fmaf(d.w, h[3], g[j]);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) part[OFF_W2 + (o + j) * NH + lane] = g[j];
    } else if (u < 10) {
        const int k = (u - 8) * 4;
        float g[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
        for (int t = 0; t < kTB; ++t) {
            const float d = m.d1[t][lane];
            const float4 z = four(&m.z[t][k]);
            g[0] = fmaf(d, z.x, g[0]);
            g[1] = fmaf(d, z.y, g[1]);
            g[2] = fmaf(d, z.z, g[2]);
            g[3] = fmaf(d, z.w, g[3]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) part[OFF_W1 + lane * NI + k + j] = g[j];
    } else if (u == 10) {
        float g = 0.0f;
#pragma unroll 16
        for (int t = 0; t < kTB; ++t) g += m.d1[t][lane];
        part[OFF_B1 + lane] = g;
    } else if (u == 11) {
        float g = 0.0f;
#pragma unroll 16
        for (int t = 0; t < kTB; ++t) g += m.d2[t][lane];
        part[OFF_B2 + lane] = g;
    } else if (u == 12) {
        float g = 0.0f;
#pragma unroll 16
        for (int t = 0; t < kTB; ++t) g = fmaf(m.dy[t], m.h2[t][lane], g);
        part[OFF_W3 + lane] = g;
    } else if (u == 13) {
        float g = 0.0f;
#pragma unroll 16
        for (int t = 0; t < kTB; ++t) g += m.dy[t];
        if (lane == 0) part[OFF_B3] = g;
    }
    return loss;
}

struct TrainArgs {
    const float *samples;   // n x 9
    const int *order;       // sample index of each position (null: identity)
    int64_t first, count;   // positions [first, first + count) form the batch
    const float *params;    // master parameters
    const float *mu, *isd;
    float *part;            // per-block partial gradients (blocks x NP)
    double *loss;           // accumulated sum of (weighted) squared errors
    float dy_scale;         // 2 / batch size
    float rel_floor;        // > 0: relative error, (y - t) / max(t, rel_floor)
};

__global__ void __launch_bounds__(kMlpThreads)
k_mlp_batch(TrainArgs a)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpTile &m = *reinterpret_cast<MlpTile *>(mlp_smem);
    const int t = threadIdx.x;
    const int64_t first = a.first + (int64_t)blockIdx.x * kTB;
    const int live = (int)min((int64_t)kTB, a.first + a.count - first);
    for (int k = t; k < NP; k += kMlpThreads) mlp_weight(m, k, a.params[k]);
    if (t < kTB * kSamp) {
        const bool on = t / kSamp < live;
        const int64_t pos = first + t / kSamp;
        const int64_t si = !on ? 0 : a.order ? a.order[pos] : pos;
        mlp_sample(m, t, on, on ? a.samples[si * kSamp + t % kSamp] : 0.0f, a.mu, a.isd);
    }
    __syncthreads();
    const double e = mlp_tile(m, live, a.dy_scale, a.rel_floor, a.part + (size_t)blockIdx.x * NP);
    if (t == 0) atomicAdd(a.loss, e);
}

// grad[i] += the nb blocks' partial sums of parameter i, in block order.
__global__ void k_fold_parts(const float *part, int nb, float *grad)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NP) return;
    float g = grad[i];
    for (int b = 0; b < nb; ++b) g += part[(size_t)b * NP + i];
    grad[i] = g;
}

struct AdamStep {
    float lr, b1, b2, eps;
};

__device__ __forceinline__ void adam(const AdamStep &s, float gi, float c1, float c2, float &p,
                                     float &m, float &v)
{
    // the fused products written out, so that every kernel rounds alike
    const float mi = fmaf(1.0f - s.b1, gi, __fmul_rn(s.b1, m));
    const float vi = fmaf(__fmul_rn(1.0f - s.b2, gi), gi, __fmul_rn(s.b2, v));
    m = mi;
    v = vi;
    p -= s.lr * (mi / c1) / (sqrtf(vi / c2) + s.eps);
}

// One Adam step; the gradient is the sum of the nb blocks' partials, added
// in block order.
__global__ void k_adam(float *p, const float *part, int nb, float *m, float *v, int n, AdamStep s,
                       float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gi = 0.0f;
    for (int b = 0; b < nb; ++b) gi += part[(size_t)b * NP + i];
    adam(s, gi, c1, c2, p[i], m[i], v[i]);
}

// An epoch of training in one cooperative launch: every batch in turn, block b
// taking its b-th kTB samples.  Each block keeps the master parameters and
// Adam's moments in shared memory; after a batch it adds up all blocks' partial
// sums and takes the same Adam step as every other, so one grid barrier a
// batch is enough (the partial sums go to two sets of rows in turn).  The next
// batch's samples are loaded under this one.  What bounds it is the chain of
// a batch: six layers' sums of 8 to 64 terms each, a barrier, the partial sums --
// 10.8 us for 512 samples, against 37 us with a launch for each batch (one thread to a
// sample) and one for each step.
constexpr int kMaxTeam = 64;             // blocks of an epoch's launch
constexpr int kEpochSpins = 1 << 22;      // polls before a barrier gives up

struct EpochArgs {
    const float *samples;
    const int *order;
    int64_t n;
    int batch;
    float *params, *m, *v;
    const float *mu, *isd;
    float *part;                         // 2 x blocks x NP
    double *loss;
    const float *c12;                    // c1, c2 of each batch
    AdamStep adam;
    float rel_floor;
    unsigned long long *arrived;         // grid barrier, zero at the start
    unsigned *failed;
    unsigned extra, spins;               // arrivals waited for beyond the blocks', polls
};

struct EpochShared {
    MlpTile tile;
    float p[NP], m[NP], v[NP], mu[NI], isd[NI];
    int ok;
};

__global__ void __launch_bounds__(kMlpThreads)
k_mlp_epoch(EpochArgs a)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    EpochShared &s = *reinterpret_cast<EpochShared *>(mlp_smem);
    const int t = threadIdx.x;
    for (int k = t; k < NP; k += kMlpThreads) {
        s.p[k] = a.params[k];
        s.m[k] = a.m[k];
        s.v[k] = a.v[k];
        mlp_weight(s.tile, k, s.p[k]);
    }
    if (t < NI) {
        s.mu[t] = a.mu[t];
        s.isd[t] = a.isd[t];
    }
    __syncthreads();
    const bool loads = t < kTB * kSamp;
    // this thread's value of its sample in the batch that starts at `first`
    auto live_of = [&](int64_t first) {
        const int64_t cnt = min((int64_t)a.batch, a.n - first) - (int64_t)blockIdx.x * kTB;
        return (int)max((int64_t)0, min((int64_t)kTB, cnt));
    };
    auto value = [&](int64_t first) {
        if (!loads || first >= a.n || t / kSamp >= live_of(first)) return 0.0f;
        const int64_t pos = first + (int64_t)blockIdx.x * kTB + t / kSamp;
        return a.samples[(int64_t)a.order[pos] * kSamp + t % kSamp];
    };
    float next = value(0);
    double loss = 0.0;
    int step = 0;
    for (int64_t first = 0; first < a.n; first += a.batch, ++step) {
        const int64_t cnt = min((int64_t)a.batch, a.n - first);
        const int nb = (int)((cnt + kTB - 1) / kTB), live = live_of(first);
        float *part = a.part + (size_t)(step & 1) * gridDim.x * NP;
        const float c1 = a.c12[2 * step], c2 = a.c12[2 * step + 1];
        if (live > 0) {
            if (loads) mlp_sample(s.tile, t, t / kSamp < live, next, s.mu, s.isd);
            __syncthreads();
            next = value(first + a.batch);
            loss += mlp_tile(s.tile, live, 2.0f / (float)cnt, a.rel_floor,
                             part + (size_t)blockIdx.x * NP);
        } else {
            next = value(first + a.batch);
        }
        __syncthreads();
        if (gridDim.x > 1 || a.extra) {
            if (t == 0) {
                const unsigned long long need =
                    (unsigned long long)(step + 1) * gridDim.x + a.extra;
                asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(a.arrived), "l"(1ULL)
                             : "memory");
                unsigned long long got = 0;
                unsigned it = 0;
                do {
                    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];"
                                 : "=l"(got) : "l"(a.arrived) : "memory");
                } while (got < need && ++it <= a.spins);
                if (got < need) atomicOr(a.failed, 1u);
                s.ok = got >= need;
            }
            __syncthreads();
            if (!s.ok) return;
        }
        // parameters t and t + 1024 together: one latency of the partial
        // sums for each eight blocks, added in order
        const int k1 = t + kMlpThreads < NP ? t + kMlpThreads : t;
        float g0 = 0.0f, g1 = 0.0f;
        for (int b0 = 0; b0 < nb; b0 += 8) {
            float v0[8], v1[8];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const float *row = part + (size_t)min(b0 + x, nb - 1) * NP;
                v0[x] = row[t];
                v1[x] = row[k1];
            }
#pragma unroll
            for (int x = 0; x < 8; ++x)
                if (b0 + x < nb) {
                    g0 += v0[x];
                    g1 += v1[x];
                }
        }
        adam(a.adam, g0, c1, c2, s.p[t], s.m[t], s.v[t]);
        mlp_weight(s.tile, t, s.p[t]);
        if (k1 != t) {
            adam(a.adam, g1, c1, c2, s.p[k1], s.m[k1], s.v[k1]);
            mlp_weight(s.tile, k1, s.p[k1]);
        }
        __syncthreads();
    }
    if (t == 0 && loss != 0.0) atomicAdd(a.loss, loss);
    if (blockIdx.x == 0)
        for (int k = t; k < NP; k += kMlpThreads) {
            a.params[k] = s.p[k];
            a.m[k] = s.m[k];
            a.v[k] = s.v[k];
        }
}

int from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return LVB_OK;
    if (e == cudaErrorMemoryAllocation) return LVB_ENOMEM;
    return LVB_EDEVICE;
}

struct DevBuf {
    void *p = nullptr;
    ~DevBuf()
    {
        if (p) cudaFree(p);
    }
};

template <class T>
cudaError_t dnew(DevBuf &b, size_t count)
{
    return cudaMalloc(&b.p, sizeof(T) * std::max<size_t>(count, 1));
}

// one pass of k_mlp_batch over positions [first, first + count) of a mean
// over `total` samples; returns the number of blocks (rows of part)
int launch_batch(const float *samples, const int *order, int64_t first, int64_t count,
                 int64_t total, const float *params, const float *mu, const float *isd,
                 float *part, double *loss, float rel_floor, cudaStream_t st)
{
    TrainArgs a;
    a.samples = samples;
    a.order = order;
    a.first = first;
    a.count = count;
    a.params = params;
    a.mu = mu;
    a.isd = isd;
    a.part = part;
    a.loss = loss;
    a.dy_scale = 2.0f / (float)total;
    a.rel_floor = rel_floor;
    const int64_t blocks = (count + kTB - 1) / kTB;
    k_mlp_batch<<<(unsigned)blocks, kMlpThreads, sizeof(MlpTile), st>>>(a);
    return (int)blocks;
}

// Blocks of an epoch's launch that are resident on the device at once.
int epoch_blocks(cudaError_t *e)
{
    int dev = 0, sms = 0, per_sm = 0;
    *e = cudaGetDevice(&dev);
    if (*e == cudaSuccess) *e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (*e == cudaSuccess)
        *e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mlp_epoch, kMlpThreads,
                                                           sizeof(EpochShared));
    return per_sm * sms;
}

constexpr int64_t kGradChunk = 1024 * kTB;   // samples per pass of lvb_mlp_grad

// The training kernels' shared memory, above the default limit (per kernel and
// device; asked for at every call).
cudaError_t allow_shared()
{
    cudaError_t e = cudaFuncSetAttribute(k_mlp_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(MlpTile));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_mlp_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(EpochShared));
    return e;
}

}  // namespace

extern "C" {

int lvb_mlp_pack(const float *params, const float *mu, const float *isd, const float *y_range,
                 float y_steps, lvb_mlp_weights *out)
{
    if (!params || !mu || !isd || !out) return LVB_EINVAL;
    if (y_range && !(y_range[0] <= y_range[1])) return LVB_EINVAL;
    if (!(y_steps >= 0.0f) || !std::isfinite(y_steps)) return LVB_EINVAL;
    lvb_mlp_weights w;
    memset(&w, 0, sizeof(w));
    w.y_lo = y_range ? y_range[0] : 0.0f;
    w.y_hi = y_range ? y_range[1] : INFINITY;
    w.y_steps = y_steps;
    // input-major device layout (lvb_mlp.h) from the [out][in] master form
    for (int o = 0; o < NH; ++o)
        for (int k = 0; k < NI; ++k) w.W1[k * NH + o] = bf16_host_rn(params[OFF_W1 + o * NI + k]);
    for (int k = 0; k < NH; ++k) w.b1[k] = params[OFF_B1 + k];
    for (int o = 0; o < NH; ++o)
        for (int k = 0; k < NH; ++k) w.W2[k * NH + o] = bf16_host_rn(params[OFF_W2 + o * NH + k]);
    for (int k = 0; k < NH; ++k) w.b2[k] = params[OFF_B2 + k];
    for (int k = 0; k < NH; ++k) w.w3[k] = bf16_host_rn(params[OFF_W3 + k]);
    w.b3 = params[OFF_B3];
    for (int k = 0; k < NI; ++k) {
        w.mu[k] = mu[k];
        w.isd[k] = isd[k];
    }
    return from_cuda(cudaMemcpy(out, &w, sizeof(w), cudaMemcpyDefault));
}

int lvb_mlp_infer(const float *feats, const float *diam, int64_t n, const lvb_mlp_weights *w,
                  float *skin, float *y, void *stream)
{
    if (!feats || !diam || !w || !skin || n < 0) return LVB_EINVAL;
    if (n == 0) return LVB_OK;
    cudaGetLastError();
    const int64_t blocks = std::min<int64_t>((n * 32 + 255) / 256, 152 * 16);
    k_mlp_infer<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(feats, diam, n, w, skin, y);
    return from_cuda(cudaGetLastError());
}

int lvb_mlp_grad(const float *samples, int64_t n, const float *params, const float *mu,
                 const float *isd, float rel_floor, float *grad, double *loss, void *stream)
{
    if (!samples || n < 1 || !params || !mu || !isd || !grad || !loss) return LVB_EINVAL;
    if (!(rel_floor >= 0.0f)) return LVB_EINVAL;
    cudaGetLastError();
    const cudaStream_t st = (cudaStream_t)stream;
    DevBuf dp, dmu, disd, dg, dl, dpart;
    cudaError_t e = allow_shared();
    if (e == cudaSuccess) e = dnew<float>(dp, NP);
    if (e == cudaSuccess) e = dnew<float>(dmu, NI);
    if (e == cudaSuccess) e = dnew<float>(disd, NI);
    if (e == cudaSuccess) e = dnew<float>(dg, NP);
    if (e == cudaSuccess) e = dnew<double>(dl, 1);
    if (e == cudaSuccess)
        e = dnew<float>(dpart, (size_t)((std::min(n, kGradChunk) + kTB - 1) / kTB) * NP);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dp.p, params, NP * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dmu.p, mu, NI * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(disd.p, isd, NI * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dg.p, 0, NP * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dl.p, 0, 8, st);
    if (e != cudaSuccess) return from_cuda(e);
    for (int64_t first = 0; first < n; first += kGradChunk) {
        const int nb = launch_batch(samples, nullptr, first, std::min(kGradChunk, n - first), n,
                                    (const float *)dp.p, (const float *)dmu.p,
                                    (const float *)disd.p, (float *)dpart.p, (double *)dl.p,
                                    rel_floor, st);
        k_fold_parts<<<(NP + 255) / 256, 256, 0, st>>>((const float *)dpart.p, nb, (float *)dg.p);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad, dg.p, NP * 4, cudaMemcpyDeviceToHost, st);
    double sse = 0.0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, dl.p, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return from_cuda(e);
    *loss = sse / (double)n;
    return LVB_OK;
}

int lvb_mlp_train(const float *samples, int64_t n, int32_t epochs, int32_t batch, float lr,
                  uint64_t seed, int32_t loss_kind, float *params, float *mu, float *isd,
                  float *y_range, float *losses, void *stream)
{
    return lvb_mlp_train_limits(samples, n, epochs, batch, lr, seed, loss_kind, params, mu, isd,
                                y_range, losses, stream, kMaxTeam, 0, kEpochSpins);
}

int lvb_mlp_train_limits(const float *samples, int64_t n, int32_t epochs, int32_t batch, float lr,
                         uint64_t seed, int32_t loss_kind, float *params, float *mu, float *isd,
                         float *y_range, float *losses, void *stream, int32_t blocks_max,
                         int32_t extra, int32_t spins)
{
    if (!samples || n < 1 || epochs < 1 || batch < 1 || !(lr > 0.0f) || !params || !mu || !isd ||
        !y_range)
        return LVB_EINVAL;
    if (loss_kind != LVB_MLP_LOSS_SQUARED && loss_kind != LVB_MLP_LOSS_RELATIVE)
        return LVB_EINVAL;
    if (n > INT32_MAX) return LVB_EINVAL;
    if (blocks_max < 0 || extra < 0 || extra > 1 || spins < 1 || spins > kEpochSpins)
        return LVB_EINVAL;
    cudaGetLastError();
    const cudaStream_t st = (cudaStream_t)stream;
    // feature normalisation from the samples (mean, 1/std), label range
    DevBuf dstat;
    cudaError_t e = dnew<double>(dstat, (size_t)kStatWarps * 2 * kSamp);
    if (e != cudaSuccess) return from_cuda(e);
    k_feature_stats<<<kStatBlocks, kStatThreads, 0, st>>>(samples, n, (double *)dstat.p);
    // the warps beyond the samples have nothing to add
    const int warps = (int)std::min<int64_t>(kStatWarps, (n + 31) / 32);
    std::vector<double> parts((size_t)warps * 2 * kSamp);
    e = cudaMemcpyAsync(parts.data(), dstat.p, sizeof(double) * parts.size(),
                        cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return from_cuda(e);
    double stat[2 * kSamp] = {0};
    for (int w = 0; w < warps; ++w)
        for (int k = 0; k < 2 * kSamp; ++k) stat[k] += parts[(size_t)w * 2 * kSamp + k];
    for (int k = 0; k < NI; ++k) {
        const double m = stat[k] / (double)n;
        const double var = std::max(stat[kSamp + k] / (double)n - m * m, 0.0);
        mu[k] = (float)m;
        isd[k] = var > 1e-30 ? (float)(1.0 / std::sqrt(var)) : 1.0f;
    }
    {
        const double m = stat[NI] / (double)n;
        const double sd = std::sqrt(std::max(stat[kSamp + NI] / (double)n - m * m, 0.0));
        y_range[0] = (float)(m / 16.0);
        y_range[1] = (float)(m + 4.0 * sd);
    }
    // relative error: labels below the output range's floor count as the floor
    const float rel_floor = loss_kind == LVB_MLP_LOSS_RELATIVE ? std::max(y_range[0], 1e-30f)
                                                               : 0.0f;
    // batches of up to kMaxTeam blocks that the device holds at once: an epoch to
    // a launch; larger ones: a launch for each batch and for each Adam step (the
    // same sums and steps)
    const int64_t batches = (n + batch - 1) / batch;
    const int64_t blocks = (std::min<int64_t>(batch, n) + kTB - 1) / kTB;
    DevBuf dp, dmu, disd, dg, dm, dv, dl, dord, dc, dbar;
    e = allow_shared();
    const int resident = e == cudaSuccess ? epoch_blocks(&e) : 0;
    const bool epoch_launch =
        blocks <= std::min(std::min(kMaxTeam, resident), (int)blocks_max);
    if (e == cudaSuccess) e = dnew<float>(dp, NP);
    if (e == cudaSuccess) e = dnew<float>(dmu, NI);
    if (e == cudaSuccess) e = dnew<float>(disd, NI);
    if (e == cudaSuccess) e = dnew<float>(dg, (size_t)(epoch_launch ? 2 : 1) * blocks * NP);
    if (e == cudaSuccess) e = dnew<float>(dm, NP);
    if (e == cudaSuccess) e = dnew<float>(dv, NP);
    if (e == cudaSuccess) e = dnew<double>(dl, 1);
    if (e == cudaSuccess) e = dnew<int>(dord, (size_t)n);
    if (e == cudaSuccess && epoch_launch) e = dnew<float>(dc, (size_t)batches * 2);
    if (e == cudaSuccess && epoch_launch) e = dnew<unsigned long long>(dbar, 2);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dp.p, params, NP * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dmu.p, mu, NI * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(disd.p, isd, NI * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dm.p, 0, NP * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dv.p, 0, NP * 4, st);
    if (e != cudaSuccess) return from_cuda(e);
    std::vector<int> order, later;   // this epoch's order and the next one's
    std::vector<float> c12;
    try {
        order.resize((size_t)n);
        if (epochs > 1) later.resize((size_t)n);
        if (epoch_launch) c12.resize((size_t)batches * 2);
    } catch (const std::bad_alloc &) {
        return LVB_ENOMEM;
    }
    for (int64_t i = 0; i < n; ++i) order[(size_t)i] = (int)i;
    std::mt19937_64 rng(seed);
    const AdamStep ad{lr, 0.9f, 0.999f, 1e-8f};
    int64_t t = 0;
    std::shuffle(order.begin(), order.end(), rng);
    for (int ep = 0; ep < epochs; ++ep) {
        e = cudaMemcpyAsync(dord.p, order.data(), sizeof(int) * (size_t)n, cudaMemcpyHostToDevice,
                            st);
        if (e == cudaSuccess) e = cudaMemsetAsync(dl.p, 0, 8, st);
        if (e != cudaSuccess) return from_cuda(e);
        if (epoch_launch) {
            for (int64_t b = 0; b < batches; ++b) {
                ++t;
                c12[(size_t)(2 * b)] = 1.0f - std::pow(ad.b1, (float)t);
                c12[(size_t)(2 * b + 1)] = 1.0f - std::pow(ad.b2, (float)t);
            }
            e = cudaMemcpyAsync(dc.p, c12.data(), sizeof(float) * c12.size(),
                                cudaMemcpyHostToDevice, st);
            if (e == cudaSuccess) e = cudaMemsetAsync(dbar.p, 0, 16, st);
            if (e != cudaSuccess) return from_cuda(e);
            EpochArgs a;
            a.samples = samples;
            a.order = (const int *)dord.p;
            a.n = n;
            a.batch = batch;
            a.params = (float *)dp.p;
            a.m = (float *)dm.p;
            a.v = (float *)dv.p;
            a.mu = (const float *)dmu.p;
            a.isd = (const float *)disd.p;
            a.part = (float *)dg.p;
            a.loss = (double *)dl.p;
            a.c12 = (const float *)dc.p;
            a.adam = ad;
            a.rel_floor = rel_floor;
            a.arrived = (unsigned long long *)dbar.p;
            a.failed = (unsigned *)((unsigned long long *)dbar.p + 1);
            a.extra = (unsigned)extra;
            a.spins = (unsigned)spins;
            e = launch_coop(k_mlp_epoch, dim3((unsigned)blocks), dim3(kMlpThreads),
                            sizeof(EpochShared), st, a);
        } else {
            for (int64_t first = 0; first < n; first += batch) {
                const int64_t cnt = std::min<int64_t>(batch, n - first);
                const int nb = launch_batch(samples, (const int *)dord.p, first, cnt, cnt,
                                            (const float *)dp.p, (const float *)dmu.p,
                                            (const float *)disd.p, (float *)dg.p, (double *)dl.p,
                                            rel_floor, st);
                ++t;
                const float c1 = 1.0f - std::pow(ad.b1, (float)t);
                const float c2 = 1.0f - std::pow(ad.b2, (float)t);
                k_adam<<<(NP + 255) / 256, 256, 0, st>>>((float *)dp.p, (const float *)dg.p, nb,
                                                         (float *)dm.p, (float *)dv.p, NP, ad, c1,
                                                         c2);
            }
            e = cudaGetLastError();
        }
        // the next epoch's order, in a buffer of its own, while the GPU works
        // on this one's
        if (ep + 1 < epochs) {
            later = order;
            std::shuffle(later.begin(), later.end(), rng);
        }
        double sse = 0.0;
        unsigned failed = 0;
        if (e == cudaSuccess) e = cudaMemcpyAsync(&sse, dl.p, 8, cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess && epoch_launch)
            e = cudaMemcpyAsync(&failed, (unsigned long long *)dbar.p + 1, sizeof(failed),
                                cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return from_cuda(e);
        if (failed) return LVB_ETIMEOUT;
        if (losses) losses[ep] = (float)(sse / (double)n);
        std::swap(order, later);
    }
    e = cudaMemcpyAsync(params, dp.p, NP * 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return from_cuda(e);
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Travel-form labels (lvb_mlp_travel_labels): samples with f0 > 0 kept in
// their order (chunked stable compaction: block b owns a contiguous chunk
// and writes its kept samples after those of the blocks before it), label
// t -> (t * margin) / (f0 * horizon), then clipped at an order statistic
// found by bisection over the binary32 bit patterns (non-negative values
// order like their bits).
// ---------------------------------------------------------------------------
namespace {

constexpr int kTlThreads = 256;
constexpr int kTlBlocks = 256;

__device__ __forceinline__ bool tl_keep(const float *s) { return s[0] > 0.0f; }

__global__ void __launch_bounds__(kTlThreads)
k_tl_count(const float *__restrict__ smp, int64_t n, int64_t chunk, int *blk_cnt)
{
    const int64_t a = (int64_t)blockIdx.x * chunk, b = min(n, a + chunk);
    int c = 0;
    for (int64_t i = a + threadIdx.x; i < b; i += kTlThreads) c += tl_keep(smp + i * kSamp);
    __shared__ int ws[kTlThreads / 32];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kTlThreads / 32; ++w) t += ws[w];
        blk_cnt[blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(kTlThreads)
k_tl_scatter(const float *__restrict__ smp, int64_t n, int64_t chunk, const int *blk_cnt,
             int horizon, float margin, float *__restrict__ out)
{
    __shared__ int ws[kTlThreads / 32];
    __shared__ int s_base;
    if (threadIdx.x == 0) {
        int base = 0;
        for (int q = 0; q < (int)blockIdx.x; ++q) base += blk_cnt[q];
        s_base = base;
    }
    __syncthreads();
    int base = s_base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t a = (int64_t)blockIdx.x * chunk, b = min(n, a + chunk);
    const float hz = (float)horizon;
    for (int64_t t0 = a; t0 < b; t0 += kTlThreads) {
        const int64_t i = t0 + threadIdx.x;
        const bool keep = i < b && tl_keep(smp + i * kSamp);
        const unsigned m = __ballot_sync(FULL, keep);
        if (lane == 0) ws[warp] = __popc(m);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < kTlThreads / 32; ++w) {
            before += w < warp ? ws[w] : 0;
            total += ws[w];
        }
        if (keep) {
            const float *s = smp + i * kSamp;
            float *o = out + (int64_t)(base + before + __popc(m & lanemask_lt())) * kSamp;
#pragma unroll
            for (int k = 0; k < NI; ++k) o[k] = s[k];
            o[NI] = __fdiv_rn(__fmul_rn(s[NI], margin), __fmul_rn(s[0], hz));
        }
        base += total;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kTlThreads)
k_tl_count_le(const float *__restrict__ out, int64_t m, unsigned t, unsigned long long *cnt)
{
    unsigned long long c = 0;
    for (int64_t i = (int64_t)blockIdx.x * kTlThreads + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * kTlThreads)
        c += __float_as_uint(out[i * kSamp + NI]) <= t;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(cnt, c);
}

__global__ void __launch_bounds__(kTlThreads)
k_tl_clip(float *out, int64_t m, float c)
{
    for (int64_t i = (int64_t)blockIdx.x * kTlThreads + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * kTlThreads)
        out[i * kSamp + NI] = fminf(out[i * kSamp + NI], c);
}

}  // namespace

extern "C" int lvb_mlp_travel_labels(const float *samples, int64_t n, int32_t horizon,
                                     float margin, float clip_q, float *out, int64_t *n_out,
                                     void *stream)
{
    if (n_out) *n_out = 0;
    if (!samples || !out || !n_out || n < 0 || horizon < 1 || samples == out) return LVB_EINVAL;
    if (!(margin > 0.0f) || !std::isfinite(margin) || !(clip_q > 0.0f) || !(clip_q <= 1.0f))
        return LVB_EINVAL;
    if (n == 0) return LVB_OK;
    const cudaStream_t st = (cudaStream_t)stream;
    const int64_t chunk = (n + kTlBlocks - 1) / kTlBlocks;
    int *blk = nullptr;
    unsigned long long *cnt = nullptr;
    cudaError_t e = cudaMalloc((void **)&blk, sizeof(int) * kTlBlocks);
    if (e == cudaSuccess) e = cudaMalloc((void **)&cnt, sizeof(unsigned long long));
    auto done = [&](int rc) {
        cudaStreamSynchronize(st);
        if (blk) cudaFree(blk);
        if (cnt) cudaFree(cnt);
        return rc;
    };
    if (e != cudaSuccess) return done(e == cudaErrorMemoryAllocation ? LVB_ENOMEM : LVB_EDEVICE);
    k_tl_count<<<kTlBlocks, kTlThreads, 0, st>>>(samples, n, chunk, blk);
    k_tl_scatter<<<kTlBlocks, kTlThreads, 0, st>>>(samples, n, chunk, blk, horizon, margin, out);
    std::vector<int> bc(kTlBlocks);
    e = cudaMemcpyAsync(bc.data(), blk, sizeof(int) * kTlBlocks, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return done(LVB_EDEVICE);
    int64_t m = 0;
    for (int v : bc) m += v;
    if (m > 0) {
        // order statistic k (0-based, ascending): the smallest bit pattern
        // t with at least k + 1 labels <= t
        const int64_t k = (int64_t)std::floor((double)clip_q * (double)(m - 1));
        const int g = (int)std::min<int64_t>((m + kTlThreads - 1) / kTlThreads, 4 * 152);
        unsigned lo = 0u, hi = 0x7fffffffu;
        while (lo < hi && e == cudaSuccess) {
            const unsigned mid = lo + (hi - lo) / 2;
            unsigned long long c = 0;
            e = cudaMemsetAsync(cnt, 0, sizeof(c), st);
            if (e == cudaSuccess) {
                k_tl_count_le<<<g, kTlThreads, 0, st>>>(out, m, mid, cnt);
                e = cudaMemcpyAsync(&c, cnt, sizeof(c), cudaMemcpyDeviceToHost, st);
            }
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            if ((int64_t)c >= k + 1) hi = mid;
            else lo = mid + 1;
        }
        if (e != cudaSuccess) return done(LVB_EDEVICE);
        float c;
        memcpy(&c, &lo, sizeof(c));
        k_tl_clip<<<g, kTlThreads, 0, st>>>(out, m, c);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return done(LVB_EDEVICE);
    *n_out = m;
    return done(LVB_OK);
}
