// clumps.cu -- narrow phase of multi-sphere clumps on the list
// (include/lvb_clump.h): the broad phase runs on the clumps' bounding
// spheres, and every clump pair of its list is resolved into the contacts
// of their sub-spheres, each at its world position x_i + R(q_i) b_a.
#include "lvb_internal.cuh"
#include "lvb_clump.h"

#include <algorithm>
#include <cmath>

using namespace lvb;

namespace {

constexpr int kThreads = 256;
constexpr int kMaxSub = 64;

enum : unsigned { CL_BAD_QUAT = 1u, CL_BAD_BOUND = 2u, CL_BAD_OFFSETS = 4u, CL_BAD_VALUE = 8u };

// The rotation matrix of a unit quaternion (w, x, y, z), each entry in
// binary32 with the roundings of lvb_clump.h.
__device__ __forceinline__ void rotmat(float4 q, float R[9])
{
    const float w = q.x, x = q.y, y = q.z, z = q.w;
    R[0] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(__fmul_rn(y, y), __fmul_rn(z, z))));
    R[1] = __fmul_rn(2.0f, __fsub_rn(__fmul_rn(x, y), __fmul_rn(w, z)));
    R[2] = __fmul_rn(2.0f, __fadd_rn(__fmul_rn(x, z), __fmul_rn(w, y)));
    R[3] = __fmul_rn(2.0f, __fadd_rn(__fmul_rn(x, y), __fmul_rn(w, z)));
    R[4] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(__fmul_rn(x, x), __fmul_rn(z, z))));
    R[5] = __fmul_rn(2.0f, __fsub_rn(__fmul_rn(y, z), __fmul_rn(w, x)));
    R[6] = __fmul_rn(2.0f, __fsub_rn(__fmul_rn(x, z), __fmul_rn(w, y)));
    R[7] = __fmul_rn(2.0f, __fadd_rn(__fmul_rn(y, z), __fmul_rn(w, x)));
    R[8] = __fsub_rn(1.0f, __fmul_rn(2.0f, __fadd_rn(__fmul_rn(x, x), __fmul_rn(y, y))));
}

// World position and radius of a sub-sphere (b: body offset and radius).
__device__ __forceinline__ float4 world(float4 c, const float R[9], float4 b)
{
    float4 o;
    o.x = __fadd_rn(c.x, __fadd_rn(__fadd_rn(__fmul_rn(R[0], b.x), __fmul_rn(R[1], b.y)),
                                   __fmul_rn(R[2], b.z)));
    o.y = __fadd_rn(c.y, __fadd_rn(__fadd_rn(__fmul_rn(R[3], b.x), __fmul_rn(R[4], b.y)),
                                   __fmul_rn(R[5], b.z)));
    o.z = __fadd_rn(c.z, __fadd_rn(__fadd_rn(__fmul_rn(R[6], b.x), __fmul_rn(R[7], b.y)),
                                   __fmul_rn(R[8], b.z)));
    o.w = b.w;
    return o;
}

// exact a + b = s + e
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// A quaternion's |q|^2 within 2^-19 of 1, in binary64; binary32 decides where
// its rounding (4e-7) leaves no doubt.
__device__ __forceinline__ bool unit(float4 q)
{
    const float f = q.x * q.x + q.y * q.y + q.z * q.z + q.w * q.w;
    if (fabsf(f - 1.0f) <= 1.4e-6f) return true;
    const double qq = (double)q.x * q.x + (double)q.y * q.y + (double)q.z * q.z +
                      (double)q.w * q.w;
    return fabs(qq - 1.0) <= 1.0 / 524288.0;
}

// |b| + r <= R (1 - 2^-12) in binary64.  One sub-sphere of each clump usually
// lies right at the bound, and binary64 is slow on this part (one instruction
// of a warp in 16 cycles an SM), so the squares |b|^2 and (R (1 - 2^-12) - r)^2
// are compared first in binary32, then in pairs of binary32 (error-free
// transformations, Knuth and Dekker: relative error about 2^-44), each with a
// margin far above its rounding; only what is closer than 1e-12 takes the
// binary64 square root.  (Squares too small or too large for binary32 tell
// nothing and go there too.)
__device__ __forceinline__ bool inside(float4 b, float R)
{
    const float tf = R * (1.0f - 1.0f / 4096.0f) * 0.999998f - b.w;
    if (tf > 0.0f && (b.x * b.x + b.y * b.y + b.z * b.z) < tf * tf * 0.999998f) return true;
    float bh, bl, th, tl, u, v, sh, sl;
    two_sum(R, -R * (1.0f / 4096.0f), bh, bl);      // R (1 - 2^-12), exact
    two_sum(bh, -b.w, th, tl);                      // less r
    tl += bl;
    const float p = __fmul_rn(th, th);
    const float pl = fmaf(th, th, -p) + 2.0f * th * tl;
    const float x2 = __fmul_rn(b.x, b.x), y2 = __fmul_rn(b.y, b.y), z2 = __fmul_rn(b.z, b.z);
    two_sum(x2, y2, u, v);
    two_sum(u, z2, sh, sl);
    sl += v + (fmaf(b.x, b.x, -x2) + fmaf(b.y, b.y, -y2) + fmaf(b.z, b.z, -z2));
    if (th > 0.0f && p > 1e-30f && p < 1e30f && __fsub_rn(p, sh) + (pl - sl) > 1e-12f * p) return true;
    const double s = (double)b.x * b.x + (double)b.y * b.y + (double)b.z * b.z;
    return sqrt(s) + (double)b.w <= (double)R * (1.0 - 1.0 / 4096.0);
}

// Input checks, one thread per clump (400k clumps, 1M sub-spheres: 107 us with
// every length in binary64, 15 us now).
__global__ void __launch_bounds__(kThreads)
k_clump_check(DevCounters *cnt, int n, const float4 *__restrict__ pos,
              const float4 *__restrict__ quat, const int *__restrict__ off,
              const float4 *__restrict__ sub)
{
    if (cnt->err) return;
    unsigned b = 0;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads) {
        const float4 x = pos[i];
        const int a0 = off[i], a1 = off[i + 1];
        if (!unit(quat[i])) b |= CL_BAD_QUAT;
        if (a0 < 0 || !(a1 > a0) || a1 - a0 > kMaxSub) {
            b |= CL_BAD_OFFSETS;
            continue;
        }
        if (!(x.w > 0.0f) || !isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z))
            b |= CL_BAD_VALUE;
        for (int a = a0; a < a1; a += 4) {   // four loads in flight
            float4 s[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = sub[min(a + u, a1 - 1)];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (a + u >= a1) continue;
                if (!(s[u].w > 0.0f) || !isfinite(s[u].x) || !isfinite(s[u].y) || !isfinite(s[u].z))
                    b |= CL_BAD_VALUE;
                else if (!inside(s[u], x.w)) b |= CL_BAD_BOUND;
            }
        }
    }
    if (b) atomicOr(&cnt->clump_bad, b);
}

struct ClumpOut {
    int *ci, *ca, *cj, *cb;
    float *delta;
    long long cap;
};

struct ClumpHit {
    int i, a, j, b;
    float dl;
};

// Whether the bounding spheres of two clumps may overlap, with a margin far
// above the rounding of the sub-spheres' world positions (a few units in the
// last place of the coordinates).
__device__ __forceinline__ bool bounds_touch(float4 p, float4 q)
{
    const float dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
    const float m = fmaxf(fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z)),
                          fmaxf(fmaxf(fabsf(q.x), fabsf(q.y)), fabsf(q.z)));
    const float c = (p.w + q.w) * 1.01f + m * 4e-6f;
    return !(dx * dx + dy * dy + dz * dz > c * c);
}

// Two steps, both with all lanes busy: each lane walks the row of a clump i,
// four partners j > i at a time, and keeps the pairs whose bounding spheres
// touch (a third of a list that also holds the skins) in the warp's queue;
// whenever 32 pairs are queued, each lane takes one and tests their
// sub-spheres.  Contacts gather in shared memory and leave with one atomic for
// up to kHits.  One thread to a clump with its pairs one after another took
// 415 us for 400k clumps (2.9M pairs, 78k contacts), 109 us this way (64 registers;
// 143 us with the 106 it would take).
constexpr int kQueue = 32 + 128, kHits = 64, kFew = 4;

__global__ void __launch_bounds__(kThreads, 4)
k_clump_contacts(RowsView rv, const float4 *__restrict__ pos, const float4 *__restrict__ quat,
                 const int *__restrict__ off, const float4 *__restrict__ sub, ClumpOut out)
{
    if (rv.cnt->err || rv.cnt->clump_bad) return;
    __shared__ int2 queue[kThreads / 32][kQueue];
    __shared__ ClumpHit hits[kThreads / 32][kHits];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i == 0) atomicAdd(rv.kernels, 1ULL);
    int nq = 0, nh = 0;   // pairs queued, contacts gathered (warp-uniform)
    auto put_out = [&]() {
        __syncwarp();
        unsigned long long k0 = 0;
        if (lane == 0) k0 = atomicAdd(&rv.cnt->clump_total, (unsigned long long)nh);
        k0 = __shfl_sync(FULL, k0, 0);
        for (int t = lane; t < nh; t += 32) {
            const unsigned long long k = k0 + t;
            if (k < (unsigned long long)out.cap) {
                const ClumpHit h = hits[warp][t];
                out.ci[k] = h.i;
                out.ca[k] = h.a;
                out.cj[k] = h.j;
                out.cb[k] = h.b;
                out.delta[k] = h.dl;
            }
        }
        nh = 0;
        __syncwarp();
    };
    // up to 32 queued pairs, one to a lane
    auto resolve = [&]() {
        __syncwarp();
        const int m = min(nq, 32);
        nq -= m;
        int2 p = make_int2(0, 0);
        int i0 = 0, ki = 0, j0 = 0, kj = 0;
        float4 xi = make_float4(0.f, 0.f, 0.f, 0.f), xj = xi;
        float Ri[9], Rj[9];
        if (lane < m) {
            p = queue[warp][nq + lane];
            i0 = off[p.x];
            ki = off[p.x + 1] - i0;
            j0 = off[p.y];
            kj = off[p.y + 1] - j0;
            xi = pos[p.x];
            xj = pos[p.y];
            rotmat(quat[p.x], Ri);
            rotmat(quat[p.y], Rj);
        }
        float4 wb[kFew];   // the partner's first sub-spheres, kept in registers
#pragma unroll
        for (int b = 0; b < kFew; ++b)
            wb[b] = b < kj ? world(xj, Rj, sub[j0 + b]) : make_float4(0.f, 0.f, 0.f, 0.f);
        auto test = [&](bool on, int a, int b, float4 wa, float4 w) {
            const float dl = overlap_rn(wa, w);
            const bool hit = on && dl > 0.0f;
            const unsigned mk = __ballot_sync(FULL, hit);
            if (!mk) return;
            if (nh + __popc(mk) > kHits) put_out();
            if (hit) hits[warp][nh + __popc(mk & lanemask_lt())] = ClumpHit{p.x, a, p.y, b, dl};
            nh += __popc(mk);
        };
        for (int a = 0; __any_sync(FULL, a < ki); ++a) {
            const bool on = a < ki;
            const float4 wa = on ? world(xi, Ri, sub[i0 + a]) : xi;
#pragma unroll
            for (int b = 0; b < kFew; ++b)
                if (__any_sync(FULL, on && b < kj)) test(on && b < kj, a, b, wa, wb[b]);
            for (int b = kFew; __any_sync(FULL, on && b < kj); ++b) {
                const bool both = on && b < kj;
                test(both, a, b, wa, both ? world(xj, Rj, sub[j0 + b]) : xj);
            }
        }
        __syncwarp();
    };
    int e = 0, len = 0;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < rv.n) {
        xi = pos[i];
        e = rv.row_off[i];
        len = min(rv.row_len[i], rv.row_cap[i]);
    }
    for (int t = 0; __any_sync(FULL, t < len); t += 4) {
        int4 j4 = make_int4(-1, -1, -1, -1);   // -1: a removed pair's slot
        if (t < len) j4 = *reinterpret_cast<const int4 *>(rv.col + e + t);
        const int j[4] = {j4.x, j4.y, j4.z, j4.w};
        float4 xj[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) xj[u] = j[u] > i ? pos[j[u]] : xi;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const bool keep = j[u] > i && bounds_touch(xi, xj[u]);   // j < i: from j's row
            const unsigned mk = __ballot_sync(FULL, keep);
            if (keep) queue[warp][nq + __popc(mk & lanemask_lt())] = make_int2(i, j[u]);
            nq += __popc(mk);
        }
        while (nq >= 32) resolve();
    }
    while (nq > 0) resolve();
    if (nh) put_out();
}

int from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return LVB_OK;
    if (e == cudaErrorMemoryAllocation) return LVB_ENOMEM;
    return LVB_EDEVICE;
}

}  // namespace

extern "C" int lvb_clump_contacts(lvb_ctx *ctx, const float *pos_r, const float *quat,
                                  const int32_t *sub_off, const float *sub, int32_t *ci,
                                  int32_t *ca, int32_t *cj, int32_t *cb, float *delta,
                                  int64_t cap, int64_t *n_contacts)
{
    if (!ctx || !pos_r || !quat || !sub_off || !sub || !n_contacts || cap < 0 ||
        (cap > 0 && (!ci || !ca || !cj || !cb || !delta)))
        return LVB_EINVAL;
    if (((uintptr_t)pos_r & 15u) || ((uintptr_t)quat & 15u) || ((uintptr_t)sub & 15u))
        return LVB_EINVAL;
    *n_contacts = 0;
    const RowsView rv = rows_view(ctx);
    const cudaStream_t st = step_stream(ctx);
    const int n = rv.n;
    // outputs in device memory are written by the kernel in place; any
    // output in host memory sends all five through device temporaries
    bool direct = true;
    if (cap > 0) {
        const void *outs[5] = {ci, ca, cj, cb, delta};
        for (const void *p : outs) direct = direct && on_device(p);
    }
    const long long cp = std::max<long long>(cap, 1);
    ClumpOut o{ci, ca, cj, cb, delta, cap};
    auto done = [&](int code) {
        if (!direct) {
            cudaStreamSynchronize(st);
            cudaFree(o.ci);
            cudaFree(o.ca);
            cudaFree(o.cj);
            cudaFree(o.cb);
            cudaFree(o.delta);
        }
        return code;
    };
    cudaGetLastError();
    cudaError_t e = cudaSuccess;
    if (!direct) {
        o = ClumpOut{nullptr, nullptr, nullptr, nullptr, nullptr, cap};
        int **ints[4] = {&o.ci, &o.ca, &o.cj, &o.cb};
        for (int **q : ints)
            if (e == cudaSuccess) e = cudaMalloc((void **)q, sizeof(int) * cp);
        if (e == cudaSuccess) e = cudaMalloc((void **)&o.delta, sizeof(float) * cp);
    }
    // both kernels stand down on a context with a device error (the list must
    // be valid) and the second one on a bad input: one wait for everything
    if (e == cudaSuccess)
        e = cudaMemsetAsync(&rv.cnt->clump_total, 0, sizeof(rv.cnt->clump_total), st);
    if (e == cudaSuccess) e = cudaMemsetAsync(&rv.cnt->clump_bad, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return done(from_cuda(e));
    const int grid = (n + kThreads - 1) / kThreads;
    k_clump_check<<<grid, kThreads, 0, st>>>(rv.cnt, n, (const float4 *)pos_r,
                                             (const float4 *)quat, sub_off, (const float4 *)sub);
    k_clump_contacts<<<grid, kThreads, 0, st>>>(rv, (const float4 *)pos_r, (const float4 *)quat,
                                                sub_off, (const float4 *)sub, o);
    e = cudaGetLastError();
    if (e != cudaSuccess) return done(from_cuda(e));
    const DevCounters *h = nullptr;
    const int rc = sync_counters_of(ctx, &h);
    if (rc) return done(rc);
    if (h->clump_bad) return done(LVB_EINVAL);
    const unsigned long long total = h->clump_total;
    const long long m = std::min<long long>((long long)total, cap);
    if (!direct && m > 0) {
        int32_t *outs[4] = {ci, ca, cj, cb};
        int *srcs[4] = {o.ci, o.ca, o.cj, o.cb};
        for (int k = 0; k < 4 && e == cudaSuccess; ++k)
            e = cudaMemcpyAsync(outs[k], srcs[k], sizeof(int) * m, cudaMemcpyDefault, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(delta, o.delta, sizeof(float) * m, cudaMemcpyDefault, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return done(from_cuda(e));
    }
    *n_contacts = (int64_t)total;
    return done((long long)total > cap ? LVB_ECAPACITY : LVB_OK);
}
