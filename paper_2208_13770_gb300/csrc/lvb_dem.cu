// lvb_dem.cu -- DEM driver on the local Verlet buffer list (include/lvb_dem.h).
//
// Per step: position half-step (x', v*), the broad-phase step at x'
// (displacement check and partial rebuild), forces (narrow phase on the
// list rows, linear spring-dashpot, walls, a', v').  dem_advance runs up to
// DEM_GRAPH_STEPS steps as one cooperative launch (k_advance, or k_advance_apart
// where the particles have many contacts); dem_phase runs
// the three parts as separate launches (k_integrate, lvb_step, k_forces), with
// identical results.  Forces are accumulated per row of the
// symmetric list, so each pair is evaluated once from each side and no
// atomics are needed; both evaluations give exactly opposite forces.
//
// The overlap delta = r_i + r_j - |x_i - x_j| is a small difference of large
// numbers: at 0.3 m coordinates a binary32 position carries ~3e-8 m of
// rounding while a resting overlap under k_n = 1e4 N/m is ~1e-8 m.  So the
// distance is evaluated exactly-rounded-ish in compensated binary32
// (error-free TwoSum / TwoProduct transformations, Knuth and Dekker), which
// brings its error to ~1e-16 m at the cost of ~30 FP32 operations per
// contact -- far cheaper on this part than binary64.
#include "lvb_step.cuh"
#include "lvb_dem.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

using namespace lvb;

namespace {

constexpr int kThreads = 256;
constexpr int kNumSMs = 152;

struct DemDev {
    int n;
    float dt, half_dt, half_dt2;
    float kn, two_zeta, g[3];
    int wall_kind, clamp_tensile, contacts_on;
    float drum_cx, drum_cz, drum_R;
    float4 *pos, *vel, *acc, *vstar;   // vel.w = vstar.w = 1 / m (the integrator
                                       // reads it with v, not from vstar)
    // friction (mu > 0): rotation and the tangential law; omega.w = 1 / I
    float mu, kt, gt_ratio;
    float4 *omega, *alpha, *wstar;     // null without friction
    RowsView rows;
    int trace;                         // per-kernel trace (copied at launch)
};

// The two buffers of x, v, a (and, with friction, w, al) of k_advance, whose
// steps read their partners' state in one and write their own in the
// other; the first of each is the driver's own array, the second are parts of one
// allocation (b.x[1]): second_buffers.
struct DemBuffers {
    float4 *x[2], *v[2], *a[2], *w[2], *al[2];
};

__device__ __forceinline__ void dtr_enter(const DemDev &d, int slot)
{
    if (d.trace && threadIdx.x == 0) atomicMin(&d.rows.cnt->tr_start[slot], global_ns());
}

__device__ __forceinline__ void dtr_exit(const DemDev &d, int slot)
{
    if (d.trace && (threadIdx.x & 31) == 0) atomicMax(&d.rows.cnt->tr_end[slot], global_ns());
}

// exact a - b = s + e (TwoSum on a and -b)
__device__ __forceinline__ void two_diff(float a, float b, float &s, float &e)
{
    s = __fsub_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
}

// exact a + b = s + e
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// |h + l| for a 3-vector given as high + low parts: returns s0 (rounded
// sqrt of the leading sum) and corr with |h + l| = s0 + corr to ~2^-46.
__device__ __forceinline__ void norm_dd(const float h[3], const float l[3], float &s0, float &corr)
{
    float p0 = __fmul_rn(h[0], h[0]), p1 = __fmul_rn(h[1], h[1]), p2 = __fmul_rn(h[2], h[2]);
    float e0 = fmaf(h[0], h[0], -p0), e1 = fmaf(h[1], h[1], -p1), e2 = fmaf(h[2], h[2], -p2);
    float s, t, u, w;
    two_sum(p0, p1, s, t);
    two_sum(s, p2, u, w);
    float lo = t + w + (e0 + e1 + e2) +
               2.0f * (h[0] * l[0] + h[1] * l[1] + h[2] * l[2]);
    s0 = __fsqrt_rn(u);
    const float rem = fmaf(-s0, s0, u) + lo;     // fma remainder is exact
    corr = s0 > 0.0f ? rem / (2.0f * s0) : 0.0f;
}

__device__ __forceinline__ float lsd(const DemDev &d, float dl, float vn, float meff)
{
    const float gam = d.two_zeta * sqrtf(meff * d.kn);
    float f = d.kn * dl - gam * vn;
    if (d.clamp_tensile && f < 0.0f) f = 0.0f;
    return f;
}

// The old state is read with streaming loads (evict first), so that the L2
// keeps the new positions this kernel writes for the broad phase that
// follows.
__global__ void __launch_bounds__(kThreads)
k_integrate(DemDev d)
{
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i == 0) atomicAdd(d.rows.kernels, 1ULL);
    dtr_enter(d, TR_INTEGRATE);
    if (i < d.n) {
        float4 x = __ldcs(d.pos + i), v = __ldcs(d.vel + i), vs;
        half_step(x, v, __ldcs(d.acc + i), vs, d.dt, d.half_dt2);
        if (d.wall_kind == DEM_WALL_SPECULAR) {   // the scene's geometry only here
            reflect(x, v, vs, d.rows.sg[d.rows.nscenes == 1 ? 0 : d.rows.scene_of[i]]);
            d.vel[i] = v;
        }
        d.pos[i] = x;
        d.vstar[i] = vs;
        if (d.omega) d.wstar[i] = star_of(d.omega[i], d.alpha[i], d.dt);   // w*.w keeps 1/I
    }
    dtr_exit(d, TR_INTEGRATE);
}

// Wall planes normal to one axis: x in [lo, hi], velocity component v.
__device__ __forceinline__ float plane_force(const DemDev &d, float x, float v, float r, float lo,
                                             float hi, float im)
{
    // a gap more than 1e-4 wider than the radius is none (the compensated
    // difference is within 2^-24 of the plain one), and most particles
    // have six of these
    const float far = r * 1.0001f;
    float F = 0.0f, hh, ll;
    if (!(__fsub_rn(x, lo) > far)) {
        two_diff(x, lo, hh, ll);                       // x - lo
        const float dlo = __fsub_rn(r, hh) - ll;
        if (dlo > 0.0f) F += lsd(d, dlo, v, 1.0f / im);
    }
    if (!(__fsub_rn(hi, x) > far)) {
        two_diff(hi, x, hh, ll);                       // hi - x
        const float dhi = __fsub_rn(r, hh) - ll;
        if (dhi > 0.0f) F -= lsd(d, dhi, -v, 1.0f / im);
    }
    return F;
}

// v* (or w*) of a partner: as the half-step stored it, or worked out again
// from the state before the half-step, which a kernel that has already
// written newer v and a elsewhere still holds (the same roundings).
struct StoredStar {
    const float4 *vs;
    __device__ __forceinline__ float4 operator()(int j) const { return vs[j]; }
};

struct DerivedStar {
    const float4 *v, *a;
    float dt;
    __device__ __forceinline__ float4 operator()(int j) const { return star_of(v[j], a[j], dt); }
};

// Whether two particles may overlap: the plain distance against the radii
// with a margin far above its rounding.
__device__ __forceinline__ bool may_touch(float4 xi, float4 xj)
{
    const float hx = __fsub_rn(xi.x, xj.x), hy = __fsub_rn(xi.y, xj.y), hz = __fsub_rn(xi.z, xj.z);
    const float Rr = xi.w + xj.w;
    return !(hx * hx + hy * hy + hz * hz > Rr * Rr * 1.0001f);
}

// One contact of the narrow phase (Eq. delta) and its force: particle i at
// xi with v* and 1/m in vi, against partner j of its row at xj.  Returns false
// when the two do not overlap (delta <= 0); else the overlap dl (compensated
// binary32), the unit normal n (from j to i), the normal force f on i
// along n (linear spring-dashpot, damping on the normal component of
// v*_i - v*_j), the partner's v* and the pair's effective mass.
template <class Star>
__device__ __forceinline__ bool contact_pair(const DemDev &d, const Star &star, float4 xi,
                                             float4 vi, int j, float4 xj, float &dl, float n[3],
                                             float &f, float4 &vj, float &meff)
{
    if (!may_touch(xi, xj)) return false;   // before the compensated distance
    vj = star(j);   // loaded under the arithmetic: what may touch mostly does
    float h[3], l[3];
    two_diff(xi.x, xj.x, h[0], l[0]);
    two_diff(xi.y, xj.y, h[1], l[1]);
    two_diff(xi.z, xj.z, h[2], l[2]);
    float s0, corr;
    norm_dd(h, l, s0, corr);
    float Rh, Rl;
    two_sum(xi.w, xj.w, Rh, Rl);
    dl = __fsub_rn(Rh, s0) + (Rl - corr);
    if (!(dl > 0.0f) || !(s0 > 0.0f)) return false;
    const float inv = 1.0f / (s0 + corr);
    n[0] = (h[0] + l[0]) * inv;
    n[1] = (h[1] + l[1]) * inv;
    n[2] = (h[2] + l[2]) * inv;
    const float vn = (vi.x - vj.x) * n[0] + (vi.y - vj.y) * n[1] + (vi.z - vj.z) * n[2];
    meff = 1.0f / (vi.w + vj.w);
    f = lsd(d, dl, vn, meff);
    return true;
}

__device__ __forceinline__ float dot_rn(float ax, float ay, float az, const float n[3])
{
    return __fadd_rn(__fadd_rn(__fmul_rn(ax, n[0]), __fmul_rn(ay, n[1])), __fmul_rn(az, n[2]));
}

// The tangential law of one contact (friction), from particle i's side:
// updates the spring xi kept in h (row i's history record of partner j)
// and returns the tangential force on i.  Every operation is rounded
// explicitly (no contraction), in an order that is exactly sign-symmetric
// under exchanging i and j (n -> -n), so that j's record stays exactly -h.
__device__ __forceinline__ float3 tangential(const DemDev &d, float ri, float4 vi, float4 wi,
                                             float rj, float4 vj, float4 wj, const float n[3],
                                             float fn, float meff, float4 &h)
{
    // s = r_i w_i + r_j w_j, c = s x n: the contact point's rotational velocity
    const float sx = __fadd_rn(__fmul_rn(ri, wi.x), __fmul_rn(rj, wj.x));
    const float sy = __fadd_rn(__fmul_rn(ri, wi.y), __fmul_rn(rj, wj.y));
    const float sz = __fadd_rn(__fmul_rn(ri, wi.z), __fmul_rn(rj, wj.z));
    const float cx = __fsub_rn(__fmul_rn(sy, n[2]), __fmul_rn(sz, n[1]));
    const float cy = __fsub_rn(__fmul_rn(sz, n[0]), __fmul_rn(sx, n[2]));
    const float cz = __fsub_rn(__fmul_rn(sx, n[1]), __fmul_rn(sy, n[0]));
    const float ux = __fsub_rn(__fsub_rn(vi.x, vj.x), cx);
    const float uy = __fsub_rn(__fsub_rn(vi.y, vj.y), cy);
    const float uz = __fsub_rn(__fsub_rn(vi.z, vj.z), cz);
    const float un = dot_rn(ux, uy, uz, n);
    const float tx = __fsub_rn(ux, __fmul_rn(un, n[0]));
    const float ty = __fsub_rn(uy, __fmul_rn(un, n[1]));
    const float tz = __fsub_rn(uz, __fmul_rn(un, n[2]));
    // the spring kept in the tangent plane, then stretched by v_t dt
    const float hn = dot_rn(h.x, h.y, h.z, n);
    float hx = __fadd_rn(__fsub_rn(h.x, __fmul_rn(hn, n[0])), __fmul_rn(tx, d.dt));
    float hy = __fadd_rn(__fsub_rn(h.y, __fmul_rn(hn, n[1])), __fmul_rn(ty, d.dt));
    float hz = __fadd_rn(__fsub_rn(h.z, __fmul_rn(hn, n[2])), __fmul_rn(tz, d.dt));
    const float gt = __fmul_rn(d.gt_ratio, __fmul_rn(d.two_zeta, __fsqrt_rn(__fmul_rn(meff, d.kn))));
    float Fx = -__fadd_rn(__fmul_rn(d.kt, hx), __fmul_rn(gt, tx));
    float Fy = -__fadd_rn(__fmul_rn(d.kt, hy), __fmul_rn(gt, ty));
    float Fz = -__fadd_rn(__fmul_rn(d.kt, hz), __fmul_rn(gt, tz));
    const float Fm = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(Fx, Fx), __fmul_rn(Fy, Fy)),
                                          __fmul_rn(Fz, Fz)));
    const float lim = __fmul_rn(d.mu, fmaxf(fn, 0.0f));
    if (Fm > lim) {   // sliding: the force at the Coulomb limit, the spring to match it
        const float sc = __fdiv_rn(lim, Fm);
        Fx = __fmul_rn(Fx, sc);
        Fy = __fmul_rn(Fy, sc);
        Fz = __fmul_rn(Fz, sc);
        hx = -__fdiv_rn(__fadd_rn(Fx, __fmul_rn(gt, tx)), d.kt);
        hy = -__fdiv_rn(__fadd_rn(Fy, __fmul_rn(gt, ty)), d.kt);
        hz = -__fdiv_rn(__fadd_rn(Fz, __fmul_rn(gt, tz)), d.kt);
    }
    h = make_float4(hx, hy, hz, 0.0f);
    return make_float3(Fx, Fy, Fz);
}

// Adds the contact of row entry e (partner j at xj), if it is one, to the force
// on i in F and, with friction, to the torque in T.
template <bool kFric, class Star>
__device__ __forceinline__ bool add_contact(const DemDev &d, const Star &star, const Star &spin,
                                            float4 xi, float4 vi, int i, int e, int j, float4 xj,
                                            float F[3], float T[3])
{
    float4 vj;
    float dl, n[3], f, meff;
    if (!contact_pair(d, star, xi, vi, j, xj, dl, n, f, vj, meff)) return false;
    F[0] += f * n[0];
    F[1] += f * n[1];
    F[2] += f * n[2];
    if (kFric) {
        float4 h = d.rows.hist[e];
        const float3 Ft = tangential(d, xi.w, vi, spin(i), xj.w, vj, spin(j), n, f, meff, h);
        d.rows.hist[e] = h;
        F[0] += Ft.x;
        F[1] += Ft.y;
        F[2] += Ft.z;
        // torque -r_i n x F_t
        T[0] -= xi.w * (n[1] * Ft.z - n[2] * Ft.y);
        T[1] -= xi.w * (n[2] * Ft.x - n[0] * Ft.z);
        T[2] -= xi.w * (n[0] * Ft.y - n[1] * Ft.x);
    }
    return true;
}

// The contacts of row i (off, len; its partners at X) in row order.  The row
// is read four entries at a time (rows start on 16 bytes) and the four
// partners' positions together, so that a row of up to four costs two memory
// latencies; only the few that may touch are taken up again, one after
// another (their positions then come from the L1).  kMany: entry by entry, with
// the next partner's position in flight.  Where many touch, taking those up again
// saves no turns, and what bounds the loop is the gathers: one of 32 partners in
// no order is some 30 passes through the L1 (1M packed spheres, 3 contacts each,
// a launch of one step: 103 -> 87 us; 1M settling ones, next to none: 54 -> 59 us).
// With friction, an entry out of contact keeps no spring.  Most had none
// already, so the records are not written over and over (16 bytes for each of
// the four entries in six of a drum's row): live[i] has a bit for each of the
// row's first 32 entries whose record may be other than zero, and only those
// are cleared (1M drum, a pass over the particles: 111 -> 80 us).
template <bool kFric, bool kMany, class Star>
__device__ __forceinline__ void row_forces(const DemDev &d, const float4 *X, const Star &star,
                                           const Star &spin, float4 xi, float4 vi, int i, int off,
                                           int len, float F[3], float T[3])
{
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const unsigned live0 = kFric && len > 0 ? d.rows.live[i] : 0u;
    unsigned live = live0;
    for (int e0 = 0; e0 < len; e0 += 4) {
        const int4 j4 = *reinterpret_cast<const int4 *>(d.rows.col + off + e0);
        unsigned in = 0;   // entries in contact
        if (kMany) {
            float4 xj = j4.x >= 0 ? X[j4.x] : zero;
#pragma unroll 1
            for (int u = 0; u < 4; ++u) {
                const int j = u < 2 ? (u == 0 ? j4.x : j4.y) : (u == 2 ? j4.z : j4.w);
                const int after = u < 2 ? (u == 0 ? j4.y : j4.z) : (u == 2 ? j4.w : -1);
                const float4 xn = after >= 0 ? X[after] : zero;
                if (j >= 0 &&
                    add_contact<kFric>(d, star, spin, xi, vi, i, off + e0 + u, j, xj, F, T))
                    in |= 1u << u;
                xj = xn;
            }
        } else {
            float4 xj[4];
            xj[0] = j4.x >= 0 ? X[j4.x] : zero;
            xj[1] = j4.y >= 0 ? X[j4.y] : zero;
            xj[2] = j4.z >= 0 ? X[j4.z] : zero;
            xj[3] = j4.w >= 0 ? X[j4.w] : zero;
            unsigned m = 0;
            if (j4.x >= 0 && may_touch(xi, xj[0])) m |= 1u;
            if (j4.y >= 0 && may_touch(xi, xj[1])) m |= 2u;
            if (j4.z >= 0 && may_touch(xi, xj[2])) m |= 4u;
            if (j4.w >= 0 && may_touch(xi, xj[3])) m |= 8u;
            while (m) {
                const int u = __ffs(m) - 1;
                m &= m - 1;
                const int j = u < 2 ? (u == 0 ? j4.x : j4.y) : (u == 2 ? j4.z : j4.w);
                if (add_contact<kFric>(d, star, spin, xi, vi, i, off + e0 + u, j, X[j], F, T))
                    in |= 1u << u;
            }
        }
        if (kFric) {
            const unsigned there = (j4.x >= 0 ? 1u : 0u) | (j4.y >= 0 ? 2u : 0u) |
                                   (j4.z >= 0 ? 4u : 0u) | (j4.w >= 0 ? 8u : 0u);
            unsigned clear = there & ~in;
            if (e0 < 32) {
                clear &= live >> e0;
                live = (live & ~(clear << e0)) | (in << e0);
            }
            for (; clear; clear &= clear - 1) d.rows.hist[off + e0 + __ffs(clear) - 1] = zero;
        }
    }
    if (kFric && live != live0) d.rows.live[i] = live;
}

// The walls' forces on particle i, added to F; im: 1/m.
__device__ __forceinline__ void wall_forces(const DemDev &d, float4 xi, float4 vi, int sc_i,
                                            float F[3])
{
    if (d.wall_kind != DEM_WALL_BOX && d.wall_kind != DEM_WALL_DRUM) return;
    const float r = xi.w, im = vi.w;
    const SceneGeom &g = d.rows.sg[sc_i];
    if (d.wall_kind == DEM_WALL_BOX) {
        F[0] += plane_force(d, xi.x, vi.x, r, g.lo[0], g.hi[0], im);
        F[2] += plane_force(d, xi.z, vi.z, r, g.lo[2], g.hi[2], im);
    }
    F[1] += plane_force(d, xi.y, vi.y, r, g.lo[1], g.hi[1], im);   // box side / drum caps
    if (d.wall_kind == DEM_WALL_DRUM) {
        // well inside the drum (by 1e-4 of its free radius, far above the
        // rounding of the plain distance): no wall
        const float px = __fsub_rn(xi.x, d.drum_cx), pz = __fsub_rn(xi.z, d.drum_cz);
        const float in = (d.drum_R - r) * 0.9999f;
        if (in > 0.0f && px * px + pz * pz < in * in) return;
        float h[3], l[3];
        two_diff(xi.x, d.drum_cx, h[0], l[0]);
        h[1] = 0.0f;
        l[1] = 0.0f;
        two_diff(xi.z, d.drum_cz, h[2], l[2]);
        float s0, corr;
        norm_dd(h, l, s0, corr);
        // delta = r + rho - R, rho = s0 + corr; (s0 - R) is exact near the wall
        const float t = __fsub_rn(s0, d.drum_R);
        const float dl = __fadd_rn(t, r) + corr;
        if (dl > 0.0f && s0 > 0.0f) {
            const float inv = 1.0f / s0;
            const float nx = -(h[0] + l[0]) * inv, nz = -(h[2] + l[2]) * inv;
            const float vn = vi.x * nx + vi.z * nz;
            const float f = lsd(d, dl, vn, 1.0f / im);
            F[0] += f * nx;
            F[2] += f * nz;
        }
    }
}

// a' = F / m + g and v' = v + (a + a') dt / 2 (v.w, 1/m, kept)
__device__ __forceinline__ float4 finish_velocity(const DemDev &d, const float F[3], float im,
                                                  float4 a, float4 &v)
{
    const float4 an = make_float4(F[0] * im + d.g[0], F[1] * im + d.g[1], F[2] * im + d.g[2],
                                  0.0f);
    v.x += (a.x + an.x) * d.half_dt;
    v.y += (a.y + an.y) * d.half_dt;
    v.z += (a.z + an.z) * d.half_dt;
    return an;
}

// al' = T / I, w' = w + (al + al') dt / 2 (w.w, 1/I, kept)
__device__ __forceinline__ float4 finish_spin(const DemDev &d, const float T[3], float4 al,
                                              float4 &w)
{
    const float4 aln = make_float4(T[0] * w.w, T[1] * w.w, T[2] * w.w, 0.0f);
    w.x += (al.x + aln.x) * d.half_dt;
    w.y += (al.y + aln.y) * d.half_dt;
    w.z += (al.z + aln.z) * d.half_dt;
    return aln;
}

// Whether the walls need the scene of each particle, and the scene of i if so.
__device__ __forceinline__ bool wall_scenes(const DemDev &d)
{
    return d.wall_kind != DEM_WALL_NONE && d.rows.nscenes > 1;
}

__device__ __forceinline__ int wall_scene(const DemDev &d, int i)
{
    return wall_scenes(d) ? d.rows.scene_of[i] : 0;
}

// The forces phase of particle i from the stored x', v* (and w*); the state
// before the step's forces is v, a (w, al), the new one goes to d.vel, d.acc
// (d.omega, d.alpha).  rows: the rows may be read (contacts on, store not failed:
// after LVB_EOVERFLOW the row offsets no longer fit the store).  The row
// bounds and the scene are loaded with the particle's own state.
template <bool kFric, bool kMany>
__device__ __forceinline__ void forces_body(const DemDev &d, int i, const float4 *vin,
                                            const float4 *ain, const float4 *win,
                                            const float4 *alin)
{
    const float4 xi = d.pos[i];
    const float4 vi = d.vstar[i];
    const float4 a = ain[i];
    float4 v = vin[i];
    const int sc_i = wall_scene(d, i), off = d.rows.row_off[i];
    int len = min(d.rows.row_len[i], d.rows.row_cap[i]);
    if (!d.contacts_on || (d.rows.cnt->err & DERR_STORE)) len = 0;
    const StoredStar star{d.vstar}, spin{d.wstar};
    float F[3] = {0.f, 0.f, 0.f}, T[3] = {0.f, 0.f, 0.f};
    row_forces<kFric, kMany>(d, d.pos, star, spin, xi, vi, i, off, len, F, T);
    wall_forces(d, xi, vi, sc_i, F);
    d.acc[i] = finish_velocity(d, F, vi.w, a, v);
    d.vel[i] = v;
    if (kFric) {
        float4 w = win[i];
        d.alpha[i] = finish_spin(d, T, alin[i], w);
        d.omega[i] = w;
    }
}

// Forces as a separate kernel, one thread per particle.  Bound by the row
// walks' dependent loads: a row taken four entries at a time wants 48 registers
// (five blocks an SM; friction 64, four blocks), which beats the full
// occupancy of an entry-by-entry walk in 32 (6.2M batch 168 -> 160 us, 2M drum
// 82 -> 77 us, 1M drum with friction 199 -> 124 us).
template <bool kFric>
__global__ void __launch_bounds__(kThreads, kFric ? 4 : 5)
k_forces(DemDev d)
{
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i == 0) atomicAdd(d.rows.kernels, 1ULL);
    dtr_enter(d, TR_FORCES);
    if (i < d.n) forces_body<kFric, false>(d, i, d.vel, d.acc, d.omega, d.alpha);
    dtr_exit(d, TR_FORCES);
}

// One pass over the particles of k_advance.  kForces: the forces at (x, v*)
// of the step before, with v* worked out again from v and a, its a' and v',
// then the position half-step and the displacement check of this step;
// else the half-step and the check only (the first step of a launch).
// Reads the state in one of the two buffers of each array, bx for x, bv for
// v, a (w, al), and writes x to buffer ox and the others to bv ^ 1: partners'
// x, v, a are read all through the pass, so none of them may be written
// there (the half-step alone touches no partner and runs in place).
// Each warp takes chunks of 32 consecutive particles, warp w of block b the
// chunks w * grid + b, + all warps, ... (so that a last, partial round
// spreads over all SMs).  The chain of dependent loads is row bounds, row,
// partners' positions, at 32 warps an SM (64 registers a thread): the bounds are
// loaded a chunk ahead and the row's first sector is asked for from DRAM
// then (512 scenes, 6.2M particles: 202 -> 185 -> 174 us a pass).  A ring of
// asynchronous copies of x, v, a and the reference state in shared memory
// was slower (the L1 that it displaces holds the rows and partners: 186 us
// there, the 2M drum 82 -> 107 us), and so were L2 prefetches of them.
template <bool kFric, bool kForces>
__device__ __forceinline__ void advance_pass(const DevState &s, const DemDev &d,
                                             const DemBuffers &b, int bx, int ox, int bv,
                                             bool rows, bool keep_star, bool inc, int step,
                                             int *nF_acc)
{
    __shared__ int pend_id[kStepMaxThreads / 32][kPending];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Pending pd{pend_id[warp], 0};
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const bool scenes = wall_scenes(d), walk = kForces && rows;
    auto bounds = [&](int c, int &o, int &l) {
        const int i = c * 32 + lane;
        o = l = 0;
        if (walk && i < s.n) {
            o = s.row_off[i];
            l = s.row_len[i];   // at most the capacity between steps: a row that
                                // outgrew it was laid out anew
        }
    };
    int c = warp * gridDim.x + blockIdx.x, off, len;
    bounds(c, off, len);
    for (; c < s.nwords; c += nw) {
        int off1, len1;   // the next chunk's
        bounds(c + nw, off1, len1);
        const int cu[1] = {c * 32};
        const int i = cu[0] + lane;
        bool f[1] = {false};
        if (i < s.n) {
            float4 x = b.x[bx][i], v = b.v[bv][i], a = b.a[bv][i], w, al;
            const float4 q = __ldcs(s.ref + i);   // read once: evicted first
            const int sc = scenes ? d.rows.scene_of[i] : 0;
            if (kForces) {
                float F[3] = {0.f, 0.f, 0.f}, Tq[3] = {0.f, 0.f, 0.f};
                const float4 vi = star_of(v, a, d.dt);
                if (len > 0) {
                    const DerivedStar star{b.v[bv], b.a[bv], d.dt},
                        spin{b.w[bv], b.al[bv], d.dt};
                    row_forces<kFric, false>(d, b.x[bx], star, spin, x, vi, i, off, len, F, Tq);
                }
                wall_forces(d, x, vi, sc, F);
                a = finish_velocity(d, F, vi.w, a, v);
                __stcs(&b.a[bv ^ 1][i], a);   // read again a whole pass later
                if (kFric) {
                    w = b.w[bv][i];
                    al = finish_spin(d, Tq, b.al[bv][i], w);
                    b.w[bv ^ 1][i] = w;
                    b.al[bv ^ 1][i] = al;
                }
            } else {
                if (kFric) {
                    w = b.w[bv][i];
                    al = b.al[bv][i];
                }
            }
            float4 vs;
            half_step(x, v, a, vs, d.dt, d.half_dt2);
            const bool mirror = d.wall_kind == DEM_WALL_SPECULAR;
            if (mirror) reflect(x, v, vs, s.sg[sc]);
            b.x[ox][i] = x;
            if (kForces) __stcs(&b.v[bv ^ 1][i], v);
            else if (mirror) b.v[bv][i] = v;
            f[0] = violates(x, q);
            if (!(isfinite(x.x) && isfinite(x.y) && isfinite(x.z)))
                atomicOr(&s.cnt->err, DERR_NAN);
            // v* for whoever reads it: the updates of this step, or (the
            // launch's last step) the forces and the caller
            if (keep_star || f[0]) {
                d.vstar[i] = vs;
                if (kFric) d.wstar[i] = star_of(w, al, d.dt);
            }
        }
        flag_chunks<1>(s, cu, f, b.x[ox], d.vstar, nullptr, inc, step, nF_acc, pd);
        off = off1;
        len = len1;
        if (len > 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(s.col + off));
    }
    flush_pending_final(s, pd, b.x[ox], d.vstar, nullptr, inc, step, nF_acc);
}

// The rest of a step as a call of its own: what it keeps in registers does
// not displace the pass's.  To a call the kernel's parameter is memory like
// any other, cached in an L1 that every grid barrier empties, so the phases
// after the pass read the context's state from a copy in shared memory
// (settling 200k 24.6 -> 23.0 us a step).  Some threads fill it and all read
// it, from before the first grid barrier on (a warp without particles comes
// straight to it), so the block barrier that follows the filling publishes it.
static __shared__ DevState s_state;

__device__ __forceinline__ void copy_state(const DevState &s)
{
    static_assert(sizeof(DevState) % 4 == 0, "copied in words");
    for (int t = threadIdx.x; t < (int)(sizeof(DevState) / 4); t += blockDim.x)
        reinterpret_cast<unsigned *>(&s_state)[t] = reinterpret_cast<const unsigned *>(&s)[t];
    __syncthreads();
}

template <bool kPartial>
static __device__ __noinline__ bool rest_of_step(const lvb_mlp_weights *w_sh, const float4 *pos,
                                                 const float4 *vel, const float4 *acc, bool inc,
                                                 int step, int slot, unsigned long long t0)
{
    return finish_step<kPartial>(s_state, w_sh, pos, vel, acc, inc, step, slot, t0);
}

// `steps` whole DEM steps as one cooperative launch, all blocks resident.
// What bounds a step here is the traffic of the state and, for small runs,
// the launches and barriers; so one pass over the particles does the forces
// of a step and the half-step and check of the next (x, v, a and the
// reference state read once, x, v, a written once: 112 bytes a particle plus
// its row, where three phases move 204), and only a grid barrier lies
// between the steps (two when something was flagged).
// The state goes back and forth between two buffers and ends in d.pos, d.vel,
// d.acc: the half-step of the first step writes x to the buffer from which
// the steps - 1 passes that follow end there, the last forces write d.vel and
// d.acc.  Those read v* (and w*) as the last pass stored it, so they need no
// second buffer.
template <bool kFric, bool kPartial>
__global__ void __launch_bounds__(kStepMaxThreads, 1)
k_advance(const __grid_constant__ DevState s, const __grid_constant__ DemDev d,
          const __grid_constant__ DemBuffers b, int steps)
{
    DevCounters *c = s.cnt;
    const unsigned err0 = c->err;
    if (err0 & DERR_SYNC) return;   // a barrier failed earlier: the context is unusable
    const unsigned done = (unsigned)c->steps;
    int bx = 0, bv = 0;   // the buffers that hold the state
    __shared__ __align__(16) lvb_mlp_weights w_sh;
    const bool net = kPartial && s.skin_kind == LVB_SKIN_LEARNED;
    if (net) weights_copy_async(&w_sh, s.mlp);
    step_kernel_begin();
    copy_state(s);
    if (step_lead()) atomicAdd(&c->kernels, 1ULL);
    // v* of everyone at every step where the trigger may update anyone
    const bool star_always = !kPartial || s.early_beta < 1.0f;
    for (int k = 1; k <= steps; ++k) {
        const unsigned long long t0 = (s.trace && step_lead()) ? global_ns() : 0ULL;
        const unsigned err = k == 1 ? err0 : *(volatile unsigned *)&c->err;
        const bool store_ok = !(err & DERR_STORE);
        const bool inc = kPartial && store_ok;
        const bool star = star_always || k == steps;
        const int step = next_step(done + k - 1), slot = step_slot(step);
        grid_barrier_begin(slot);
        int *nF_acc = &c->nF_acc[slot];
        if (k == 1) {
            const int ox = ~steps & 1;
            advance_pass<kFric, false>(s, d, b, 0, ox, 0, false, star, inc, step, nF_acc);
            bx = ox;
            if (net) weights_copy_wait();
        } else {
            advance_pass<kFric, true>(s, d, b, bx, bx ^ 1, bv, store_ok && d.contacts_on, star,
                                      inc, step, nF_acc);
            bx ^= 1;
            bv ^= 1;
        }
        if (!rest_of_step<kPartial>(&w_sh, b.x[bx], d.vstar, b.a[bv], inc, step, slot, t0)) return;
    }
    flush_work(s);
    const unsigned long long t3 = (s.trace && step_lead()) ? global_ns() : 0ULL;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n; i += gridDim.x * blockDim.x)
        forces_body<kFric, false>(d, i, b.v[bv], b.a[bv], b.w[bv], b.al[bv]);
    if (s.trace) {
        if (!grid_barrier(s)) return;
        if (step_lead()) trace_add(c, TR_TAIL, t3, global_ns());
    }
}

// The same steps with the forces apart, for particles with many contacts and for
// specular walls with contacts: the half-step and check, the rest of the step, the
// forces, a grid barrier; the state in place, in d.pos, d.vel, d.acc.  A joined
// pass gathers v and a of a partner in contact (w and al), these forces the stored
// v* (w*), and where many partners lie far away those gathers bound a dense bed.
// 1M packed spheres in no order with 0.9, 1.5, 2.2 and 3.7 contacts each, us a step:
// joined 77, 86, 93 and 100, apart 78, 79, 77 and 78 (with friction, 0.8, 1.2, 2.0 and
// 4.1 contacts: 163, 194, 227, 283 and 181, 194, 194, 208).  In the order of their
// places: 61, 67, 71, 74 and 75, 76, 74, 74 (with friction 118, 136, 152, 166 and 159,
// 166, 165, 169; with 5.9, 171 and 165); 3,000 in no order with 1.6 contacts 13.0 and
// 13.4.
template <bool kFric, bool kPartial>
__global__ void __launch_bounds__(kStepMaxThreads, 1)
k_advance_apart(const __grid_constant__ DevState s, const __grid_constant__ DemDev d,
                const __grid_constant__ DemBuffers b, int steps)
{
    DevCounters *c = s.cnt;
    const unsigned err0 = c->err;
    if (err0 & DERR_SYNC) return;
    const unsigned done = (unsigned)c->steps;
    __shared__ __align__(16) lvb_mlp_weights w_sh;
    if (kPartial && s.skin_kind == LVB_SKIN_LEARNED) weights_copy_async(&w_sh, s.mlp);
    step_kernel_begin();
    copy_state(s);
    if (step_lead()) atomicAdd(&c->kernels, 1ULL);
    for (int k = 1; k <= steps; ++k) {
        const unsigned long long t0 = (s.trace && step_lead()) ? global_ns() : 0ULL;
        const unsigned err = k == 1 ? err0 : *(volatile unsigned *)&c->err;
        const bool inc = kPartial && !(err & DERR_STORE);
        const int step = next_step(done + k - 1), slot = step_slot(step);
        grid_barrier_begin(slot);
        advance_pass<kFric, false>(s, d, b, 0, 0, 0, false, true, inc, step, &c->nF_acc[slot]);
        weights_copy_wait();
        if (!rest_of_step<kPartial>(&w_sh, d.pos, d.vstar, d.acc, inc, step, slot, t0)) return;
        const unsigned long long t3 = (s.trace && step_lead()) ? global_ns() : 0ULL;
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d.n; i += gridDim.x * blockDim.x)
            forces_body<kFric, true>(d, i, d.vel, d.acc, d.omega, d.alpha);
        if (k < steps || s.trace) {   // the next half-step moves what others still read
            if (!grid_barrier(s)) return;
            if (s.trace && step_lead()) trace_add(c, TR_TAIL, t3, global_ns());
        }
    }
    flush_work(s);
}

// How much the contacts of a sample of the particles, 32 to a warp from places spread
// over the arrays, speak for the second form: a contact with a partner more than
// kFar places away (whose sector no other particle of the block has asked for) two, with
// friction any other contact one.  The sum in the upper half of *out (host
// memory), the particles in the lower.  One block.
constexpr int kFar = 16384;   // 256 KB of positions, an L1

__global__ void __launch_bounds__(1024)
k_sample(DemDev d, unsigned long long *out)
{
    __shared__ unsigned long long sum;
    if (threadIdx.x == 0) {
        sum = 0;
        atomicAdd(d.rows.kernels, 1ULL);
    }
    __syncthreads();
    const int warps = blockDim.x >> 5, chunks = (d.n + 31) / 32, q = threadIdx.x >> 5;
    const int i = (int)((long long)q * chunks / min(warps, chunks)) * 32 + (threadIdx.x & 31);
    if (q < chunks && i < d.n && !(d.rows.cnt->err & DERR_STORE)) {
        const float4 xi = d.pos[i];
        const int off = d.rows.row_off[i], len = min(d.rows.row_len[i], d.rows.row_cap[i]);
        unsigned long long n = 0;
        for (int e = 0; e < len; ++e) {
            const int j = d.rows.col[off + e];
            if (j >= 0 && may_touch(xi, d.pos[j]))
                n += abs(i - j) > kFar ? 2 : d.omega ? 1 : 0;
        }
        atomicAdd(&sum, (n << 32) + 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) *(volatile unsigned long long *)out = sum;
}

// The contacts of the current state, each pair once (i < j from row i),
// with the force on i and the overlap; positions in the output from one
// atomic counter, so in no particular order.
__global__ void __launch_bounds__(kThreads)
k_contact_list(DemDev d, unsigned long long *cnt, long long cap, int *ci, int *cj, float *f3,
               float *delta, float *xi3, int both)
{
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if (i == 0) atomicAdd(d.rows.kernels, 1ULL);
    if (i >= d.n || !d.contacts_on || (d.rows.cnt->err & DERR_STORE)) return;
    const float4 xi = d.pos[i];
    const float4 vi = d.vstar[i];
    const bool fric = d.omega != nullptr;
    const int off = d.rows.row_off[i];
    const int len = min(d.rows.row_len[i], d.rows.row_cap[i]);
    for (int e = 0; e < len; ++e) {
        const int j = d.rows.col[off + e];
        // a removed pair's slot, or (one side only) the pair from j's row
        if (j < 0 || (!both && j <= i)) continue;
        float dl, n[3], f, meff;
        float4 vj;
        const float4 xj = d.pos[j];
        if (!contact_pair(d, StoredStar{d.vstar}, xi, vi, j, xj, dl, n, f, vj, meff)) continue;
        float Ft[3] = {0.f, 0.f, 0.f}, h[3] = {0.f, 0.f, 0.f};
        if (fric) {
            // F_t = -k_t xi - gamma_t v_t from the spring as the step left it
            const float4 r = d.rows.hist[off + e];
            h[0] = r.x;
            h[1] = r.y;
            h[2] = r.z;
            const float4 wi = d.wstar[i], wj = d.wstar[j];
            const float ri = xi.w, rj = xj.w;
            const float sx = __fadd_rn(__fmul_rn(ri, wi.x), __fmul_rn(rj, wj.x));
            const float sy = __fadd_rn(__fmul_rn(ri, wi.y), __fmul_rn(rj, wj.y));
            const float sz = __fadd_rn(__fmul_rn(ri, wi.z), __fmul_rn(rj, wj.z));
            const float u[3] = {
                __fsub_rn(__fsub_rn(vi.x, vj.x), __fsub_rn(__fmul_rn(sy, n[2]), __fmul_rn(sz, n[1]))),
                __fsub_rn(__fsub_rn(vi.y, vj.y), __fsub_rn(__fmul_rn(sz, n[0]), __fmul_rn(sx, n[2]))),
                __fsub_rn(__fsub_rn(vi.z, vj.z), __fsub_rn(__fmul_rn(sx, n[1]), __fmul_rn(sy, n[0])))};
            const float un = dot_rn(u[0], u[1], u[2], n);
            const float gt =
                __fmul_rn(d.gt_ratio, __fmul_rn(d.two_zeta, __fsqrt_rn(__fmul_rn(meff, d.kn))));
            for (int c = 0; c < 3; ++c)
                Ft[c] = -__fadd_rn(__fmul_rn(d.kt, h[c]),
                                   __fmul_rn(gt, __fsub_rn(u[c], __fmul_rn(un, n[c]))));
        }
        const unsigned long long k = atomicAdd(cnt, 1ULL);
        if (k < (unsigned long long)cap) {
            ci[k] = i;
            cj[k] = j;
            f3[3 * k + 0] = f * n[0] + Ft[0];
            f3[3 * k + 1] = f * n[1] + Ft[1];
            f3[3 * k + 2] = f * n[2] + Ft[2];
            delta[k] = dl;
            if (xi3) {
                xi3[3 * k + 0] = h[0];
                xi3[3 * k + 1] = h[1];
                xi3[3 * k + 2] = h[2];
            }
        }
    }
}

__global__ void k_dem_setup(DemDev d, const float4 *__restrict__ pos, const float4 *__restrict__ vel,
                            float rho)
{
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < d.n; i += gridDim.x * kThreads) {
        const float4 p = pos[i];
        const float4 v = vel[i];
        const double r = p.w;
        const double m = (double)rho * (4.0 / 3.0) * 3.14159265358979323846 * r * r * r;
        d.pos[i] = p;
        const float im = (float)(1.0 / m);
        d.vel[i] = make_float4(v.x, v.y, v.z, im);
        d.vstar[i] = make_float4(v.x, v.y, v.z, im);
        d.acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (d.omega) {   // at rest, I = 2/5 m r^2
            const float iI = (float)(1.0 / (0.4 * m * r * r));
            d.omega[i] = make_float4(0.f, 0.f, 0.f, iI);
            d.wstar[i] = make_float4(0.f, 0.f, 0.f, iI);
            d.alpha[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// After the caller overwrote v: 1 / m back into v.w (from v*.w).
__global__ void k_restore_im(DemDev d)
{
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < d.n; i += gridDim.x * kThreads)
        d.vel[i].w = d.vstar[i].w;
}

// initial a0 = F(x0, v0)/m + g: the force kernel with a = 0 and dt = 0
// leaves v unchanged and writes a0.
}  // namespace

struct dem_ctx {
    DemDev d{};
    DemBuffers b{};
    dem_params prm{};
    lvb_ctx *bp = nullptr;
    cudaStream_t stream = nullptr;
    int advance_blocks[2] = {0, 0};   // launch shapes of k_advance and k_advance_apart,
    int advance_threads = 0;     // worked out for the broad phase's step_version
    int shape_of = -1;           // shape_of
    // the last sample of the contacts (k_sample; mapped host memory, null
    // without contacts) and the steps enqueued since it was asked for
    unsigned long long *sample = nullptr, *sample_d = nullptr;
    int64_t since = 0;
};

namespace {

int from_cuda(cudaError_t e)
{
    if (e == cudaSuccess) return LVB_OK;
    if (e == cudaErrorMemoryAllocation) return LVB_ENOMEM;
    return LVB_EDEVICE;
}

int grid_n(int n) { return (n + kThreads - 1) / kThreads; }

void dem_free(dem_ctx *c)
{
    if (c->bp) lvb_destroy(c->bp);
    float4 *ptrs[] = {c->d.pos, c->d.vel, c->d.acc, c->d.vstar, c->d.omega, c->d.alpha,
                      c->d.wstar, c->b.x[1]};
    for (float4 *p : ptrs)
        if (p) cudaFree(p);
    if (c->sample) cudaFreeHost(c->sample);
}

// The driver's copy of the row-store addresses follows the broad phase's
// (a grown store moves), and the trace switch follows its option.
void refresh(dem_ctx *c)
{
    c->d.rows = rows_view(c->bp);
    c->d.trace = *c->d.rows.trace;
}

int launch_phase(dem_ctx *c, int phase)
{
    refresh(c);
    if (phase == DEM_PHASE_INTEGRATE) {
        k_integrate<<<grid_n(c->d.n), kThreads, 0, c->stream>>>(c->d);
    } else if (phase == DEM_PHASE_BROAD) {
        int rc = lvb_step(c->bp, (const float *)c->d.pos, (const float *)c->d.vstar,
                          (const float *)c->d.acc);
        if (rc) return rc;
    } else if (phase == DEM_PHASE_FORCES) {
        if (c->d.omega) k_forces<true><<<grid_n(c->d.n), kThreads, 0, c->stream>>>(c->d);
        else k_forces<false><<<grid_n(c->d.n), kThreads, 0, c->stream>>>(c->d);
    } else {
        return LVB_EINVAL;
    }
    return from_cuda(cudaGetLastError());
}

auto advance_kernel(const dem_ctx *c, bool apart)
{
    const bool partial = step_state(c->bp).trigger == LVB_TRIGGER_PARTIAL;
    if (apart) {
        if (partial) return c->d.omega ? k_advance_apart<true, true> : k_advance_apart<false, true>;
        return c->d.omega ? k_advance_apart<true, false> : k_advance_apart<false, false>;
    }
    if (partial) return c->d.omega ? k_advance<true, true> : k_advance<false, true>;
    return c->d.omega ? k_advance<true, false> : k_advance<false, false>;
}

// Asks for a sample of the contacts.  The answer is there when
// the stream has come to it; until then the last one stands (both forms of the
// steps give the same results).
cudaError_t ask_sample(dem_ctx *c)
{
    if (!c->sample) return cudaSuccess;
    c->since = 0;
    k_sample<<<1, 1024, 0, c->stream>>>(c->d, c->sample_d);
    return cudaGetLastError();
}

constexpr int64_t kSampleEvery = 500;   // steps (the sample takes as long as one or two)

// Whether the particles have many contacts: one and a half far ones each, in the
// sample, or with friction three of any kind.
bool many_contacts(const dem_ctx *c)
{
    if (!c->sample) return false;
    const unsigned long long v = *(volatile unsigned long long *)c->sample;
    const unsigned sum = (unsigned)(v >> 32), seen = (unsigned)v;
    return seen > 0 && sum >= 3 * seen;
}

// Whether the steps keep their forces apart.  (Mirrored velocities cannot be worked
// out again from v and a, as a joined pass does for a contact's partner.)
bool keeps_apart(const dem_ctx *c)
{
    return (c->d.wall_kind == DEM_WALL_SPECULAR && c->d.contacts_on) || many_contacts(c);
}

// The second buffers of joined passes, 48 bytes a particle (80 with friction).
// dem_init allocates them where they are a small part of the memory (spare: only
// if they are at most an eighth of what is free), so that the first call need not;
// otherwise a launch that needs them does, also while a stream is being captured,
// and a program that never has one keeps the memory.  False: there is not enough
// (the form with the forces apart needs none).
bool second_buffers(dem_ctx *c, bool spare = false)
{
    if (c->b.x[1]) return true;
    const size_t each = ((size_t)c->d.n + 15) / 16 * 16;   // on 256 bytes
    const size_t bytes = sizeof(float4) * each * (c->d.omega ? 5 : 3);
    size_t room = 0, all = 0;
    if (spare && (cudaMemGetInfo(&room, &all) != cudaSuccess || bytes > room / 8)) return false;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    float4 *p = nullptr;
    const cudaError_t e = cudaMalloc((void **)&p, bytes);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) {
        cudaGetLastError();   // not this call's failure
        return false;
    }
    c->b.x[1] = p;
    c->b.v[1] = p + each;
    c->b.a[1] = p + 2 * each;
    if (c->d.omega) {
        c->b.w[1] = p + 3 * each;
        c->b.al[1] = p + 4 * each;
    }
    return true;
}

// Launch shapes: the broad phase's block size, as many blocks as are resident on
// the device at once, and no more than have work.
int advance_shape(dem_ctx *c)
{
    const int version = step_version(c->bp);
    if (c->shape_of == version) return LVB_OK;
    const int threads = step_threads(c->bp);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // a run of up to 2,048 particles stays on one block, whose barriers cost
    // next to nothing
    const int want = c->d.n <= 2 * threads ? 1 : (c->d.n + threads - 1) / threads;
    for (int apart = 0; apart < 2 && e == cudaSuccess; ++apart) {
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, (const void *)advance_kernel(c, apart), threads, 0);
        if (e == cudaSuccess && per_sm < 1) return LVB_EDEVICE;
        c->advance_blocks[apart] = std::min(want, per_sm * sms);
    }
    if (e != cudaSuccess) return from_cuda(e);
    c->advance_threads = threads;
    c->shape_of = version;
    return LVB_OK;
}

// `steps` whole steps as one cooperative launch.
int launch_advance(dem_ctx *c, int steps)
{
    int rc = grow_stores_if_asked(c->bp);
    if (rc) return rc;
    rc = advance_shape(c);
    if (rc) return rc;
    refresh(c);
    if (c->since >= kSampleEvery) {
        const cudaError_t e = ask_sample(c);
        if (e != cudaSuccess) return from_cuda(e);
    }
    c->since += steps;
    const bool apart = keeps_apart(c) || (steps > 1 && !second_buffers(c));
    const dim3 grid(c->advance_blocks[apart]), block(c->advance_threads);
    return from_cuda(launch_coop(advance_kernel(c, apart), grid, block, 0, c->stream,
                                 step_state(c->bp), c->d, c->b, steps));
}

}  // namespace

extern "C" {

static int dem_init_impl(dem_ctx **out, int32_t n_scenes, const int64_t *offsets, int64_t n,
                         const float *pos_r, const float *vel, const dem_params *prm, float dt,
                         const lvb_box *box, const lvb_skin_policy *skin, int32_t trigger,
                         float cell_factor, void *stream)
{
    if (!out) return LVB_EINVAL;
    *out = nullptr;
    if (!pos_r || !vel || !prm || !box || !skin || n < 1 || n > INT32_MAX - 64) return LVB_EINVAL;
    if (!(dt > 0.0f) || !(prm->kn >= 0.0f) || !(prm->rho > 0.0f) ||
        !(prm->restitution > 0.0f && prm->restitution <= 1.0f))
        return LVB_EINVAL;
    if (prm->wall_kind < DEM_WALL_NONE || prm->wall_kind > DEM_WALL_SPECULAR) return LVB_EINVAL;
    if (!(prm->mu >= 0.0f) || !std::isfinite(prm->mu)) return LVB_EINVAL;
    if (prm->mu > 0.0f && (!(prm->kt_ratio > 0.0f) || !std::isfinite(prm->kt_ratio) ||
                           !(prm->gt_ratio >= 0.0f) || !std::isfinite(prm->gt_ratio) ||
                           trigger != LVB_TRIGGER_PARTIAL))
        return LVB_EINVAL;
    if (((uintptr_t)pos_r & 15u) || ((uintptr_t)vel & 15u)) return LVB_EINVAL;
    cudaGetLastError();   // clear a stale error of an unrelated earlier call
    dem_ctx *c = new (std::nothrow) dem_ctx();
    if (!c) return LVB_ENOMEM;
    c->prm = *prm;
    c->stream = (cudaStream_t)stream;
    DemDev &d = c->d;
    d.n = (int)n;
    d.dt = dt;
    d.half_dt = 0.5f * dt;
    d.half_dt2 = (float)(0.5 * (double)dt * (double)dt);
    d.kn = prm->kn;
    const double le = std::log((double)prm->restitution);
    d.two_zeta = (float)(2.0 * (-le / std::sqrt(M_PI * M_PI + le * le)));
    for (int k = 0; k < 3; ++k) d.g[k] = prm->g[k];
    d.wall_kind = prm->wall_kind;
    d.clamp_tensile = prm->clamp_tensile;
    d.contacts_on = prm->contacts_on;
    d.drum_cx = prm->drum_cx;
    d.drum_cz = prm->drum_cz;
    d.drum_R = prm->drum_R;
    d.mu = prm->mu;
    d.kt = prm->kt_ratio * prm->kn;
    d.gt_ratio = prm->gt_ratio;
    cudaError_t e = cudaMalloc((void **)&d.pos, sizeof(float4) * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&d.vel, sizeof(float4) * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&d.acc, sizeof(float4) * n);
    if (e == cudaSuccess) e = cudaMalloc((void **)&d.vstar, sizeof(float4) * n);
    if (prm->mu > 0.0f) {
        if (e == cudaSuccess) e = cudaMalloc((void **)&d.omega, sizeof(float4) * n);
        if (e == cudaSuccess) e = cudaMalloc((void **)&d.alpha, sizeof(float4) * n);
        if (e == cudaSuccess) e = cudaMalloc((void **)&d.wstar, sizeof(float4) * n);
    }
    if (d.contacts_on) {
        if (e == cudaSuccess)
            e = cudaHostAlloc((void **)&c->sample, sizeof(*c->sample), cudaHostAllocMapped);
        if (e == cudaSuccess) {
            *c->sample = 0;
            e = cudaHostGetDevicePointer((void **)&c->sample_d, c->sample, 0);
        }
    }
    if (e != cudaSuccess) {
        dem_free(c);
        delete c;
        return from_cuda(e);
    }
    c->b.x[0] = d.pos;
    c->b.v[0] = d.vel;
    c->b.a[0] = d.acc;
    c->b.w[0] = d.omega;
    c->b.al[0] = d.alpha;
    k_dem_setup<<<std::min(grid_n((int)n), 4 * kNumSMs), kThreads, 0, c->stream>>>(
        d, (const float4 *)pos_r, (const float4 *)vel, prm->rho);
    int rc = offsets ? lvb_batch_init(&c->bp, n_scenes, offsets, (const float *)d.pos, box, skin,
                                      trigger, cell_factor, (const float *)d.vstar,
                                      (const float *)d.acc, stream)
                     : lvb_init(&c->bp, n, (const float *)d.pos, box, skin, trigger, cell_factor,
                                (const float *)d.vstar, (const float *)d.acc, stream);
    if (rc) {
        c->bp = nullptr;
        dem_free(c);
        delete c;
        return rc;
    }
    if (prm->mu > 0.0f) {   // the tangential springs live in the contact history
        rc = lvb_set_option(c->bp, LVB_OPT_HISTORY, 1);
        if (rc) {
            dem_free(c);
            delete c;
            return rc;
        }
    }
    d.rows = rows_view(c->bp);
    // a0 from the forces at (x0, v0): one force pass with a = 0, dt = 0
    // (the tangential springs start at zero: this pass leaves them alone,
    // and al0 = 0)
    DemDev d0 = d;
    d0.half_dt = 0.0f;
    d0.omega = d0.alpha = d0.wstar = nullptr;
    k_forces<false><<<grid_n(d.n), kThreads, 0, c->stream>>>(d0);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = ask_sample(c);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) {
        dem_free(c);
        delete c;
        return from_cuda(e);
    }
    if (!keeps_apart(c)) second_buffers(c, true);
    *out = c;
    return LVB_OK;
}

int dem_init(dem_ctx **out, int64_t n, const float *pos_r, const float *vel,
             const dem_params *prm, float dt, const lvb_box *box, const lvb_skin_policy *skin,
             int32_t trigger, float cell_factor, void *stream)
{
    return dem_init_impl(out, 1, nullptr, n, pos_r, vel, prm, dt, box, skin, trigger,
                         cell_factor, stream);
}

int dem_batch_init(dem_ctx **out, int32_t n_scenes, const int64_t *offsets, const float *pos_r,
                   const float *vel, const dem_params *prm, float dt, const lvb_box *boxes,
                   const lvb_skin_policy *skin, int32_t trigger, float cell_factor, void *stream)
{
    if (!offsets || n_scenes < 1) return LVB_EINVAL;
    return dem_init_impl(out, n_scenes, offsets, offsets[n_scenes], pos_r, vel, prm, dt, boxes,
                         skin, trigger, cell_factor, stream);
}

int dem_phase(dem_ctx *c, int32_t phase)
{
    if (!c) return LVB_EINVAL;
    cudaGetLastError();
    // the row store may have been re-laid out; pointers stay the same
    return launch_phase(c, phase);
}

int dem_advance(dem_ctx *c, int64_t steps)
{
    if (!c || steps < 0) return LVB_EINVAL;
    cudaGetLastError();   // clear a stale error of an unrelated earlier call
    for (int64_t done = 0; done < steps;) {
        const int64_t m = std::min<int64_t>(DEM_GRAPH_STEPS, steps - done);
        const int rc = launch_advance(c, (int)m);
        if (rc) return rc;
        done += m;
    }
    return LVB_OK;
}

static int contact_list(dem_ctx *c, int both, int32_t *ci, int32_t *cj, float *force3,
                        float *delta, float *xi3, int64_t cap, int64_t *n_contacts);

int dem_get_contact_forces(dem_ctx *c, int32_t *ci, int32_t *cj, float *force3, float *delta,
                           int64_t cap, int64_t *n_contacts)
{
    return contact_list(c, 0, ci, cj, force3, delta, nullptr, cap, n_contacts);
}

int dem_get_contact_history(dem_ctx *c, int32_t sides, int32_t *ci, int32_t *cj, float *force3,
                            float *delta, float *xi3, int64_t cap, int64_t *n_contacts)
{
    if (sides != 1 && sides != 2) return LVB_EINVAL;
    return contact_list(c, sides == 2, ci, cj, force3, delta, xi3, cap, n_contacts);
}

int dem_get_rot_state(dem_ctx *c, float *omega, float *alpha, float *omega_star)
{
    if (!c) return LVB_EINVAL;
    const size_t b = sizeof(float4) * (size_t)c->d.n;
    cudaError_t e = cudaSuccess;
    float *outs[3] = {omega, alpha, omega_star};
    const float4 *srcs[3] = {c->d.omega, c->d.alpha, c->d.wstar};
    for (int k = 0; k < 3 && e == cudaSuccess; ++k) {
        if (!outs[k]) continue;
        if (srcs[k]) e = cudaMemcpyAsync(outs[k], srcs[k], b, cudaMemcpyDefault, c->stream);
        else e = cudaMemsetAsync(outs[k], 0, b, c->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return from_cuda(e);
}

static int contact_list(dem_ctx *c, int both, int32_t *ci, int32_t *cj, float *force3,
                        float *delta, float *xi3, int64_t cap, int64_t *n_contacts)
{
    if (!c || !n_contacts || cap < 0 || (cap > 0 && (!ci || !cj || !force3 || !delta)))
        return LVB_EINVAL;
    *n_contacts = 0;
    refresh(c);
    const long long cp = std::max<long long>(cap, 1);
    int *di = nullptr, *dj = nullptr;
    float *df = nullptr, *dd = nullptr, *dx = nullptr;
    unsigned long long *cnt = nullptr;
    cudaError_t e = cudaMalloc((void **)&cnt, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc((void **)&di, sizeof(int) * cp);
    if (e == cudaSuccess) e = cudaMalloc((void **)&dj, sizeof(int) * cp);
    if (e == cudaSuccess) e = cudaMalloc((void **)&df, sizeof(float) * 3 * cp);
    if (e == cudaSuccess) e = cudaMalloc((void **)&dd, sizeof(float) * cp);
    if (e == cudaSuccess && xi3) e = cudaMalloc((void **)&dx, sizeof(float) * 3 * cp);
    unsigned long long total = 0;
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(total), c->stream);
    if (e == cudaSuccess) {
        k_contact_list<<<grid_n(c->d.n), kThreads, 0, c->stream>>>(c->d, cnt, cap, di, dj, df,
                                                                     dd, dx, both);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&total, cnt, sizeof(total), cudaMemcpyDeviceToHost, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    const long long m = std::min<long long>((long long)total, cap);
    if (e == cudaSuccess && m > 0) {
        e = cudaMemcpyAsync(ci, di, sizeof(int) * m, cudaMemcpyDefault, c->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(cj, dj, sizeof(int) * m, cudaMemcpyDefault, c->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(force3, df, sizeof(float) * 3 * m, cudaMemcpyDefault, c->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(delta, dd, sizeof(float) * m, cudaMemcpyDefault, c->stream);
        if (e == cudaSuccess && xi3)
            e = cudaMemcpyAsync(xi3, dx, sizeof(float) * 3 * m, cudaMemcpyDefault, c->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    }
    cudaFree(cnt);
    cudaFree(di);
    cudaFree(dj);
    cudaFree(df);
    cudaFree(dd);
    if (dx) cudaFree(dx);
    if (e != cudaSuccess) return from_cuda(e);
    *n_contacts = (int64_t)total;
    const int rc = lvb_sync(c->bp);
    if (rc) return rc;
    return (long long)total > cap ? LVB_ECAPACITY : LVB_OK;
}

int dem_get_state(dem_ctx *c, float *pos_r, float *vel, float *acc, float *vstar)
{
    if (!c) return LVB_EINVAL;
    const size_t b = sizeof(float4) * (size_t)c->d.n;
    cudaError_t e = cudaSuccess;
    if (pos_r) e = cudaMemcpyAsync(pos_r, c->d.pos, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && vel) e = cudaMemcpyAsync(vel, c->d.vel, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && acc) e = cudaMemcpyAsync(acc, c->d.acc, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && vstar)
        e = cudaMemcpyAsync(vstar, c->d.vstar, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return from_cuda(e);
}

int dem_set_state(dem_ctx *c, const float *pos_r, const float *vel, const float *acc)
{
    if (!c) return LVB_EINVAL;
    const size_t b = sizeof(float4) * (size_t)c->d.n;
    cudaError_t e = cudaSuccess;
    if (pos_r) e = cudaMemcpyAsync(c->d.pos, pos_r, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && vel) e = cudaMemcpyAsync(c->d.vel, vel, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && vel) {
        const int grid = std::min(grid_n((int)c->d.n), 4 * kNumSMs);
        k_restore_im<<<grid, kThreads, 0, c->stream>>>(c->d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && acc) e = cudaMemcpyAsync(c->d.acc, acc, b, cudaMemcpyDefault, c->stream);
    if (e == cudaSuccess && pos_r) {
        refresh(c);
        e = ask_sample(c);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    return from_cuda(e);
}

int dem_lvb(dem_ctx *c, lvb_ctx **out)
{
    if (!c || !out) return LVB_EINVAL;
    *out = c->bp;
    return LVB_OK;
}

int dem_device_state(dem_ctx *c, float **pos_r, float **vel, float **acc, float **vstar)
{
    if (!c) return LVB_EINVAL;
    if (pos_r) *pos_r = (float *)c->d.pos;
    if (vel) *vel = (float *)c->d.vel;
    if (acc) *acc = (float *)c->d.acc;
    if (vstar) *vstar = (float *)c->d.vstar;
    return LVB_OK;
}

int dem_sync(dem_ctx *c)
{
    if (!c) return LVB_EINVAL;
    return lvb_sync(c->bp);
}

int dem_destroy(dem_ctx *c)
{
    if (!c) return LVB_EINVAL;
    cudaStreamSynchronize(c->stream);
    dem_free(c);
    delete c;
    return LVB_OK;
}

}  // extern "C"
