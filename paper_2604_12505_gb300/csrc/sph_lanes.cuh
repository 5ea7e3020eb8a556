// sph_lanes.cuh -- the particle sums of Eqs. 10-19 by several lanes per
// particle.  A lane evaluates a few consecutive candidates; the sums then go
// on from lane to lane, so that they add in the order in which one lane alone
// would, and equal its sums bit for bit.  (Broadcasting every candidate to all
// lanes instead is bound by the shuffles: 48 per 16 candidates, against 8.)
// Where the compiler could contract a product and a sum in more than one way,
// the rounding of density_kernel and force_kernel is written out.
#pragma once

#include <cfloat>

#include "sph_common.cuh"

namespace sph {

constexpr int kChunk = 4;  // candidates that a lane evaluates at once

// Lane l's value, of the LN lanes of this lane's particle.
template <int LN, class V>
__device__ __forceinline__ V from_lane(V v, int l)
{
    return __shfl_sync(0xffffffffu, v, l, LN);
}

// Up to three runs of a sorted list, one after the other: entry k lies at
// at(k).  A warp's particles are walked together, as far as the longest: `most`.
struct Runs {
    int o0, o1, o2, n0, n1, n, most;
    __device__ int at(int k) const { return k + (k < n0 ? o0 : k < n1 ? o1 : o2); }
};
// From the runs' starts and lengths, 16 bits each.
__device__ __forceinline__ unsigned pack_run(int a, int z) { return (unsigned)a | (unsigned)max(z - a, 0) << 16; }
__device__ __forceinline__ Runs unpack_runs(unsigned p0, unsigned p1, unsigned p2)
{
    Runs R;
    R.n0 = (int)(p0 >> 16);
    R.n1 = R.n0 + (int)(p1 >> 16);
    R.n = R.n1 + (int)(p2 >> 16);
    R.o0 = (int)(p0 & 0xffffu);
    R.o1 = (int)(p1 & 0xffffu) - R.n0;
    R.o2 = (int)(p2 & 0xffffu) - R.n1;
    R.most = __reduce_max_sync(0xffffffffu, R.n);
    return R;
}
// Run r of a particle was found by its lane r, LN >= 4.
template <int LN>
__device__ __forceinline__ Runs lane_runs(unsigned mine)
{
    return unpack_runs(from_lane<LN>(mine, 0), from_lane<LN>(mine, 1), from_lane<LN>(mine, 2));
}

// The bracket of Eq. 22 at distance r = sqrt(r2), as rounded for fluid and for
// ghosts; the caller selects by r < 2h.
__device__ __forceinline__ float fluid_bracket(const TankDev& T, float r2)
{
    const float inv_r = rsqrtf(fmaxf(r2, FLT_MIN));
    const float q = r2 * inv_r * T.inv_h;
    const float qa = 2.0f - q, qb = fmaxf(1.0f - q, 0.0f);
    return fmaf(-4.0f * qb * qb, qb, qa * qa * qa);
}
__device__ __forceinline__ float ghost_bracket(const TankDev& T, float r2)
{
    const float inv_r = rsqrtf(fmaxf(r2, FLT_MIN));
    const float q = __fmul_rn(r2 * inv_r, T.inv_h);
    const float qa = __fsub_rn(2.0f, q), qb = fmaxf(__fsub_rn(1.0f, q), 0.0f);
    return fmaf(-4.0f * qb * qb, qb, qa * qa * qa);
}

// Eqs. 10 and 12 between particles d apart, over the distance (r2 > 0).
__device__ __forceinline__ float pair_force(const TankDev& T, float4 pi, float2 ri, float4 pj, float2 rj, float2 d, float r2)
{
    const float inv_r = rsqrtf(fmaxf(r2, FLT_MIN));
    const float q = __fmul_rn(r2 * inv_r, T.inv_h);
    const float qa = __fsub_rn(2.0f, q), qb = fmaxf(__fsub_rn(1.0f, q), 0.0f);
    const float gW = T.cdW * fmaf(12.0f * qb, qb, __fmul_rn(-3.0f * qa, qa)) * inv_r;
    const float press = -(ri.y + rj.y);                                  // Eq. 10
    const float vr = fmaf(pi.w - pj.w, d.y, __fmul_rn(pi.z - pj.z, d.x));
    const float visc = __fdividef(T.visc_a * vr, (ri.x + rj.x) * (r2 + T.epsh2));  // Eq. 12
    return T.m * (press + visc) * gW;
}

// Eqs. 16 and 18 of a ghost, likewise.
__device__ __forceinline__ float ghost_force(const TankDev& T, float4 pi, float2 ri, float4 gv, float2 d2, float r2)
{
    const float ddx = d2.x, ddy = d2.y;
    const float mm = T.m * T.m;
    const float qg = T.gp_clamp ? fmaxf(ri.y, 0.f) : ri.y;
    const float inv_r = rsqrtf(r2);
    const float rr = r2 * inv_r;
    const float d = T.h - rr;
    const float gWs = T.cdS * d * d * inv_r;                         // (dW_s3/dr)/r
    const float fp = T.gp_sign * 2.0f * mm * qg * gWs;              // Eq. 16
    const float vr = (pi.z - gv.x) * ddx + (pi.w - gv.y) * ddy;
    const float fv = __fdividef(mm * T.beta2 * fminf(vr, 0.f), (ri.x + ri.x) * (r2 + T.epsh2)) * gWs;  // Eq. 18
    return fp + fv;
}

// Eqs. 17, 19 and the torque: a ghost's force over the distance, the distance
// and its arm; of(l) is lane l's sum.
struct WallSum {
    float fx, fy, t;
    __device__ void add(float f, float2 d, float2 arm)
    {
        const float x = __fmul_rn(f, d.x), y = __fmul_rn(f, d.y);
        fx = __fsub_rn(fx, x);
        fy = __fsub_rn(fy, y);
        t = __fsub_rn(t, fmaf(arm.x, y, -__fmul_rn(arm.y, x)));
    }
    template <int LN>
    __device__ WallSum of(int l) const
    {
        return {from_lane<LN>(fx, l), from_lane<LN>(fy, l), from_lane<LN>(t, l)};
    }
};
struct BothSum : WallSum {  // and the acceleration of the particle
    float ax, ay, inv_m;
    __device__ void add(float f, float2 d, float2 arm)
    {
        ax = fmaf(__fmul_rn(f, d.x), inv_m, ax);
        ay = fmaf(__fmul_rn(f, d.y), inv_m, ay);
        WallSum::add(f, d, arm);
    }
    template <int LN>
    __device__ BothSum of(int l) const
    {
        return {WallSum::of<LN>(l), from_lane<LN>(ax, l), from_lane<LN>(ay, l), inv_m};
    }
};

// Eq. 14's fluid sum of particle e of a sorted list over its runs R.
template <int LN>
__device__ __forceinline__ float fluid_sum(const TankDev& T, const Runs& R, int e, float4 pi, float2 li, const float4* pv,
                                           const float2* plo, int sub)
{
    float Sf = 0.f;
    for (int k0 = 0; k0 < R.most; k0 += LN * kChunk) {
        float f[kChunk];
#pragma unroll
        for (int u = 0; u < kChunk; ++u) {
            const int k = k0 + sub * kChunk + u;
            const int j = k < R.n ? R.at(k) : e;
            const float2 d = sep_ff(pi, li, pv[j], plo[j]);
            const float r2 = dist2(d.x, d.y);
            const float w = fluid_bracket(T, r2);
            f[u] = r2 < T.R2 && k < R.n ? w : 0.0f;
        }
#pragma unroll
        for (int l = 0; l < LN; ++l) {
            float t = Sf;
#pragma unroll
            for (int u = 0; u < kChunk; ++u) t += f[u];
            Sf = from_lane<LN>(t, l);
        }
    }
    return Sf;
}

// Eq. 14's ghost sum over the ghosts Q, the factor cW with the sum.
template <int LN>
__device__ __forceinline__ float ghost_sum(const TankDev& T, const Runs& Q, float4 pi, float2 li, const float4* gp, int sub)
{
    float Sg = 0.f;
    for (int k0 = 0; k0 < Q.most; k0 += LN * kChunk) {
        float f[kChunk];
#pragma unroll
        for (int u = 0; u < kChunk; ++u) {
            const int k = k0 + sub * kChunk + u;
            const float2 d = sep_fg(pi, li, gp[k < Q.n ? Q.at(k) : 0]);
            const float r2 = dist2(d.x, d.y);
            const float w = ghost_bracket(T, r2);
            f[u] = k < Q.n && r2 < T.R2 ? w : 0.0f;
        }
#pragma unroll
        for (int l = 0; l < LN; ++l) {
            float t = Sg;
#pragma unroll
            for (int u = 0; u < kChunk; ++u) t = fmaf(T.cW, f[u], t);
            Sg = from_lane<LN>(t, l);
        }
    }
    return Sg;
}

// Eqs. 10 and 12 as (ax, ay), zero before; returns the neighbours that this lane met.
template <int LN>
__device__ __forceinline__ int fluid_forces(const TankDev& T, const Runs& R, int e, float4 pi, float2 li, float2 ri,
                                            const float4* pv, const float2* plo, const float2* rho, int sub, float& ax,
                                            float& ay)
{
    int met = 0;
    for (int k0 = 0; k0 < R.most; k0 += LN * kChunk) {
        float f[kChunk];
        float2 d[kChunk];
#pragma unroll
        for (int u = 0; u < kChunk; ++u) {
            const int k = k0 + sub * kChunk + u;
            const int j = k < R.n ? R.at(k) : e;
            const float4 pj = pv[j];
            d[u] = sep_ff(pi, li, pj, plo[j]);
            const float r2 = dist2(d[u].x, d[u].y);
            const bool nb = r2 < T.R2 && j != e;
            const float s = pair_force(T, pi, ri, pj, rho[j], d[u], r2);
            f[u] = nb && r2 > 0.f ? s : 0.f;
            met += nb;
        }
#pragma unroll
        for (int l = 0; l < LN; ++l) {
            float tx = ax, ty = ay;
#pragma unroll
            for (int u = 0; u < kChunk; ++u) {
                tx = fmaf(f[u], d[u].x, tx);
                ty = fmaf(f[u], d[u].y, ty);
            }
            ax = from_lane<LN>(tx, l);
            ay = from_lane<LN>(ty, l);
        }
    }
    // At a position that is not finite the sums of zero forces are not zero.  (Such
    // a particle lies in the grid's outermost cells, where fluid inside the wall
    // has it in no stencil.)
    if (const float a = ax + ay; a != a && !(isfinite(pi.x) && isfinite(pi.y))) ax = ay = 0.f;
    return met;
}

// Eqs. 16-19 with the ghosts Q, added to W; returns the ghosts that this lane met.
template <int LN, class W_>
__device__ __forceinline__ int ghost_forces(const TankDev& T, const Runs& Q, float4 pi, float2 li, float2 ri,
                                            const float4* gp, const float4* gvel, int sub, W_& W)
{
    int n_met = 0;
    if (Q.most == 0) return 0;
    // a particle that reaches no ghost, one off the grid among them, goes
    // through the rounds of its warp with forces of zero over finite distances
    if (Q.n == 0) {
        pi.x = pi.y = 0.f;
        li = make_float2(0.f, 0.f);
    }
    for (int k0 = 0; k0 < Q.most; k0 += LN * kChunk) {
        float f[kChunk];
        float2 d[kChunk], arm[kChunk];
        bool any = false;
#pragma unroll
        for (int u = 0; u < kChunk; ++u) {
            const int k = k0 + sub * kChunk + u, g = k < Q.n ? Q.at(k) : 0;
            d[u] = sep_fg(pi, li, gp[g]);
            const float r2 = dist2(d[u].x, d[u].y);
            const bool met = k < Q.n && r2 < T.h2;
            f[u] = 0.f;
            arm[u] = make_float2(0.f, 0.f);
            if (met && r2 > 0.f) {
                const float4 gv = gvel[g];
                f[u] = ghost_force(T, pi, ri, gv, d[u], r2);
                arm[u] = make_float2(gv.z, gv.w);
            }
            n_met += met;
            any |= met;
        }
        const unsigned hit = __ballot_sync(0xffffffffu, any);
#pragma unroll
        for (int l = 0; l < LN; ++l)
            if (hit & (0xffffffffu / ((1u << LN) - 1u) << l)) {  // some particle's lane l
                W_ V = W;
#pragma unroll
                for (int u = 0; u < kChunk; ++u) V.add(f[u], d[u], arm[u]);
                W = V.template of<LN>(l);
            }
    }
    return n_met;
}

}  // namespace sph
