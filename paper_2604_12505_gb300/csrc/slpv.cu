// slpv.cu -- the self-scheduled LPV surrogate of the identification study
// (Section 4, Eqs. 24-27; Section 5.3.2) behind the C ABI of include/slpv.h:
// free-run loss and its gradient by backpropagation through time, Adam, the
// free run of the augmented model and its closed loop with the PD law of
// Eq. 28.
//
// The state (nx <= 8), the scheduling network (two layers of four tanh
// neurons) and the 7 x 7 matrices of the paper's model are far below a
// tensor-core tile, and every step depends on the previous one, so the work
// is FP32 FMA chains.  The fit splits each trajectory's recurrences over a
// few lanes and does everything that is not serial in k over all samples at
// once; sums are taken in a fixed order, so results are deterministic.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/slpv.h"

namespace sph {
int set_last_error(int code, const char* msg);
}

namespace slpvk {

constexpr int NU = 3, NY = 3, NH = 4;

// Offsets of the blocks of theta (see include/slpv.h).
template <int NX>
struct Lay {
    static constexpr int NZ = NX + NU, NO = NX + NY, NM = NO * NZ;
    static constexpr int M0 = 0, M1 = NM, W1 = 2 * NM, B1 = W1 + NH * NZ, W2 = B1 + NH, B2 = W2 + NH * NH;
    static constexpr int W3 = B2 + NH, B3 = W3 + NH, N = B3 + 1;
};

inline int n_params(int nx)
{
    const int nz = nx + NU, no = nx + NY;
    return 2 * no * nz + NH * nz + NH + NH * NH + NH + NH + 1;
}

// Training stages: which entries of theta move (never the D blocks).
enum { kStageAll = 0, kStageLti = 1, kStageScheduling = 2 };

// Whether theta[q] is trained in `stage`: all entries, M_0 only (the LTI
// stage), or M_1 and the network only (M_0 held).
__host__ __device__ inline bool trainable(int q, int nx, int stage)
{
    const int nz = nx + NU, nm = (nx + NY) * nz;
    if (q < 2 * nm) {
        if (stage == kStageLti && q >= nm) return false;
        if (stage == kStageScheduling && q < nm) return false;
        const int r = (q % nm) / nz, j = (q % nm) % nz;
        return !(r >= nx && j >= nx);
    }
    return stage != kStageLti;
}

// Scheduling map eta(z) = w3 . tanh(W2 tanh(W1 z + b1) + b2) + b3.
template <int NX>
__device__ __forceinline__ float eta(const float* th, const float* z, float* h1, float* h2)
{
    using Q = Lay<NX>;
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        float a = th[Q::B1 + i];
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j) a = fmaf(th[Q::W1 + i * Q::NZ + j], z[j], a);
        h1[i] = tanhf(a);
    }
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        float a = th[Q::B2 + i];
#pragma unroll
        for (int j = 0; j < NH; ++j) a = fmaf(th[Q::W2 + i * NH + j], h1[j], a);
        h2[i] = tanhf(a);
    }
    float p = th[Q::B3];
#pragma unroll
    for (int i = 0; i < NH; ++i) p = fmaf(th[Q::W3 + i], h2[i], p);
    return p;
}

// o = (M_0 + p M_1) z = [x_{k+1}; y_k] (Eqs. 24, 25).
template <int NX>
__device__ __forceinline__ void mz(const float* th, float p, const float* z, float* o)
{
    using Q = Lay<NX>;
#pragma unroll
    for (int r = 0; r < Q::NO; ++r) {
        float a = 0.f;
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j) a = fmaf(fmaf(p, th[Q::M1 + r * Q::NZ + j], th[Q::M0 + r * Q::NZ + j]), z[j], a);
        o[r] = a;
    }
}

// ---------------------------------------------------------------------------
// Loss and gradient in four passes.
//
// Only two recurrences run along k: the state x_{k+1} and the adjoint
// lambda_k.  The adjoint's step is linear, lambda_k = J_k^T lambda_{k+1} +
// c_k, with J_k and c_k functions of x_k alone, and so are every sample's
// residual and its contribution to the gradient once lambda is known:
//   state_kernel    x_k for all k (serial; NX lanes or more per trajectory)
//   sample_kernel   squared errors, J_k and c_k (one thread per sample)
//   adjoint_kernel  lambda_k (in segments of the time axis; one lane per state)
//   outer_kernel    the gradient's outer products over all samples
//   final_kernel    sums of the block partials, the l2 term, the mask
// One thread per trajectory running both recurrences with everything on the
// chain took 2,600 cycles per sample: 2.73 ms for 24 trajectories of 2,200
// samples (n_x = 4), now 0.39 ms (state 339 us, adjoint 19, outer 11, sample
// 9, final 6).  The state chain's latencies add up to 293 cycles of its 318
// a sample: 7 FMAs, tanhf (62), a shuffle (26), 4 FMAs, tanhf, a shuffle, 4
// FMAs, 8 FMAs and a shuffle.
// ---------------------------------------------------------------------------

// Lanes that share a trajectory in the serial passes: one per state and at
// least one per neuron.
template <int NX>
constexpr int kLanes = NX <= 4 ? 4 : 8;

template <int N>
__device__ __forceinline__ void load_vec(const float* __restrict__ p, float* v)  // N even, p 8-byte aligned (16 for N % 4 == 0)
{
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 q = *reinterpret_cast<const float4*>(p + i);
            v[i] = q.x, v[i + 1] = q.y, v[i + 2] = q.z, v[i + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 2) {
            const float2 q = *reinterpret_cast<const float2*>(p + i);
            v[i] = q.x, v[i + 1] = q.y;
        }
    }
}

// Asynchronous copies into shared memory, a queue of whole chunks: the serial
// passes read their inputs there, so that no step waits on a global load (a
// register ring of loads was measured first: a wait on one load also waited
// for later ones, 200 of 527 cycles a step).
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait()  // until at most the N youngest chunks are in flight
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
    __syncwarp();
}
constexpr int kStages = 4;   // chunks in shared memory: one in use, three in flight
constexpr int kChunk = 32;   // steps per chunk of the state pass

template <int N>
__device__ __forceinline__ void store_vec(float* p, const float* v)
{
    if constexpr (N % 4 == 0) {
#pragma unroll
        for (int i = 0; i < N; i += 4) *reinterpret_cast<float4*>(p + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 2) *reinterpret_cast<float2*>(p + i) = make_float2(v[i], v[i + 1]);
    }
}

// States x_k, k in [k0, k0 + len), of every trajectory into xh[traj][ld][NX]
// (row k - k0), from carry[traj][NX] (k0 = 0: from rest); the state after the
// window goes to carry.  Lane l of a trajectory's group computes neuron l % 4
// of each layer and row l % NX of M(p) z, each by the same chain of FMAs as
// the sample pass, so both see the same bits; shuffles hand the neurons and
// the new state around.  Bound by that chain: two layers (an FMA chain, a
// tanhf and a shuffle each), eta's output, the row's FMAs and a shuffle.
// One warp per block: the few trajectories of a fit spread over the SMs.
template <int NX>
__global__ void __launch_bounds__(32) state_kernel(const float* __restrict__ theta, const float* __restrict__ u,
                                                   const float* __restrict__ scales, int n_traj, int T, int k0, int len,
                                                   int ld, float* __restrict__ carry, float* __restrict__ xh)
{
    using Q = Lay<NX>;
    constexpr int L = kLanes<NX>, PER = 32 / L;
    const int l = (int)threadIdx.x % L, nr = l % NH, row = l % NX;
    const int tr = blockIdx.x * PER + (int)threadIdx.x / L;
    const bool own = tr < n_traj && l < NX;
    const size_t t = tr < n_traj ? tr : n_traj - 1;
    float w1[Q::NZ], w2[NH], w3[NH], m0[Q::NZ], m1[Q::NZ], x[NX];
#pragma unroll
    for (int j = 0; j < Q::NZ; ++j) {
        w1[j] = theta[Q::W1 + nr * Q::NZ + j];
        m0[j] = theta[Q::M0 + row * Q::NZ + j];
        m1[j] = theta[Q::M1 + row * Q::NZ + j];
    }
#pragma unroll
    for (int j = 0; j < NH; ++j) {
        w2[j] = theta[Q::W2 + nr * NH + j];
        w3[j] = theta[Q::W3 + j];
    }
    const float b1 = theta[Q::B1 + nr], b2 = theta[Q::B2 + nr], b3 = theta[Q::B3];
    float isu[NU];
#pragma unroll
    for (int c = 0; c < NU; ++c) isu[c] = 1.0f / scales[c];
#pragma unroll
    for (int i = 0; i < NX; ++i) x[i] = k0 ? carry[t * NX + i] : 0.f;
    float* xo = xh + t * ld * NX + row;
    __shared__ float su[kStages][PER][kChunk * NU + 1];
    const int n_chunk = (len + kChunk - 1) / kChunk, grp = (int)threadIdx.x / L;
    const float* ul = u + (t * T + k0) * NU + l;
    auto fetch = [&](int c) {  // the lanes of a group copy their trajectory's inputs
        float* dst = &su[c % kStages][grp][l];
        const float* src = ul + (size_t)c * (kChunk * NU);
        const int n = (len - c * kChunk) * NU - l;
        if (n > kChunk * NU - L) {
#pragma unroll
            for (int i = 0; i < kChunk * NU; i += L) copy_async<4>(dst + i, src + i);
        } else {
            for (int i = 0; i < n; i += L) copy_async<4>(dst + i, src + i);
        }
        copy_commit();
    };
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c) fetch(c);
    float mine = x[0];
#pragma unroll
    for (int i = 1; i < NX; ++i) mine = row == i ? x[i] : mine;
    auto step = [&](int k, const float* us) {
        if (own) xo[(size_t)k * NX] = mine;
        float z[Q::NZ], h1[NH], h2[NH];
#pragma unroll
        for (int i = 0; i < NX; ++i) z[i] = x[i];
#pragma unroll
        for (int c = 0; c < NU; ++c) z[NX + c] = us[c] * isu[c];
        float a = b1;
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j) a = fmaf(w1[j], z[j], a);
        float h = tanhf(a);
#pragma unroll
        for (int j = 0; j < NH; ++j) h1[j] = __shfl_sync(0xffffffffu, h, j, L);
        a = b2;
#pragma unroll
        for (int j = 0; j < NH; ++j) a = fmaf(w2[j], h1[j], a);
        h = tanhf(a);
#pragma unroll
        for (int j = 0; j < NH; ++j) h2[j] = __shfl_sync(0xffffffffu, h, j, L);
        float p = b3;
#pragma unroll
        for (int j = 0; j < NH; ++j) p = fmaf(w3[j], h2[j], p);
        a = 0.f;
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j) a = fmaf(fmaf(p, m1[j], m0[j]), z[j], a);
        mine = a;
#pragma unroll
        for (int i = 0; i < NX; ++i) x[i] = __shfl_sync(0xffffffffu, a, i, L);
    };
    for (int c = 0; c < n_chunk; ++c) {
        copy_wait<kStages - 2>();
        fetch(c + kStages - 1);  // its buffer was read in the chunk before: that reading is behind the wait's barrier
        const float* us = su[c % kStages][grp];
        const int n = min(kChunk, len - c * kChunk);
        if (n == kChunk) {
#pragma unroll 4
            for (int s = 0; s < kChunk; ++s) step(c * kChunk + s, us + s * NU);
        } else {
            for (int s = 0; s < n; ++s) step(c * kChunk + s, us + s * NU);
        }
    }
    if (own) carry[t * NX + row] = mine;
}

// z_k = [x_k; u_k / s_u], the scheduling and the outputs of one sample.
template <int NX>
struct Sample {
    float z[Lay<NX>::NZ], h1[NH], h2[NH], p, res[NY];  // res: y_hat - y / s_y
};

template <int NX>
__device__ __forceinline__ void eval_sample(const float* th, const float* __restrict__ scales, const float* x,
                                            const float* __restrict__ u, const float* __restrict__ y, Sample<NX>& S)
{
    using Q = Lay<NX>;
    load_vec<NX>(x, S.z);
#pragma unroll
    for (int c = 0; c < NU; ++c) S.z[NX + c] = u[c] * (1.0f / scales[c]);
    S.p = eta<NX>(th, S.z, S.h1, S.h2);
#pragma unroll
    for (int c = 0; c < NY; ++c) {
        float a = 0.f;
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j)
            a = fmaf(fmaf(S.p, th[Q::M1 + (NX + c) * Q::NZ + j], th[Q::M0 + (NX + c) * Q::NZ + j]), S.z[j], a);
        S.res[c] = a - y[c] * (1.0f / scales[3 + c]);
    }
}

// e[i] = d eta / d (pre-activation of neuron i of the first layer).
template <int NX>
__device__ __forceinline__ void eta_back(const float* th, const float* h1, const float* h2, float* d2, float* e)
{
    using Q = Lay<NX>;
#pragma unroll
    for (int i = 0; i < NH; ++i) d2[i] = th[Q::W3 + i] * (1.0f - h2[i] * h2[i]);
#pragma unroll
    for (int i = 0; i < NH; ++i) {
        float b = 0.f;
#pragma unroll
        for (int j = 0; j < NH; ++j) b = fmaf(th[Q::W2 + j * NH + i], d2[j], b);
        e[i] = b * (1.0f - h1[i] * h1[i]);
    }
}

// One thread per sample of the window (k fastest): the squared error, summed
// per block in FP64 into loss_part[block], and, when the gradient is wanted,
// the adjoint's step as a record adj[traj][k] of kRec floats: dx_{k+1,r} /
// dx_{k,j} at j NX + r, then the output residuals' part of each lambda_{k,j}.
// With M(p) and p = eta(z), do_r / dz_j = M(p)_rj + (M_1 z)_r E_j, E = W1^T e.
constexpr int kSampleThreads = 64;
template <int NX>
constexpr int kRec = (NX * NX + NX + 3) / 4 * 4;  // whole 16-byte vectors

template <int NX>
__global__ void __launch_bounds__(kSampleThreads)
    sample_kernel(const float* __restrict__ theta, const float* __restrict__ u, const float* __restrict__ y,
                  const float* __restrict__ scales, int n_traj, int T, int k0, int len, int ld, int xld, int xk0,
                  float inv_n, int want_grad, const float* __restrict__ xh, float* __restrict__ adj,
                  double* __restrict__ loss_part)
{
    using Q = Lay<NX>;
    __shared__ float th[Q::N];
    __shared__ double red[kSampleThreads / 32];
    for (int i = threadIdx.x; i < Q::N; i += kSampleThreads) th[i] = theta[i];
    __syncthreads();
    const long long n = (long long)n_traj * len;
    double lsum = 0.0;
    for (long long s = blockIdx.x * (long long)kSampleThreads + threadIdx.x; s < n;
         s += (long long)gridDim.x * kSampleThreads) {
        const size_t t = (size_t)(s / len);
        const int k = (int)(s % len);
        Sample<NX> S;
        const size_t row = (t * T + k0 + k) * 3;
        eval_sample<NX>(th, scales, xh + (t * xld + (k0 - xk0) + k) * NX, u + row, y + row, S);
        float e2 = 0.f;
#pragma unroll
        for (int c = 0; c < NY; ++c) e2 = fmaf(S.res[c], S.res[c], e2);
        lsum += (double)e2;
        if (!want_grad) continue;
        float d2[NH], e[NH], m1z[Q::NO], ar[NY];
        eta_back<NX>(th, S.h1, S.h2, d2, e);
#pragma unroll
        for (int r = 0; r < Q::NO; ++r) {
            m1z[r] = 0.f;
#pragma unroll
            for (int j = 0; j < Q::NZ; ++j) m1z[r] = fmaf(th[Q::M1 + r * Q::NZ + j], S.z[j], m1z[r]);
        }
        float sr = 0.f;  // the residuals' part of dJ/dp
#pragma unroll
        for (int c = 0; c < NY; ++c) {
            ar[c] = 2.0f * S.res[c] * inv_n;
            sr = fmaf(ar[c], m1z[NX + c], sr);
        }
        float* o = adj + (t * ld + k) * kRec<NX>;
        float cv[NX];
#pragma unroll
        for (int j = 0; j < NX; ++j) {
            float E = 0.f, J[NX];
#pragma unroll
            for (int i = 0; i < NH; ++i) E = fmaf(th[Q::W1 + i * Q::NZ + j], e[i], E);
            auto M = [&](int r) { return fmaf(S.p, th[Q::M1 + r * Q::NZ + j], th[Q::M0 + r * Q::NZ + j]); };
#pragma unroll
            for (int r = 0; r < NX; ++r) J[r] = fmaf(m1z[r], E, M(r));
            store_vec<NX>(o + j * NX, J);
            float v = sr * E;
#pragma unroll
            for (int c = 0; c < NY; ++c) v = fmaf(M(NX + c), ar[c], v);
            cv[j] = v;
        }
        store_vec<NX>(o + NX * NX, cv);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lsum;
    __syncthreads();
    if (threadIdx.x == 0) {
        double v = red[0];
        for (int w = 1; w < kSampleThreads / 32; ++w) v += red[w];
        loss_part[blockIdx.x] = v;
    }
}

// lambda_k = J_k^T lambda_{k+1} + c_k over the window, backwards from
// carry_in[traj][NX] (first, the last window: from zero); lam[traj][ld][NX]
// receives lambda_{k+1} at row k, carry_out the window's first lambda.  Lane j
// owns lambda_j: a step is NX shuffles and a chain of NX / 2 FMAs and an add.
// The records pass through shared memory in chunks, copied by the lanes of
// their own trajectory.
//
// The step is affine, so the time axis is cut into n_seg segments of seg_len
// samples that run side by side: with MAP, each but the first takes the unit
// vectors without and the zero vector with c_k from its end to its start, which
// is its map (map[traj][seg][NX + 1][NX]); then each segment starts from what
// the maps of the later ones give.  24 trajectories of 2,200 samples: 87 us in
// one chain, 19 in 28 segments (maps 7,
// lambdas 12).
template <int NX>
constexpr int kAdjChunk = NX <= 4 ? 16 : 8;

template <int NX, bool MAP>
__global__ void __launch_bounds__(32)
    adjoint_kernel(const float* __restrict__ adj, int n_traj, int len, int ld, int n_seg, int seg_len, int first,
                   const float* __restrict__ carry_in, float* __restrict__ carry_out, float* __restrict__ map,
                   float* __restrict__ lam)
{
    constexpr int L = kLanes<NX>, PER = 32 / L, C = kAdjChunk<NX>, R = kRec<NX>;
    // a trajectory's chunk padded by 4 floats: the groups of a warp read distinct banks
    __shared__ __align__(16) float sj[kStages][PER][C * R + 4];
    const int l = (int)threadIdx.x % L, j = l % NX, grp = (int)threadIdx.x / L;
    const int g = blockIdx.x * PER + grp;
    const int col = MAP ? g % (NX + 1) : NX;  // the map's column that this group computes
    const int sg = MAP ? g / (NX + 1) : g, per_traj = MAP ? n_seg - 1 : n_seg;
    const int tr = sg / per_traj, seg = sg % per_traj + (MAP ? 1 : 0);
    const bool own = tr < n_traj && l < NX;
    const size_t t = tr < n_traj ? tr : n_traj - 1;
    const int k0 = seg * seg_len, own_n = min(len - k0, seg_len);  // the segment's samples
    const float v_end = MAP ? (j == col ? 1.f : 0.f) : first ? 0.f : carry_in[t * NX + j];
    float v = v_end;
    int n = own_n, n_chunk = (seg_len + C - 1) / C;  // samples to go back over; chunks, the same in all groups of a warp
    auto at_map = [&](int s, int c) { return map + ((t * n_seg + s) * (NX + 1) + c) * NX + j; };
    if constexpr (!MAP) {
#pragma unroll 4
        for (int s = n_seg - 1; s >= 1; --s) {
            float w = *at_map(s, NX);
#pragma unroll
            for (int r = 0; r < NX; ++r) w = fmaf(*at_map(s, r), __shfl_sync(0xffffffffu, v, r, L), w);
            if (s > seg) v = w;
        }
        // a map that overflowed says nothing of the lambda it maps: from the window's end instead
        const unsigned bad = __ballot_sync(0xffffffffu, !isfinite(v));
        if (bad) {
            if (bad >> (threadIdx.x - l) & ((1u << L) - 1u)) {
                v = v_end;
                n = len - k0;
            }
            n_chunk = __reduce_max_sync(0xffffffffu, (n + C - 1) / C);
        }
    }
    float* lt = lam + (t * ld + k0) * NX + j;
    const float* at = adj + (t * ld + k0) * R;
    // chunk c holds steps n - (c + 1) C and on, C of them; those below 0 are not there
    auto fetch = [&](int c) {
        const int lo = n - (c + 1) * C;
        float* dst = &sj[c % kStages][grp][4 * l];
        const float* src = at + (ptrdiff_t)lo * R + 4 * l;
        if (lo >= 0) {
#pragma unroll
            for (int i = 0; i < C * R; i += 4 * L)
                if (C * R % (4 * L) == 0 || i + 4 * l < C * R) copy_async<16>(dst + i, src + i);
        } else {
            for (int i = 0; i + 4 * l < C * R; i += 4 * L)
                if (i + 4 * l >= -lo * R) copy_async<16>(dst + i, src + i);
        }
        copy_commit();
    };
    auto step = [&](int k, const float* rec, bool in) {
        if (!MAP && own && in && k < own_n) lt[(ptrdiff_t)k * NX] = v;
        float J[NX], a = col == NX ? rec[NX * NX + j] : 0.f, m = 0.f;
        load_vec<NX>(rec + j * NX, J);
#pragma unroll
        for (int r = 0; r < NX; r += 2) {
            a = fmaf(J[r], __shfl_sync(0xffffffffu, v, r, L), a);
            m = fmaf(J[r + 1], __shfl_sync(0xffffffffu, v, r + 1, L), m);
        }
        v = in ? a + m : v;
    };
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c) fetch(c);
    for (int c = 0; c < n_chunk; ++c) {
        copy_wait<kStages - 2>();
        fetch(c + kStages - 1);
        const int lo = n - (c + 1) * C;
        const float* rec = sj[c % kStages][grp];
        if (__all_sync(0xffffffffu, lo >= 0)) {
#pragma unroll
            for (int q = C - 1; q >= 0; --q) step(lo + q, rec + q * R, true);
        } else {
            for (int q = C - 1; q >= 0; --q) step(lo + q, rec + q * R, lo + q >= 0);
        }
    }
    if constexpr (MAP) {
        if (own) *at_map(seg, col) = v;
    } else {
        if (own && seg == 0) carry_out[t * NX + j] = v;
    }
}

// The gradient's data term: every entry of theta is a sum over the samples of
// a product of two of the sample's quantities (a z^T for M_0, p a z^T for M_1,
// d1 z^T for W1, d2 h1^T for W2, ...).  A block takes tiles of kTile samples:
// each thread puts one sample's quantities into shared memory, then each
// entry's threads sum the tile (FP32 in parts of kPart samples, added up in
// FP64).  part[block][q].
template <int NX>
struct Outer {
    using Q = Lay<NX>;
    // rows of the tile: a, p a, d1, d2, s, z, h1, h2, 1
    static constexpr int A = 0, PA = Q::NO, D1 = 2 * Q::NO, D2 = D1 + NH, S = D2 + NH, Z = S + 1, H1 = Z + Q::NZ,
                         H2 = H1 + NH, ONE = H2 + NH, ROWS = ONE + 1;
    static constexpr int kTile = 128, kLd = kTile + 1;   // odd row stride: rows of one column lie in distinct banks
    static constexpr int kThreads = ((Q::N + 31) / 32) * 32 < kTile ? kTile : ((Q::N + 31) / 32) * 32;
    static constexpr int kPart = 32;
};

template <int NX>
__global__ void __launch_bounds__(Outer<NX>::kThreads)
    outer_kernel(const float* __restrict__ theta, const float* __restrict__ u, const float* __restrict__ y,
                 const float* __restrict__ scales, int n_traj, int T, int k0, int len, int ld, float inv_n, int first,
                 const float* __restrict__ xh, const float* __restrict__ lam, double* __restrict__ part)
{
    using Q = Lay<NX>;
    using O = Outer<NX>;
    __shared__ float th[Q::N];
    __shared__ float tile[O::ROWS][O::kLd];
    const int tid = threadIdx.x;
    for (int i = tid; i < Q::N; i += O::kThreads) th[i] = theta[i];
    // the two rows whose product this thread's entry sums
    int ra = O::ONE, rb = O::ONE;
    {
        const int q = tid;
        auto outer = [&](int base, int cols, int r0, int c0) { ra = r0 + (q - base) / cols, rb = c0 + (q - base) % cols; };
        if (q < Q::M1) outer(Q::M0, Q::NZ, O::A, O::Z);
        else if (q < Q::W1) outer(Q::M1, Q::NZ, O::PA, O::Z);
        else if (q < Q::B1) outer(Q::W1, Q::NZ, O::D1, O::Z);
        else if (q < Q::W2) ra = O::D1 + q - Q::B1;
        else if (q < Q::B2) outer(Q::W2, NH, O::D2, O::H1);
        else if (q < Q::W3) ra = O::D2 + q - Q::B2;
        else if (q < Q::B3) ra = O::S, rb = O::H2 + q - Q::W3;
        else if (q == Q::B3) ra = O::S;
    }
    const long long n = (long long)n_traj * len;
    double acc = 0.0;
    for (long long s0 = blockIdx.x * (long long)O::kTile; s0 < n; s0 += (long long)gridDim.x * O::kTile) {
        __syncthreads();
        if (tid < O::kTile) {
            const long long s = s0 + tid;
            float q[O::ROWS];
#pragma unroll
            for (int i = 0; i < O::ROWS; ++i) q[i] = 0.f;
            if (s < n) {
                const size_t t = (size_t)(s / len);
                const int k = (int)(s % len);
                Sample<NX> S;
                const size_t row = (t * T + k0 + k) * 3;
                eval_sample<NX>(th, scales, xh + (t * T + k0 + k) * NX, u + row, y + row, S);
                float a[Q::NO], d2[NH], e[NH];
                load_vec<NX>(lam + (t * ld + k) * NX, a);
#pragma unroll
                for (int c = 0; c < NY; ++c) a[NX + c] = 2.0f * S.res[c] * inv_n;
                float sp = 0.f;  // dJ/dp
#pragma unroll
                for (int r = 0; r < Q::NO; ++r) {
                    float m1z = 0.f;
#pragma unroll
                    for (int j = 0; j < Q::NZ; ++j) m1z = fmaf(th[Q::M1 + r * Q::NZ + j], S.z[j], m1z);
                    sp = fmaf(a[r], m1z, sp);
                    q[O::A + r] = a[r];
                    q[O::PA + r] = S.p * a[r];
                }
                eta_back<NX>(th, S.h1, S.h2, d2, e);
#pragma unroll
                for (int i = 0; i < NH; ++i) {
                    q[O::D1 + i] = sp * e[i];
                    q[O::D2 + i] = sp * d2[i];
                    q[O::H1 + i] = S.h1[i];
                    q[O::H2 + i] = S.h2[i];
                }
                q[O::S] = sp;
                q[O::ONE] = 1.0f;
#pragma unroll
                for (int j = 0; j < Q::NZ; ++j) q[O::Z + j] = S.z[j];
            }
#pragma unroll
            for (int i = 0; i < O::ROWS; ++i) tile[i][tid] = q[i];
        }
        __syncthreads();
        for (int b = 0; b < O::kTile; b += O::kPart) {
            float f = 0.f;
#pragma unroll 8
            for (int i = b; i < b + O::kPart; ++i) f = fmaf(tile[ra][i], tile[rb][i], f);
            acc += (double)f;
        }
    }
    if (tid < Q::N) {
        double* o = part + (size_t)blockIdx.x * Q::N + tid;
        *o = first ? acc : *o + acc;  // windows add up in order
    }
}

// Block q < N: grad[q] = sum of the partials (fixed order) + sigma2 theta[q],
// zero where the stage holds it; block N: loss = sum_sq inv_n + sigma2/2 |theta|^2.
// One warp per block: lane-strided sums, then a shuffle tree.
__global__ void __launch_bounds__(32)
    final_kernel(const double* __restrict__ part, int nblk, const double* __restrict__ loss_part, int nloss, int N,
                 int nx, const float* __restrict__ theta, float sigma2, double inv_n, int stage,
                 double* __restrict__ loss, float* __restrict__ grad)
{
    const int q = (int)blockIdx.x + (grad ? 0 : N), lane = threadIdx.x;  // without a gradient only the loss
    double v = 0.0, t2 = 0.0;
    if (q < N) {
        for (int b = lane; b < nblk; b += 32) v += part[(size_t)b * N + q];
    } else {
        for (int b = lane; b < nloss; b += 32) v += loss_part[b];
        for (int i = lane; i < N; i += 32) t2 += (double)theta[i] * (double)theta[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        v += __shfl_down_sync(0xffffffffu, v, o);
        t2 += __shfl_down_sync(0xffffffffu, t2, o);
    }
    if (lane) return;
    if (q < N) grad[q] = trainable(q, nx, stage) ? (float)(v + (double)sigma2 * (double)theta[q]) : 0.f;
    else *loss = v * inv_n + 0.5 * (double)sigma2 * t2;
}

// ---------------------------------------------------------------------------
// Adam with step rejection (one block, one thread per entry of theta)
// ---------------------------------------------------------------------------
struct AdamDev {
    float *th, *m, *v, *thb, *lr_scale;
    double* acc_loss;
    int* t;
};

__global__ void adam_kernel(AdamDev A, const float* __restrict__ grad, const double* __restrict__ loss,
                            double* __restrict__ hist, int it, int N, float lr)
{
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const int q = threadIdx.x;
    const double L = *loss, La = *A.acc_loss;
    const int t0 = *A.t;
    float sc = *A.lr_scale;
    const bool ok = isfinite(L) && (La < 0.0 || L <= 10.0 * La);
    if (q == 0 && hist) hist[it] = L;
    __syncthreads();
    if (ok) {  // the iterate is accepted: it becomes the fall-back point, then one Adam step
        const int t = t0 + 1;
        if (q < N) {
            A.thb[q] = A.th[q];
            const float g = grad[q];
            const float m = b1 * A.m[q] + (1.0f - b1) * g;
            const float v = b2 * A.v[q] + (1.0f - b2) * g * g;
            A.m[q] = m;
            A.v[q] = v;
            const float mh = m / (1.0f - powf(b1, (float)t)), vh = v / (1.0f - powf(b2, (float)t));
            A.th[q] -= lr * sc * mh / (sqrtf(vh) + eps);
        }
        if (q == 0) {
            *A.t = t;
            *A.acc_loss = L;
        }
    } else if (t0 > 0) {  // back to the fall-back point, the same step at half the size
        sc *= 0.5f;
        if (q < N) {
            const float mh = A.m[q] / (1.0f - powf(b1, (float)t0)), vh = A.v[q] / (1.0f - powf(b2, (float)t0));
            A.th[q] = A.thb[q] - lr * sc * mh / (sqrtf(vh) + eps);
        }
        if (q == 0) *A.lr_scale = sc;
    }
}

// ---------------------------------------------------------------------------
// L-BFGS (one block, one thread per entry of theta; FP64 state)
// ---------------------------------------------------------------------------
constexpr int kLM = 10;   // curvature pairs kept
constexpr int kLT = 320;  // threads: at least n_theta (315 for nx = 8)

struct LbDev {
    double *W, *g, *d, *S, *Y, *rho, *gd;
    int* count;  // [0] pairs held, [1] next slot
    int N;
};

__device__ double block_dot(double v, double* red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < kLT / 32; ++w) t += red[w];
    return t;  // every thread, fixed order
}

// W = theta, g = grad (zero on fixed entries), no pairs.
__global__ void lb_init_kernel(const float* __restrict__ th, const float* __restrict__ grad, LbDev L)
{
    const int i = threadIdx.x;
    L.W[i] = i < L.N ? (double)th[i] : 0.0;
    L.g[i] = i < L.N ? (double)grad[i] : 0.0;
    if (i == 0) L.count[0] = L.count[1] = 0;
}

// d = -H g by the two-loop recursion (newest pair first), H_0 = (s.y / y.y) I
// of the newest pair; d = -g (history cleared) when that is no descent
// direction.  gd[0] = g.d, gd[1] = g.g.
__global__ void lb_dir_kernel(LbDev L)
{
    __shared__ double red[kLT / 32];
    __shared__ double alpha[kLM];
    const int i = threadIdx.x;
    const int n = L.count[0], next = L.count[1];
    double q = L.g[i];
    for (int k = 0; k < n; ++k) {
        const int j = (next - 1 - k + kLM) % kLM;
        const double a = L.rho[j] * block_dot(L.S[j * kLT + i] * q, red);
        if (i == 0) alpha[j] = a;
        q -= a * L.Y[j * kLT + i];
    }
    double gamma = 1.0;
    if (n > 0) {
        const int j = (next - 1 + kLM) % kLM;
        const double yy = block_dot(L.Y[j * kLT + i] * L.Y[j * kLT + i], red);
        gamma = yy > 0.0 ? 1.0 / (L.rho[j] * yy) : 1.0;
    }
    __syncthreads();
    double r = gamma * q;
    for (int k = n - 1; k >= 0; --k) {
        const int j = (next - 1 - k + kLM) % kLM;
        const double b = L.rho[j] * block_dot(L.Y[j * kLT + i] * r, red);
        r += L.S[j * kLT + i] * (alpha[j] - b);
    }
    const double gi = L.g[i];
    const double gd = -block_dot(gi * r, red);
    const double gg = block_dot(gi * gi, red);
    if (gd < 0.0) {
        L.d[i] = -r;
        if (i == 0) L.gd[0] = gd;
    } else {
        L.d[i] = -gi;
        if (i == 0) {
            L.gd[0] = -gg;
            L.count[0] = 0;
        }
    }
    if (i == 0) L.gd[1] = gg;
}

// theta = W + step d (the trial point; fixed entries have d = 0).
__global__ void lb_try_kernel(float* __restrict__ th, LbDev L, double step)
{
    const int i = threadIdx.x;
    if (i < L.N) th[i] = (float)(L.W[i] + step * L.d[i]);
}

// Accepts the trial point: s = step d, y = g_new - g, stored when s.y > 0.
__global__ void lb_accept_kernel(const float* __restrict__ grad, LbDev L, double step)
{
    __shared__ double red[kLT / 32];
    const int i = threadIdx.x;
    const double gn = i < L.N ? (double)grad[i] : 0.0;
    const double s = step * L.d[i], y = gn - L.g[i];
    const double sy = block_dot(s * y, red);
    const double yy = block_dot(y * y, red);
    const int next = L.count[1];
    __syncthreads();
    if (sy > 1e-12 * yy && sy > 0.0) {
        L.S[next * kLT + i] = s;
        L.Y[next * kLT + i] = y;
        if (i == 0) {
            L.rho[next] = 1.0 / sy;
            L.count[0] = min(L.count[0] + 1, kLM);
            L.count[1] = (next + 1) % kLM;
        }
    }
    L.W[i] += s;
    L.g[i] = gn;
}

// ---------------------------------------------------------------------------
// Free run of the augmented model (velocities and positions, physical units)
// ---------------------------------------------------------------------------
template <int NX>
__global__ void predict_kernel(const float* __restrict__ theta, const float* __restrict__ scales,
                               const float* __restrict__ u, int n_traj, int T, float Ts, float* __restrict__ vel,
                               float* __restrict__ pos)
{
    using Q = Lay<NX>;
    __shared__ float th[Q::N];
    for (int i = threadIdx.x; i < Q::N; i += blockDim.x) th[i] = theta[i];
    __syncthreads();
    const int tr = blockIdx.x * blockDim.x + threadIdx.x;
    if (tr >= n_traj) return;
    float isu[NU], sy[NY], x[NX], e[NY] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        isu[c] = 1.0f / scales[c];
        sy[c] = scales[3 + c];
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) x[i] = 0.f;
    for (int k = 0; k < T; ++k) {
        float z[Q::NZ], h1[NH], h2[NH], o[Q::NO];
#pragma unroll
        for (int i = 0; i < NX; ++i) z[i] = x[i];
        const size_t row = ((size_t)tr * T + k) * 3;
#pragma unroll
        for (int c = 0; c < NU; ++c) z[NX + c] = u[row + c] * isu[c];
        const float p = eta<NX>(th, z, h1, h2);
        mz<NX>(th, p, z, o);
#pragma unroll
        for (int c = 0; c < NY; ++c) {
            const float v = o[NX + c] * sy[c];
            if (vel) vel[row + c] = v;
            if (pos) pos[row + c] = e[c];
            e[c] = fmaf(Ts, v, e[c]);
        }
#pragma unroll
        for (int i = 0; i < NX; ++i) x[i] = o[i];
    }
}

// ---------------------------------------------------------------------------
// Closed loop with the PD law of Eq. 28 (one thread per run)
// ---------------------------------------------------------------------------
// Two FP32 FMAs in one instruction, each rounded to nearest.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
        "fma.rn.f32x2 w, x, y, z;\n\tmov.b64 {%0, %1}, w;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// The parameters with the rows of each matrix in pairs, for two FMAs at once.
template <int NX>
struct Pairs {
    using Q = Lay<NX>;
    static constexpr int NP = (Q::NO + 1) / 2;   // row pairs of M_0 and M_1 (the last row's partner is zero)
    float2 m0[Q::NZ][NP], m1[Q::NZ][NP];
    float2 w1[Q::NZ][NH / 2], w2[NH][NH / 2], b1[NH / 2], b2[NH / 2];
    float w3[NH], b3;

    __device__ void load(const float* __restrict__ th, int i0, int di)
    {
        for (int i = i0; i < Q::NZ * 2 * NP; i += di) {
            const int j = i / (2 * NP), r = i % (2 * NP);
            (&m0[j][0].x)[r] = r < Q::NO ? th[Q::M0 + r * Q::NZ + j] : 0.f;
            (&m1[j][0].x)[r] = r < Q::NO ? th[Q::M1 + r * Q::NZ + j] : 0.f;
        }
        for (int i = i0; i < Q::NZ * NH; i += di) (&w1[i / NH][0].x)[i % NH] = th[Q::W1 + (i % NH) * Q::NZ + i / NH];
        for (int i = i0; i < NH * NH; i += di) (&w2[i / NH][0].x)[i % NH] = th[Q::W2 + (i % NH) * NH + i / NH];
        for (int i = i0; i < NH; i += di) {
            (&b1[0].x)[i] = th[Q::B1 + i];
            (&b2[0].x)[i] = th[Q::B2 + i];
            w3[i] = th[Q::W3 + i];
        }
        if (i0 == 0) b3 = th[Q::B3];
    }

    // a = b1 + W1 z over the columns [j0, j1) of z, continuing from a
    __device__ __forceinline__ void layer1(const float* z, int j0, int j1, float2* a) const
    {
#pragma unroll
        for (int j = 0; j < Q::NZ; ++j)
            if (j >= j0 && j < j1)
#pragma unroll
                for (int i = 0; i < NH / 2; ++i) a[i] = fma2(w1[j][i], both(z[j]), a[i]);
    }

    // eta from the first layer's pre-activations (the operations of eta(), in its order)
    __device__ __forceinline__ float rest(const float2* a) const
    {
        float2 c[NH / 2];
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) c[i] = b2[i];
#pragma unroll
        for (int j = 0; j < NH; ++j) {
            const float h = tanhf(j & 1 ? a[j / 2].y : a[j / 2].x);
#pragma unroll
            for (int i = 0; i < NH / 2; ++i) c[i] = fma2(w2[j][i], both(h), c[i]);
        }
        float p = b3;
#pragma unroll
        for (int i = 0; i < NH; ++i) p = fmaf(w3[i], tanhf(i & 1 ? c[i / 2].y : c[i / 2].x), p);
        return p;
    }
};

// One thread per run, one warp per block.  A chunk of kLoopChunk samples of the
// inputs passes through shared memory, copied a chunk ahead by four lanes
// per run (a lane reading its own row touches a line of its own with every
// load), and a chunk of the outputs is written back the same way.  The
// parameters stay in shared memory, so that the kernel keeps its 13.5 warps per
// SM of 65,536 runs resident (in registers they allowed eight).
// 65,536 runs of 600 samples (n_x = 4): 1.79 -> 0.97 ms, 2.3 TB/s; bound by the
// 503 instructions of a warp's sample, of which the 16 tanhf are more than half.
// wide: kWideF, F is 16-byte aligned, so that a sample's two forces are one copy;
// kWideOut, out is 8-byte aligned, so that two values are one store.
// FEW: as long as every block has a scheduler to itself (152 SMs x 4), the
// time is one warp's chain.  Then the parameters are held in registers, and a
// second warp copies the inputs in, converts them, and copies the outputs
// out: 10 runs of 214 samples 110 -> 72 us (n_x 2), 3,000 runs 125 -> 86 (n_x
// 4).  At 25,000 runs, where warps share a scheduler, the 16 warps of the other
// form are the more.
enum { kWideF = 1, kWideOut = 2 };
constexpr int kLoopChunk = 4, kLoopStages = 2;
constexpr int kFewBlocks = 152 * 4;

template <int NX, bool FEW>
__global__ void __launch_bounds__(FEW ? 64 : 32, FEW ? 4 : 16)
    closed_loop_kernel(const float* __restrict__ theta, const float* __restrict__ scales, int B, int T,
                       const double* __restrict__ F, const double* __restrict__ tau, const double* __restrict__ ref,
                       float Ts, float J, float w, float xi, float* __restrict__ out, int wide)
{
    using Q = Lay<NX>;
    constexpr int C = kLoopChunk, NP = Pairs<NX>::NP;
    __shared__ __align__(16) Pairs<NX> P;
    __shared__ __align__(16) double2 sF[kLoopStages][C][32];
    __shared__ double sT[kLoopStages][C][32], sR[kLoopStages][C][32];
    __shared__ __align__(16) float4 sI[FEW ? 2 : 1][FEW ? C : 1][32];  // FEW: the inputs as FP32
    __shared__ __align__(8) float sO[FEW ? 2 : 1][32][C * 6 + 2];  // stride of 26 words: 64-bit accesses of a column meet distinct banks
    const int lane = threadIdx.x & 31, first = blockIdx.x * 32, n_run = min(32, B - first);
    const bool copies = FEW ? threadIdx.x >= 32 : true;  // this warp moves the data
    P.load(theta, threadIdx.x, FEW ? 64 : 32);
    for (int i = threadIdx.x; i < kLoopStages * C * 32; i += blockDim.x) {  // lanes beyond B run on zeros
        (&sF[0][0][0])[i] = make_double2(0.0, 0.0);
        (&sT[0][0][0])[i] = (&sR[0][0][0])[i] = 0.0;
    }
    if (FEW) __syncthreads();
    else __syncwarp();
    float isu[NU], sy[NY], x[NX], e[NY] = {0.f, 0.f, 0.f}, un[NU] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        isu[c] = 1.0f / scales[c];
        sy[c] = scales[3 + c];
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) x[i] = 0.f;
    const float kp = J * w * w, kd = 2.0f * xi * J * w;
    const int n_chunk = (T + C - 1) / C, cs = lane % C;  // this lane copies sample cs of runs lane / C, + 8, ...
    auto fetch = [&](int c) {
        const int k = c * C + cs, st = c % kLoopStages;
        if (k < T) {
#pragma unroll
            for (int r = lane / C; r < 32; r += 32 / C)
                if (r < n_run) {
                    const size_t o = (size_t)(first + r) * T + k;
                    if (wide & kWideF) {
                        copy_async<16>(&sF[st][cs][r], F + 2 * o);
                    } else {
                        copy_async<8>(&sF[st][cs][r].x, F + 2 * o);
                        copy_async<8>(&sF[st][cs][r].y, F + 2 * o + 1);
                    }
                    copy_async<8>(&sT[st][cs][r], tau + o);
                    copy_async<8>(&sR[st][cs][r], ref + o);
                }
        }
        copy_commit();
    };
    auto input = [&](int st, int q) {
        const double2 f = sF[st][q][lane];
        return make_float4((float)f.x, (float)f.y, (float)sT[st][q][lane], (float)sR[st][q][lane]);
    };
    auto convert = [&](int c) {
#pragma unroll
        for (int q = 0; q < C; ++q) sI[c & 1][q][lane] = input(c % kLoopStages, q);
    };
    auto step = [&](const float4& in, int q, float* row) {
        if constexpr (!FEW || NX > 6) asm volatile("" ::: "memory");  // the parameters are read again every step: hoisted out of the loop they spill
        const float Fx = in.x, Fy = in.y, tk = in.z, rk = in.w;
        float z[Q::NZ];
        float2 ax[NH / 2], a[NH / 2];
#pragma unroll
        for (int i = 0; i < NX; ++i) z[i] = x[i];
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) ax[i] = P.b1[i];
        P.layer1(z, 0, NX, ax);  // the state's part, the same for both evaluations of eta
        // the sample: thetadot from the scheduling of the held input
#pragma unroll
        for (int c = 0; c < NU; ++c) z[NX + c] = un[c];
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) a[i] = ax[i];
        P.layer1(z, NX, Q::NZ, a);
        float p = P.rest(a);
        float wd = 0.f;
        constexpr int wr = NX + 2;  // the row of thetadot; its D entries are zero
#pragma unroll
        for (int j = 0; j < NX; ++j)
            wd = fmaf(fmaf(p, wr & 1 ? P.m1[j][wr / 2].y : P.m1[j][wr / 2].x, wr & 1 ? P.m0[j][wr / 2].y : P.m0[j][wr / 2].x),
                      z[j], wd);
        wd *= sy[2];
        const float tc = kp * (rk - e[2]) - kd * wd;
        un[0] = Fx * isu[0];
        un[1] = Fy * isu[1];
        un[2] = (tk + tc) * isu[2];
#pragma unroll
        for (int c = 0; c < NU; ++c) z[NX + c] = un[c];
#pragma unroll
        for (int i = 0; i < NH / 2; ++i) a[i] = ax[i];
        P.layer1(z, NX, Q::NZ, a);
        p = P.rest(a);
        float o[2 * NP];  // (M_0 + p M_1) z, row pairs; the D block is zero
#pragma unroll
        for (int r = 0; r < NP; ++r) {
            float2 s = make_float2(0.f, 0.f);
#pragma unroll
            for (int j = 0; j < Q::NZ; ++j)
                if (j < NX || 2 * r < NX) s = fma2(fma2(both(p), P.m1[j][r], P.m0[j][r]), both(z[j]), s);
            o[2 * r] = s.x;
            o[2 * r + 1] = s.y;
        }
        float v[NY];
#pragma unroll
        for (int c = 0; c < NY; ++c) v[c] = o[NX + c] * sy[c];
        float2* ob = reinterpret_cast<float2*>(row + 6 * q);
        ob[0] = make_float2(e[0], e[1]);
        ob[1] = make_float2(e[2], v[0]);
        ob[2] = make_float2(v[1], v[2]);
#pragma unroll
        for (int c = 0; c < NY; ++c) e[c] = fmaf(Ts, v[c], e[c]);
#pragma unroll
        for (int i = 0; i < NX; ++i) x[i] = o[i];
    };
    // a chunk's samples of each run are 24 n consecutive bytes
    auto write = [&](int c) {
        const int n = min(C, T - c * C);
        const auto& o = sO[FEW ? c & 1 : 0];
        float* ob = out + ((size_t)first * T + c * C) * 6;
        if (n == C && (wide & kWideOut)) {
#pragma unroll 4
            for (int i = lane; i < n_run * (C * 3); i += 32) {
                const int r = i / (C * 3), h = i % (C * 3);
                *reinterpret_cast<float2*>(ob + (size_t)r * T * 6 + 2 * h) = *reinterpret_cast<const float2*>(&o[r][2 * h]);
            }
        } else {
            for (int i = lane; i < n_run * (n * 6); i += 32) {
                const int r = i / (n * 6), h = i % (n * 6);
                ob[(size_t)r * T * 6 + h] = o[r][h];
            }
        }
    };
    static_assert(kLoopStages == 2, "a chunk under way while one is read");
    if (copies) fetch(0);
    if constexpr (FEW) {
        if (copies) {
            copy_wait<0>();
            convert(0);
            fetch(1);
        }
    }
    for (int c = 0; c < n_chunk; ++c) {
        const int n = min(C, T - c * C);
        if constexpr (FEW) {
            __syncthreads();  // chunk c is there, the outputs of the one before are
            if (copies) {
                copy_wait<0>();
                convert(c + 1);
                fetch(c + 2);
                if (c > 0) write(c - 1);
            } else {
                for (int q = 0; q < n; ++q) step(sI[c & 1][q][lane], q, sO[c & 1][lane]);
            }
        } else {
            copy_wait<0>();
            fetch(c + 1);
            for (int q = 0; q < n; ++q) step(input(c % kLoopStages, q), q, sO[0][lane]);
            __syncwarp();
            write(c);
            // the next chunk's copy_wait is the barrier before sO is written again
        }
    }
    if constexpr (FEW) {
        __syncthreads();
        if (copies) write(n_chunk - 1);
    }
}

// ---------------------------------------------------------------------------
// Data scales: root mean square per channel (fixed-order FP64 sums)
// ---------------------------------------------------------------------------
constexpr int kStatBlocks = 152, kStatThreads = 256;

__global__ void stats_kernel(const float* __restrict__ u, const float* __restrict__ y, long long n,
                             double* __restrict__ part)
{
    __shared__ double s[6][kStatThreads];
    double a[6] = {0, 0, 0, 0, 0, 0};
    for (long long i = blockIdx.x * (long long)kStatThreads + threadIdx.x; i < n; i += (long long)gridDim.x * kStatThreads) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double uu = u[3 * i + c], yy = y[3 * i + c];
            a[c] += uu * uu;
            a[3 + c] += yy * yy;
        }
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) s[c][threadIdx.x] = a[c];
    __syncthreads();
    if (threadIdx.x < 6) {
        double t = 0.0;
        for (int i = 0; i < kStatThreads; ++i) t += s[threadIdx.x][i];
        part[blockIdx.x * 6 + threadIdx.x] = t;
    }
}

__global__ void stats_final_kernel(const double* __restrict__ part, int nblk, long long n, float* __restrict__ scales)
{
    const int c = threadIdx.x;
    if (c >= 6) return;
    double t = 0.0;
    for (int b = 0; b < nblk; ++b) t += part[b * 6 + c];
    scales[c] = (float)sqrt(t / (double)n);
}

// ---------------------------------------------------------------------------
// Least-squares LTI start: y_{k+1} = A1 y_k + B1 u_k over all samples
// (normalised), normal equations G = sum phi phi^T, R = sum phi t^T with
// phi = [y_k; u_k], t = y_{k+1}; per-block FP64 partials, fixed-order sums.
// ---------------------------------------------------------------------------
constexpr int kLsThreads = 128;
constexpr int kLsVals = 36 + 18;  // G (6 x 6) and R (6 x 3)

__global__ void ls_gram_kernel(const float* __restrict__ u, const float* __restrict__ y,
                               const float* __restrict__ scales, int n_traj, int T, double* __restrict__ part)
{
    __shared__ double red[kLsThreads];
    double acc[kLsVals];
#pragma unroll
    for (int i = 0; i < kLsVals; ++i) acc[i] = 0.0;
    const long long n = (long long)n_traj * (T - 1);
    for (long long s = blockIdx.x * (long long)kLsThreads + threadIdx.x; s < n; s += (long long)gridDim.x * kLsThreads) {
        const int tr = (int)(s / (T - 1)), k = (int)(s % (T - 1));
        const size_t r0 = ((size_t)tr * T + k) * 3, r1 = r0 + 3;
        double ph[6], t[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ph[c] = (double)y[r0 + c] / (double)scales[3 + c];
            ph[3 + c] = (double)u[r0 + c] / (double)scales[c];
            t[c] = (double)y[r1 + c] / (double)scales[3 + c];
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) {
#pragma unroll
            for (int j = 0; j < 6; ++j) acc[i * 6 + j] = fma(ph[i], ph[j], acc[i * 6 + j]);
#pragma unroll
            for (int c = 0; c < 3; ++c) acc[36 + i * 3 + c] = fma(ph[i], t[c], acc[36 + i * 3 + c]);
        }
    }
    for (int v = 0; v < kLsVals; ++v) {  // block sums in thread order
        red[threadIdx.x] = acc[v];
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int i = 0; i < kLsThreads; ++i) t += red[i];
            part[blockIdx.x * kLsVals + v] = t;
        }
        __syncthreads();
    }
}

// Sums the partials, solves (G + 1e-12 tr(G)/6 I) Theta = R by Cholesky and
// writes theta: A_0 = [[A1, 0], [0, 0]], B_0 = [[B1], [0]], C_0 = [I, 0], the
// rest zero.
template <int NX>
__global__ void ls_solve_kernel(const double* __restrict__ part, int nblk, float* __restrict__ theta,
                                int* __restrict__ status)
{
    using Q = Lay<NX>;
    for (int i = threadIdx.x; i < Q::N; i += blockDim.x) theta[i] = 0.f;
    __syncthreads();
    if (threadIdx.x != 0) return;
    double G[36], R[18];
    for (int v = 0; v < kLsVals; ++v) {
        double t = 0.0;
        for (int b = 0; b < nblk; ++b) t += part[b * kLsVals + v];
        if (v < 36) G[v] = t; else R[v - 36] = t;
    }
    double tr = 0.0;
    for (int i = 0; i < 6; ++i) tr += G[i * 6 + i];
    for (int i = 0; i < 6; ++i) G[i * 6 + i] += 1e-12 * tr / 6.0;
    // Cholesky G = L L^T in place (lower triangle)
    for (int j = 0; j < 6; ++j) {
        double d = G[j * 6 + j];
        for (int k = 0; k < j; ++k) d -= G[j * 6 + k] * G[j * 6 + k];
        if (!(d > 0.0)) {
            *status = 1;
            return;
        }
        d = sqrt(d);
        G[j * 6 + j] = d;
        for (int i = j + 1; i < 6; ++i) {
            double s = G[i * 6 + j];
            for (int k = 0; k < j; ++k) s -= G[i * 6 + k] * G[j * 6 + k];
            G[i * 6 + j] = s / d;
        }
    }
    double X[18];
    for (int c = 0; c < 3; ++c) {  // L z = r, L^T x = z
        double z[6];
        for (int i = 0; i < 6; ++i) {
            double s = R[i * 3 + c];
            for (int k = 0; k < i; ++k) s -= G[i * 6 + k] * z[k];
            z[i] = s / G[i * 6 + i];
        }
        for (int i = 5; i >= 0; --i) {
            double s = z[i];
            for (int k = i + 1; k < 6; ++k) s -= G[k * 6 + i] * X[k * 3 + c];
            X[i * 3 + c] = s / G[i * 6 + i];
        }
    }
    // y_{k+1}[c] = sum_i X[i][c] phi[i]: A1[c][j] = X[j][c], B1[c][j] = X[3 + j][c]
    for (int c = 0; c < 3; ++c) {
        for (int j = 0; j < 3; ++j) {
            theta[Q::M0 + c * Q::NZ + j] = (float)X[j * 3 + c];
            theta[Q::M0 + c * Q::NZ + NX + j] = (float)X[(3 + j) * 3 + c];
        }
        theta[Q::M0 + (NX + c) * Q::NZ + c] = 1.0f;
    }
    *status = 0;
}

}  // namespace slpvk

using namespace slpvk;

struct slpv_model {
    slpv_config cfg{};
    int N = 0;
    float *th = nullptr, *m = nullptr, *v = nullptr, *thb = nullptr, *lr_scale = nullptr, *grad = nullptr;
    float* scales = nullptr;
    double *acc_loss = nullptr, *loss = nullptr;
    int* t = nullptr;
    double *part = nullptr, *loss_part = nullptr;  // block partials of the gradient and the loss
    float *xh = nullptr, *win = nullptr, *carry = nullptr;  // state history; adjoint window; state and adjoint between windows
    size_t xh_cap = 0, win_cap = 0, carry_cap = 0;
    int loss_cap = 0;
    double* spart = nullptr;
    double* lb = nullptr;  // L-BFGS state, allocated on first use
    int* lb_count = nullptr;
};

namespace {

#define SCK(call)                                                                                        \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) return sph::set_last_error(SPH_E_CUDA, (std::string(#call ": ") +        \
                                                                       cudaGetErrorString(e_)).c_str()); \
    } while (0)

int inval(const char* msg) { return sph::set_last_error(SPH_E_INVAL, msg); }

bool nx_ok(int nx) { return nx == 2 || nx == 4 || nx == 6 || nx == 8; }

template <class F>
cudaError_t by_nx(int nx, F&& f)
{
    switch (nx) {
    case 2: return f(std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 8: return f(std::integral_constant<int, 8>{});
    default: return cudaErrorInvalidValue;
    }
}

// Bytes of a window of the time axis: the per-sample buffers of the adjoint
// (NX^2 + 2 NX floats a sample) and, for the loss alone, the states, are
// bounded by this and stay in L2; a fit of a few dozen trajectories is one window.
constexpr size_t kWindowBytes = 64ull << 20;
constexpr int kSampleBlocks = 152 * 8, kOuterBlocks = 152 * 2;

int grow(float** p, size_t* cap, size_t n)
{
    if (n <= *cap) return SPH_OK;
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    if (cudaMalloc(p, n * sizeof(float)) != cudaSuccess)
        return sph::set_last_error(SPH_E_NOMEM, "slpv: workspace allocation failed");
    *cap = n;
    return SPH_OK;
}

int blocks_for(long long n, int per, int most) { return (int)std::min<long long>((n + per - 1) / per, most); }

// Launches the loss (and gradient) into m->loss / grad_out.
int loss_grad_launch(slpv_model* m, const float* u, const float* y, int n_traj, int T, int stage, float* grad_out,
                     cudaStream_t st)
{
    const bool want = grad_out != nullptr;
    const int nx = m->cfg.nx;
    const size_t per = want ? (size_t)(nx * nx + nx + 3) / 4 * 4 + nx : (size_t)nx;  // floats of a sample in the window
    const int W = (int)std::min<size_t>((size_t)T, std::max<size_t>(kWindowBytes / 4 / per / (size_t)n_traj, 16));
    int rc = grow(&m->win, &m->win_cap, (size_t)n_traj * W * per);
    // The adjoint in segments of 64 samples and more, at most 32, while their
    // maps are few enough to run at once; fewer than 4 do not pay for the maps
    // (4 cut the time to about a half).
    const int seg_most = std::min({W / 64, 32, 6144 / std::max(1, std::min(n_traj, 6144) * (nx + 1))});
    const int n_seg_most = want && seg_most >= 4 ? seg_most : 1;
    // state and adjoint between windows (the adjoint's read and written in turn), the maps
    const size_t maps = (size_t)n_traj * n_seg_most * (nx + 1) * nx;
    if (!rc) rc = grow(&m->carry, &m->carry_cap, 3 * (size_t)n_traj * nx + (n_seg_most > 1 ? maps : 0));
    if (!rc && want) rc = grow(&m->xh, &m->xh_cap, (size_t)n_traj * T * nx);
    if (rc) return rc;
    const double inv_nd = 1.0 / ((double)n_traj * T);
    const float inv_n = (float)inv_nd;
    const int n_win = (T + W - 1) / W;
    const int sblk = blocks_for((long long)n_traj * W, kSampleThreads, kSampleBlocks);
    if (n_win * (long long)sblk > (long long)m->loss_cap) {
        cudaFree(m->loss_part);
        m->loss_part = nullptr;
        m->loss_cap = 0;
        SCK(cudaMalloc(&m->loss_part, (size_t)n_win * sblk * sizeof(double)));
        m->loss_cap = n_win * sblk;
    }
    int oblk = 0, n_loss = 0;
    cudaError_t e = by_nx(nx, [&](auto c) {
        constexpr int NX = decltype(c)::value;
        const int sgrid = (n_traj * kLanes<NX> + 31) / 32;
        float* lam = m->win + (size_t)n_traj * W * kRec<NX>;
        auto sample = [&](int w, const float* xh, int xld, int xk0) {
            const int k0 = w * W, len = std::min(W, T - k0);
            const int nb = blocks_for((long long)n_traj * len, kSampleThreads, kSampleBlocks);
            sample_kernel<NX><<<nb, kSampleThreads, 0, st>>>(m->th, u, y, m->scales, n_traj, T, k0, len, W, xld, xk0,
                                                             inv_n, want ? 1 : 0, xh, m->win, m->loss_part + n_loss);
            n_loss += nb;
        };
        if (!want) {  // the states of a window at a time
            for (int w = 0; w < n_win; ++w) {
                const int k0 = w * W;
                state_kernel<NX><<<sgrid, 32, 0, st>>>(m->th, u, m->scales, n_traj, T, k0, std::min(W, T - k0), W,
                                                       m->carry, m->win);
                sample(w, m->win, W, k0);
            }
            return cudaGetLastError();
        }
        state_kernel<NX><<<sgrid, 32, 0, st>>>(m->th, u, m->scales, n_traj, T, 0, T, T, m->carry, m->xh);
        oblk = blocks_for((long long)n_traj * W, Outer<NX>::kTile, kOuterBlocks);
        for (int w = n_win - 1; w >= 0; --w) {
            const int k0 = w * W, len = std::min(W, T - k0), first = w == n_win - 1 ? 1 : 0;
            sample(w, m->xh, T, 0);
            const int want_len = (len + n_seg_most - 1) / n_seg_most;
            const int seg_len = n_seg_most > 1 ? (want_len + kAdjChunk<NX> - 1) / kAdjChunk<NX> * kAdjChunk<NX> : len;
            const int n_seg = (len + seg_len - 1) / seg_len;
            float* carry[2] = {m->carry + (size_t)n_traj * NX, m->carry + 2 * (size_t)n_traj * NX};
            float* map = m->carry + 3 * (size_t)n_traj * NX;
            auto blocks = [&](long long groups) { return (unsigned)((groups * kLanes<NX> + 31) / 32); };
            if (n_seg > 1)
                adjoint_kernel<NX, true><<<blocks((long long)n_traj * (n_seg - 1) * (NX + 1)), 32, 0, st>>>(
                    m->win, n_traj, len, W, n_seg, seg_len, first, nullptr, nullptr, map, nullptr);
            adjoint_kernel<NX, false><<<blocks((long long)n_traj * n_seg), 32, 0, st>>>(
                m->win, n_traj, len, W, n_seg, seg_len, first, carry[(w + 1) & 1], carry[w & 1], map, lam);
            outer_kernel<NX><<<oblk, Outer<NX>::kThreads, 0, st>>>(m->th, u, y, m->scales, n_traj, T, k0, len, W, inv_n,
                                                                   first, m->xh, lam, m->part);
        }
        return cudaGetLastError();
    });
    SCK(e);
    final_kernel<<<want ? m->N + 1 : 1, 32, 0, st>>>(m->part, oblk, m->loss_part, n_loss, m->N, nx, m->th,
                                                     m->cfg.sigma2, inv_nd, stage, m->loss, grad_out);
    SCK(cudaGetLastError());
    return SPH_OK;
}

int check_data(const slpv_model* m, const void* u, int n_traj, int T)
{
    if (!m || !u || n_traj < 1 || T < 1) return inval("slpv: NULL pointer or empty data");
    return SPH_OK;
}

}  // namespace

extern "C" {

int slpv_n_params(int32_t nx, int32_t* n_theta)
{
    if (!n_theta || !nx_ok(nx)) return inval("slpv_n_params: nx must be 2, 4, 6 or 8");
    *n_theta = n_params(nx);
    return SPH_OK;
}

int slpv_destroy(slpv_model* m)
{
    if (!m) return SPH_OK;
    cudaFree(m->th);
    cudaFree(m->m);
    cudaFree(m->v);
    cudaFree(m->thb);
    cudaFree(m->lr_scale);
    cudaFree(m->grad);
    cudaFree(m->scales);
    cudaFree(m->acc_loss);
    cudaFree(m->loss);
    cudaFree(m->t);
    cudaFree(m->part);
    cudaFree(m->loss_part);
    cudaFree(m->xh);
    cudaFree(m->win);
    cudaFree(m->carry);
    cudaFree(m->spart);
    cudaFree(m->lb);
    cudaFree(m->lb_count);
    delete m;
    return SPH_OK;
}

int slpv_create(const slpv_config* cfg, slpv_model** out)
{
    if (!cfg || !out) return inval("slpv_create: NULL pointer");
    *out = nullptr;
    if (!nx_ok(cfg->nx) || !(cfg->sigma2 >= 0.0f)) return inval("slpv_create: nx must be 2, 4, 6 or 8, sigma2 >= 0");
    slpv_model* m = new slpv_model;
    m->cfg = *cfg;
    m->N = n_params(cfg->nx);
    const size_t nb = (size_t)m->N * sizeof(float);
    bool ok = cudaMalloc(&m->th, nb) == cudaSuccess && cudaMalloc(&m->m, nb) == cudaSuccess &&
              cudaMalloc(&m->v, nb) == cudaSuccess && cudaMalloc(&m->thb, nb) == cudaSuccess &&
              cudaMalloc(&m->grad, nb) == cudaSuccess && cudaMalloc(&m->lr_scale, sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->scales, 6 * sizeof(float)) == cudaSuccess &&
              cudaMalloc(&m->acc_loss, sizeof(double)) == cudaSuccess &&
              cudaMalloc(&m->loss, sizeof(double)) == cudaSuccess && cudaMalloc(&m->t, sizeof(int)) == cudaSuccess &&
              cudaMalloc(&m->spart, kStatBlocks * 6 * sizeof(double)) == cudaSuccess &&
              cudaMalloc(&m->part, (size_t)kOuterBlocks * m->N * sizeof(double)) == cudaSuccess;
    if (!ok) {
        slpv_destroy(m);
        return sph::set_last_error(SPH_E_NOMEM, "slpv_create: cudaMalloc failed");
    }
    const float one[6] = {1, 1, 1, 1, 1, 1};
    if (cudaMemset(m->th, 0, nb) != cudaSuccess ||
        cudaMemcpy(m->scales, one, sizeof(one), cudaMemcpyHostToDevice) != cudaSuccess) {
        slpv_destroy(m);
        return sph::set_last_error(SPH_E_CUDA, "slpv_create: initialisation failed");
    }
    *out = m;
    return SPH_OK;
}

int slpv_set_params(slpv_model* m, const float* theta, const float* scales)
{
    if (!m) return inval("slpv_set_params: NULL model");
    if (theta) {
        std::vector<float> h(theta, theta + m->N);
        for (int q = 0; q < m->N; ++q)
            if (q < 2 * (m->cfg.nx + NY) * (m->cfg.nx + NU) && !trainable(q, m->cfg.nx, kStageAll)) h[q] = 0.f;
        SCK(cudaMemcpy(m->th, h.data(), m->N * sizeof(float), cudaMemcpyHostToDevice));
    }
    if (scales) {
        for (int c = 0; c < 6; ++c)
            if (!(scales[c] > 0.0f) || !std::isfinite(scales[c])) return inval("slpv_set_params: scales must be > 0");
        SCK(cudaMemcpy(m->scales, scales, 6 * sizeof(float), cudaMemcpyHostToDevice));
    }
    return SPH_OK;
}

int slpv_get_params(const slpv_model* m, float* theta, float* scales)
{
    if (!m) return inval("slpv_get_params: NULL model");
    if (theta) SCK(cudaMemcpy(theta, m->th, m->N * sizeof(float), cudaMemcpyDeviceToHost));
    if (scales) SCK(cudaMemcpy(scales, m->scales, 6 * sizeof(float), cudaMemcpyDeviceToHost));
    return SPH_OK;
}

int slpv_normalize(slpv_model* m, const float* u, const float* y, int32_t n_traj, int32_t T, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!y) return inval("slpv_normalize: NULL y");
    cudaStream_t st = (cudaStream_t)stream;
    const long long n = (long long)n_traj * T;
    stats_kernel<<<kStatBlocks, kStatThreads, 0, st>>>(u, y, n, m->spart);
    stats_final_kernel<<<1, 32, 0, st>>>(m->spart, kStatBlocks, n, m->scales);
    SCK(cudaGetLastError());
    float h[6];
    SCK(cudaMemcpyAsync(h, m->scales, sizeof(h), cudaMemcpyDeviceToHost, st));
    SCK(cudaStreamSynchronize(st));
    for (int c = 0; c < 6; ++c)
        if (!(h[c] > 0.0f) || !std::isfinite(h[c])) return inval("slpv_normalize: a channel is identically zero");
    return SPH_OK;
}

int slpv_loss_grad(slpv_model* m, const float* u, const float* y, int32_t n_traj, int32_t T, int32_t stage,
                   double* loss_out, float* grad_out, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!y || !loss_out) return inval("slpv_loss_grad: NULL y or loss_out");
    if (stage < 0 || stage > 2) return inval("slpv_loss_grad: stage must be 0, 1 or 2");
    cudaStream_t st = (cudaStream_t)stream;
    rc = loss_grad_launch(m, u, y, n_traj, T, stage, grad_out, st);
    if (rc) return rc;
    SCK(cudaMemcpyAsync(loss_out, m->loss, sizeof(double), cudaMemcpyDeviceToDevice, st));
    return SPH_OK;
}

int slpv_train(slpv_model* m, const float* u, const float* y, int32_t n_traj, int32_t T, int32_t iters, float lr,
               int32_t stage, double* loss_hist, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!y || iters < 0 || !(lr > 0.0f)) return inval("slpv_train: NULL y, iters < 0 or lr <= 0");
    if (stage < 0 || stage > 2) return inval("slpv_train: stage must be 0, 1 or 2");
    cudaStream_t st = (cudaStream_t)stream;
    const size_t nb = (size_t)m->N * sizeof(float);
    const float one = 1.0f;
    const double neg = -1.0;
    SCK(cudaMemsetAsync(m->m, 0, nb, st));
    SCK(cudaMemsetAsync(m->v, 0, nb, st));
    SCK(cudaMemsetAsync(m->t, 0, sizeof(int), st));
    SCK(cudaMemcpyAsync(m->thb, m->th, nb, cudaMemcpyDeviceToDevice, st));
    SCK(cudaMemcpyAsync(m->lr_scale, &one, sizeof(float), cudaMemcpyHostToDevice, st));
    SCK(cudaMemcpyAsync(m->acc_loss, &neg, sizeof(double), cudaMemcpyHostToDevice, st));
    const int threads = ((m->N + 31) / 32) * 32;
    AdamDev A{m->th, m->m, m->v, m->thb, m->lr_scale, m->acc_loss, m->t};
    for (int it = 0; it < iters; ++it) {
        rc = loss_grad_launch(m, u, y, n_traj, T, stage, m->grad, st);
        if (rc) return rc;
        adam_kernel<<<1, threads, 0, st>>>(A, m->grad, m->loss, loss_hist, it, m->N, lr);
        SCK(cudaGetLastError());
    }
    // end on the last accepted iterate
    SCK(cudaMemcpyAsync(m->th, m->thb, nb, cudaMemcpyDeviceToDevice, st));
    return SPH_OK;
}

int slpv_lbfgs(slpv_model* m, const float* u, const float* y, int32_t n_traj, int32_t T, int32_t iters,
               int32_t stage, double* loss_hist, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!y || iters < 0) return inval("slpv_lbfgs: NULL y or iters < 0");
    if (stage < 0 || stage > 2) return inval("slpv_lbfgs: stage must be 0, 1 or 2");
    cudaStream_t st = (cudaStream_t)stream;
    if (!m->lb) {
        const size_t n = (size_t)kLT * (3 + 2 * kLM) + kLM + 2;
        if (cudaMalloc(&m->lb, n * sizeof(double)) != cudaSuccess || cudaMalloc(&m->lb_count, 2 * sizeof(int)) != cudaSuccess)
            return sph::set_last_error(SPH_E_NOMEM, "slpv_lbfgs: cudaMalloc failed");
        SCK(cudaMemset(m->lb, 0, n * sizeof(double)));
    }
    LbDev L;
    L.W = m->lb;
    L.g = L.W + kLT;
    L.d = L.g + kLT;
    L.S = L.d + kLT;
    L.Y = L.S + (size_t)kLM * kLT;
    L.rho = L.Y + (size_t)kLM * kLT;
    L.gd = L.rho + kLM;
    L.count = m->lb_count;
    L.N = m->N;
    auto eval = [&](bool grad, double* f) -> int {
        int r = loss_grad_launch(m, u, y, n_traj, T, stage, grad ? m->grad : nullptr, st);
        if (r) return r;
        SCK(cudaMemcpyAsync(f, m->loss, sizeof(double), cudaMemcpyDeviceToHost, st));
        SCK(cudaStreamSynchronize(st));
        return SPH_OK;
    };
    double f = 0.0;
    if ((rc = eval(true, &f))) return rc;
    if (!std::isfinite(f)) return sph::set_last_error(SPH_E_DIVERGED, "slpv_lbfgs: the loss at the start is not finite");
    lb_init_kernel<<<1, kLT, 0, st>>>(m->th, m->grad, L);
    SCK(cudaGetLastError());
    constexpr double kArmijo = 1e-4;
    int it = 0;
    for (; it < iters; ++it) {
        lb_dir_kernel<<<1, kLT, 0, st>>>(L);
        SCK(cudaGetLastError());
        double gd[2];
        int cnt[2];
        SCK(cudaMemcpyAsync(gd, L.gd, sizeof(gd), cudaMemcpyDeviceToHost, st));
        SCK(cudaMemcpyAsync(cnt, L.count, sizeof(cnt), cudaMemcpyDeviceToHost, st));
        SCK(cudaStreamSynchronize(st));
        if (!(gd[0] < 0.0)) break;  // stationary
        double step = cnt[0] > 0 ? 1.0 : std::min(1.0, 0.01 / std::sqrt(gd[1]));  // after a reset: 0.01 in theta
        bool ok = false;
        double fn = 0.0;
        for (int tries = 0; tries < 40; ++tries) {
            lb_try_kernel<<<1, kLT, 0, st>>>(m->th, L, step);
            SCK(cudaGetLastError());
            if ((rc = eval(false, &fn))) return rc;
            if (std::isfinite(fn) && fn <= f + kArmijo * step * gd[0]) {
                ok = true;
                break;
            }
            step *= 0.5;
        }
        if (!ok) {  // no decrease along d: back to the last accepted point
            lb_try_kernel<<<1, kLT, 0, st>>>(m->th, L, 0.0);
            SCK(cudaGetLastError());
            break;
        }
        if ((rc = eval(true, &fn))) return rc;
        lb_accept_kernel<<<1, kLT, 0, st>>>(m->grad, L, step);
        SCK(cudaGetLastError());
        f = fn;
        if (loss_hist) loss_hist[it] = f;
    }
    if (loss_hist)
        for (int k = it; k < iters; ++k) loss_hist[k] = f;
    SCK(cudaStreamSynchronize(st));
    return SPH_OK;
}

int slpv_init_ls(slpv_model* m, const float* u, const float* y, int32_t n_traj, int32_t T, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!y || T < 2) return inval("slpv_init_ls: NULL y or T < 2");
    if (m->cfg.nx < 3) return inval("slpv_init_ls: the start needs nx >= 3 (the velocities are states)");
    cudaStream_t st = (cudaStream_t)stream;
    constexpr int nblk = 152;
    double* part = nullptr;
    int* status = nullptr;
    SCK(cudaMalloc(&part, (size_t)nblk * kLsVals * sizeof(double)));
    cudaError_t e = cudaMalloc(&status, sizeof(int));
    if (e != cudaSuccess) {
        cudaFree(part);
        return sph::set_last_error(SPH_E_NOMEM, "slpv_init_ls: cudaMalloc failed");
    }
    ls_gram_kernel<<<nblk, kLsThreads, 0, st>>>(u, y, m->scales, n_traj, T, part);
    e = by_nx(m->cfg.nx, [&](auto c) {
        constexpr int NX = decltype(c)::value;
        ls_solve_kernel<NX><<<1, 128, 0, st>>>(part, nblk, m->th, status);
        return cudaGetLastError();
    });
    int hs = 1;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hs, status, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(part);
    cudaFree(status);
    SCK(e);
    if (hs != 0) return sph::set_last_error(SPH_E_DIVERGED, "slpv_init_ls: the normal equations are singular");
    return SPH_OK;
}

int slpv_predict(const slpv_model* m, const float* u, int32_t n_traj, int32_t T, double Ts, float* vel_out,
                 float* pos_out, void* stream)
{
    int rc = check_data(m, u, n_traj, T);
    if (rc) return rc;
    if (!(Ts > 0.0)) return inval("slpv_predict: Ts must be > 0");
    cudaStream_t st = (cudaStream_t)stream;
    const int threads = 128, blocks = (n_traj + threads - 1) / threads;
    SCK(by_nx(m->cfg.nx, [&](auto c) {
        constexpr int NX = decltype(c)::value;
        predict_kernel<NX><<<blocks, threads, 0, st>>>(m->th, m->scales, u, n_traj, T, (float)Ts, vel_out, pos_out);
        return cudaGetLastError();
    }));
    return SPH_OK;
}

int slpv_simulate(const slpv_model* m, int32_t B, int32_t T, const double* F, const double* tau,
                  const double* theta_ref, double Ts, double J, double omega, double xi, float* out, void* stream)
{
    if (!m || !F || !tau || !theta_ref || !out || B < 1 || T < 1) return inval("slpv_simulate: NULL pointer or empty");
    if (!(Ts > 0.0) || !(J > 0.0)) return inval("slpv_simulate: Ts and J must be > 0");
    cudaStream_t st = (cudaStream_t)stream;
    const int wide = ((reinterpret_cast<uintptr_t>(F) & 15) == 0 ? kWideF : 0) |
                     ((reinterpret_cast<uintptr_t>(out) & 7) == 0 ? kWideOut : 0);
    SCK(by_nx(m->cfg.nx, [&](auto c) {
        constexpr int NX = decltype(c)::value;
        auto go = [&](auto kernel, int threads) {
            kernel<<<(B + 31) / 32, threads, 0, st>>>(m->th, m->scales, B, T, F, tau, theta_ref, (float)Ts, (float)J,
                                                      (float)omega, (float)xi, out, wide);
        };
        if ((B + 31) / 32 <= kFewBlocks) go(closed_loop_kernel<NX, true>, 64);
        else go(closed_loop_kernel<NX, false>, 32);
        return cudaGetLastError();
    }));
    return SPH_OK;
}

}  // extern "C"
