// lpv_kernels.cu -- tensor-core kernels of the LPV surrogate (Section 4).
//
// One warp carries 16 (or 8) trajectories through the recurrence
//     [x_{k+1}; y_k] = W w_k,   w_k = [z_k; p_1 z_k; p_2 z_k],  z_k = [x_k; u_k; 0]
// as one mma.sync.m16n8k16 (BF16 in, FP32 accumulate) product per 16x16x8
// tile.  Each operand is split into two BF16 halves (v = hi + lo) and the
// product is hi*hi + hi*lo + lo*hi, which keeps about 16 significant bits
// per half: a recurrent state rounded to plain BF16 every step would drift.
//
// Register layouts (PTX m16n8k16, groupID g = lane / 4, t = lane % 4):
//   A 16x16: rows g, g+8; columns 2t, 2t+1, 2t+8, 2t+9
//   D 16x8 : rows g, g+8; columns 2t, 2t+1 (of the n-tile)
// With features ordered [x (n_x), u (n_u), 0...] in each 16-column block and
// outputs ordered [x_next (n_x), y (n_y), 0...], the accumulator of n-tiles
// 0 and 1 holds exactly the entries of the next step's first A block that
// this thread owns, and the scheduled blocks p_i z are thread-local scalings:
// the recurrence runs without shuffles.  The adjoint uses the same identity;
// the weight gradient sum_k G_k^T w_k is one more MMA, in
// warps of its own, whose operands are transposed in registers.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstddef>
#include <cstdint>
#include <type_traits>

#include "lpv_common.cuh"
#include "lpv_launch.h"

namespace lpv {

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1)
{
    asm(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// The same with a zero accumulator.
__device__ __forceinline__ void mma16816_0(float* d, const uint32_t* a, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// Two FP32 operations in one instruction, each rounded to nearest.
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tsub.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 r;
    asm("{.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 z, x, y;\n\t"
        "mov.b64 {%0, %1}, z;}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
    return r;
}

// (v0, v1) -> packed bf16x2 (v0 in the low half), split into hi and lo parts.
__device__ __forceinline__ void split2(float v0, float v1, uint32_t& hi, uint32_t& lo)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(v0, v1);
    hi = *reinterpret_cast<const uint32_t*>(&h);
    const float2 r = sub2(make_float2(v0, v1), make_float2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u)));
    const __nv_bfloat162 l = __floats2bfloat162_rn(r.x, r.y);
    lo = *reinterpret_cast<const uint32_t*>(&l);
}

// B fragments of the forward product D[row][o] = sum_f w[row][f] Wp[o][f].
__device__ __forceinline__ void load_fwd_frags(const float* __restrict__ Wp, uint32_t (*bhi)[2][2],
                                               uint32_t (*blo)[2][2], int nkt, int g, int t)
{
#pragma unroll
    for (int kt = 0; kt < kMaxKT; ++kt) {
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const float* w = Wp + (nt * 8 + g) * (kFB * kMaxKT) + kt * kFB;
            if (kt < nkt) {
                split2(w[2 * t], w[2 * t + 1], bhi[kt][nt][0], blo[kt][nt][0]);
                split2(w[8 + 2 * t], w[9 + 2 * t], bhi[kt][nt][1], blo[kt][nt][1]);
            } else {
                bhi[kt][nt][0] = bhi[kt][nt][1] = blo[kt][nt][0] = blo[kt][nt][1] = 0u;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// The free run and its gradient.
//
// Serial in k are the state and its adjoint, each a product of the split
// operands per step; everything else runs beside or after them:
//   fwd_kernel     the free run: x_k and the residuals for the adjoint
//   adj_kernel     lambda_k and, in other warps, sum_k G_k^T w_k with
//                  G_k = [lambda_{k+1}; dJ/dy_k]
// The serial passes are bound by the instructions of one warp's step, which
// nothing else overlaps: few warps per block (a fit's few dozen blocks each
// get an SM of their own), the inputs laid out in shared memory as the lanes hold
// them, the number of scheduling blocks and whether the lower columns are all
// state known at compile time.  RG is the number of 8-trajectory row groups
// of a warp, 2 filling the product's 16 rows; with 1 half the rows are idle,
// but so is half of the work per step around the product, and a step is
// shorter.  Runs that leave schedulers idle anyway take RG = 1
// (row_groups).  820 trajectories of 1,000 samples (n_x 12, n_u 3, n_y 4,
// n_p 2): 175 us forward, 173 us adjoint and gradient, 6 us reduction.  Four
// warps to a block that loaded u, y and p from their rows (28 memory
// instructions of up to 16 lines a step) and kept the weight gradient, with
// its transposes through shared memory, on the adjoint's chain took 1,939 +
// 1,469 + 31 us.
//
// What the free run leaves for the adjoint is a row of 16 floats per trajectory
// and step, hist[traj][k]: the state in the first n_x columns, the residuals'
// part of G_k after it, the columns in the lanes' order (2t, 2t+1, 2t+8, 2t+9
// at place 4t).  (As two fragments of 8 rows, z_k and G_k, it took twice the
// room, 32 times for one trajectory, in the same time.)
// ---------------------------------------------------------------------------
constexpr int kC = 4;         // steps per chunk of staged inputs
constexpr int kStages = 4;    // chunks in shared memory: one in use, three in flight
constexpr int kFrag = 128;    // floats of a step of 8 trajectories, [lane][4]

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

// Staged channels of a step: column c of a row at its place (from column 8 on
// when the columns below are all state, n_x >= 8; all 16 when LOW), zero where
// no channel lies; and the scheduling of a row.  Rows are apart so that the
// eight of a warp read distinct banks.
template <bool LOW>
constexpr int kFirstCol = LOW ? 0 : 8;

template <bool LOW>
__device__ __forceinline__ void load_vals(const float* row, int t, float* v)  // columns 2t, 2t+1, 2t+8, 2t+9
{
    const float2 b = *reinterpret_cast<const float2*>(row + 8 - kFirstCol<LOW> + 2 * t);
    float2 a = make_float2(0.f, 0.f);
    if (LOW) a = *reinterpret_cast<const float2*>(row + 2 * t);
    v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}

// One stage of a warp's inputs.
template <bool LOW, int RG>
struct InStage {
    float u[kC][RG][8][16 - kFirstCol<LOW>];
    float y[kC][RG][8][16 - kFirstCol<LOW>];
    float p[kC][RG][8][2];
};

// A row's n channels to consecutive places.
__device__ __forceinline__ void copy_row(float* dst, const float* src, int n)
{
#pragma unroll 4
    for (int j = 0; j < n; ++j) copy_async<4>(dst + j, src + j);
}

// D = [z; p_1 z; ...] W^T for RG row groups: z[i] of column i, row group
// (i >> 1) & 1, and the normalised scheduling pp of each row.
template <int NP, int RG>
__device__ __forceinline__ void product(float* D, const float* z, const float (*pp)[2], const uint32_t (*bhi)[2][2],
                                        const uint32_t (*blo)[2][2])
{
    if constexpr (RG == 1) {
        // the idle rows 8-15 take the low parts: one product gives hi.hi and
        // lo.hi, the other hi.lo (and lo.lo, not used)
        uint32_t a[1 + NP][4];
        float c1[8];
#pragma unroll
        for (int kt = 0; kt <= NP; ++kt) {
            float2 v0 = make_float2(z[0], z[1]), v1 = make_float2(z[4], z[5]);
            if (kt) {
                const float2 f = make_float2(pp[0][kt ? kt - 1 : 0], pp[0][kt ? kt - 1 : 0]);
                v0 = mul2(v0, f);
                v1 = mul2(v1, f);
            }
            split2(v0.x, v0.y, a[kt][0], a[kt][1]);
            split2(v1.x, v1.y, a[kt][2], a[kt][3]);
        }
#pragma unroll
        for (int kt = 0; kt <= NP; ++kt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                auto mma = [kt](float* c, const uint32_t* x, uint32_t b0, uint32_t b1) {
                    if (kt) mma16816(c, x, b0, b1);
                    else mma16816_0(c, x, b0, b1);
                };
                mma(D + 4 * nt, a[kt], bhi[kt][nt][0], bhi[kt][nt][1]);
                mma(c1 + 4 * nt, a[kt], blo[kt][nt][0], blo[kt][nt][1]);
            }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const float2 e = add2(make_float2(c1[4 * nt], c1[4 * nt + 1]), make_float2(D[4 * nt + 2], D[4 * nt + 3]));
            const float2 f = add2(make_float2(D[4 * nt], D[4 * nt + 1]), e);
            D[4 * nt] = f.x;
            D[4 * nt + 1] = f.y;
        }
    } else {
        // three independent accumulation chains (hi.hi, hi.lo, lo.hi) over the k-tiles
        uint32_t ahi[1 + NP][4], alo[1 + NP][4];
#pragma unroll
        for (int kt = 0; kt <= NP; ++kt)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float2 v = make_float2(z[2 * i], z[2 * i + 1]);
                if (kt) {
                    const float f = pp[i & 1][kt ? kt - 1 : 0];
                    v = mul2(v, make_float2(f, f));
                }
                split2(v.x, v.y, ahi[kt][i], alo[kt][i]);
            }
        float c1[8], c2[8];
#pragma unroll
        for (int kt = 0; kt <= NP; ++kt)
#pragma unroll
            for (int nt = 0; nt < 2; ++nt) {
                auto mma = [kt](float* c, const uint32_t* x, uint32_t b0, uint32_t b1) {
                    if (kt) mma16816(c, x, b0, b1);
                    else mma16816_0(c, x, b0, b1);
                };
                mma(D + 4 * nt, ahi[kt], bhi[kt][nt][0], bhi[kt][nt][1]);
                mma(c1 + 4 * nt, ahi[kt], blo[kt][nt][0], blo[kt][nt][1]);
                mma(c2 + 4 * nt, alo[kt], bhi[kt][nt][0], bhi[kt][nt][1]);
            }
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const float2 f = add2(make_float2(D[i], D[i + 1]), add2(make_float2(c1[i], c1[i + 1]), make_float2(c2[i], c2[i + 1])));
            D[i] = f.x;
            D[i + 1] = f.y;
        }
    }
}

// Free-run simulation of 8 RG trajectories per warp.  MODE 0 writes the
// prediction (physical units); MODE 1 accumulates the squared error of the
// normalised outputs and records x_k and the residuals' part of G_k.
template <int MODE, bool LOW, int NP, int RG>
__global__ void __launch_bounds__(32) fwd_kernel(const float* __restrict__ Wp, Dims d, const float* __restrict__ u,
                                                 const float* __restrict__ p, const float* __restrict__ y, int n_traj,
                                                 int T, float* __restrict__ y_out, float* __restrict__ hist,
                                                 double* __restrict__ loss_part, float grad_scale)
{
    __shared__ __align__(16) InStage<LOW, RG> sm[kStages];
    const int lane = threadIdx.x, g = lane >> 2, t = lane & 3, wid = blockIdx.x, first = wid * 8 * RG;
    {   // rows beyond the data and places without a channel stay zero
        float* z = reinterpret_cast<float*>(sm);
        for (int i = lane; i < (int)(sizeof(sm) / sizeof(float)); i += 32) z[i] = 0.f;
        __syncwarp();
    }
    uint32_t bhi[kMaxKT][2][2], blo[kMaxKT][2][2];
    load_fwd_frags(Wp, bhi, blo, 1 + NP, g, t);
    bool is_x[4], is_y[RG][4];
    float fu[4], fy[4], pm[2], ips[RG][2];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = 8 * (j >> 1) + 2 * t + (j & 1), q = c - d.nx;
        is_x[j] = q < 0;
        fu[j] = q >= 0 && q < d.nu ? d.inv_su[q] : 0.f;
        fy[j] = MODE == 0 ? (q >= 0 && q < d.ny ? d.sy[q] : 0.f) : (q >= 0 && q < d.ny ? d.inv_sy[q] : 0.f);
#pragma unroll
        for (int r = 0; r < RG; ++r) is_y[r][j] = q >= 0 && q < d.ny && first + 8 * r + g < n_traj;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        pm[j] = j < NP ? d.pm[j] : 0.f;
#pragma unroll
        for (int r = 0; r < RG; ++r) ips[r][j] = j < NP && first + 8 * r + g < n_traj ? d.inv_ps[j] : 0.f;
    }
    // the four lanes of a row copy the four steps of its chunk
    const int n_chunk = (T + kC - 1) / kC;
    auto fetch = [&](int c) {
        const int k = c * kC + t;
        if (k < T) {
            InStage<LOW, RG>& S = sm[c % kStages];
#pragma unroll
            for (int r = 0; r < RG; ++r) {
                const int tr = first + 8 * r + g;
                if (tr < n_traj) {
                    const size_t row = (size_t)tr * T + k;
                    copy_row(&S.u[t][r][g][d.nx - kFirstCol<LOW>], u + row * d.nu, d.nu);
                    if (MODE == 1) copy_row(&S.y[t][r][g][d.nx - kFirstCol<LOW>], y + row * d.ny, d.ny);
#pragma unroll
                    for (int j = 0; j < NP; ++j) copy_async<4>(&S.p[t][r][g][j], p + row * NP + j);
                }
            }
        }
        copy_commit();
    };
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c) fetch(c);
    float s[RG][4] = {};   // x_0 = 0; zero in the columns that hold no state
    float lsum_f = 0.f;    // widened to FP64 once, after the loop
    float* ho[RG];         // where this lane's part of the next row goes; beyond the data always the spare row
    int h_step[RG];
#pragma unroll
    for (int r = 0; r < RG; ++r) {
        const int tr = min(first + 8 * r + g, n_traj);
        ho[r] = hist + (size_t)tr * T * 16 + 4 * t;
        h_step[r] = tr < n_traj ? 16 : 0;
    }
    auto step = [&](const InStage<LOW, RG>& S, int q, int k) {
        float z[8], pp[RG][2];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r >= RG) {
                z[2 * r] = z[2 * r + 1] = z[4 + 2 * r] = z[5 + 2 * r] = 0.f;
                continue;
            }
            float uv[4];
            load_vals<LOW>(S.u[q][r][g], t, uv);
            const float2 pv = *reinterpret_cast<const float2*>(S.p[q][r][g]);
            pp[r][0] = (pv.x - pm[0]) * ips[r][0];
            pp[r][1] = (pv.y - pm[1]) * ips[r][1];
#pragma unroll
            for (int j = 0; j < 4; ++j)  // at a column either the state or the input is zero: the sum is exact
                z[4 * (j >> 1) + 2 * r + (j & 1)] = LOW || j >= 2 ? s[r][j] + uv[j] * fu[j] : s[r][j];
        }
        float D[8];
        product<NP, RG>(D, z, pp, bhi, blo);
#pragma unroll
        for (int r = 0; r < RG; ++r) {
            float yv[4], res[4] = {0.f, 0.f, 0.f, 0.f};
            if (MODE == 1) load_vals<LOW>(S.y[q][r][g], t, yv);
#pragma unroll
            for (int j = LOW ? 0 : 2; j < 4; ++j) {
                const float o = D[4 * (j >> 1) + 2 * r + (j & 1)];
                if (MODE == 0) {
                    if (is_y[r][j])
                        y_out[((size_t)(first + 8 * r + g) * T + k) * d.ny + (8 * (j >> 1) + 2 * t + (j & 1) - d.nx)] =
                            o * fy[j];
                } else {
                    res[j] = is_y[r][j] ? o - yv[j] * fy[j] : 0.f;
                    lsum_f = fmaf(res[j], res[j], lsum_f);
                    res[j] *= grad_scale;
                }
            }
            if (MODE == 1) {
                float h[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) h[j] = (LOW || j >= 2) && !is_x[j] ? res[j] : s[r][j];
                *reinterpret_cast<float4*>(ho[r]) = make_float4(h[0], h[1], h[2], h[3]);
                ho[r] += h_step[r];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float o = D[4 * (j >> 1) + 2 * r + (j & 1)];
                s[r][j] = (LOW || j >= 2) ? (is_x[j] ? o : 0.f) : o;
            }
        }
    };
    for (int c = 0; c < n_chunk; ++c) {
        copy_wait<kStages - 2>();
        fetch(c + kStages - 1);  // its buffer was read before the wait's barrier
        const InStage<LOW, RG>& S = sm[c % kStages];
        if ((c + 1) * kC <= T) {
#pragma unroll
            for (int q = 0; q < kC; ++q) step(S, q, c * kC + q);
        } else {
            for (int q = 0; c * kC + q < T; ++q) step(S, q, c * kC + q);
        }
    }
    if (MODE == 1) {
        double lsum = (double)lsum_f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_down_sync(0xffffffffu, lsum, o);
        if (lane == 0) loss_part[wid] = lsum;
    }
}

// B fragments of the adjoint product gw[row][f] = sum_o G[row][o] Wp[o][f]
// (k = output o, n = feature f; two n-tiles of features per scheduling block).
template <int NT>
__device__ __forceinline__ void load_bwd_frags(const float* __restrict__ Wp, uint32_t (*bhi)[2], uint32_t (*blo)[2],
                                               int g, int t)
{
    constexpr int ld = kFB * kMaxKT;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        const int f = nt * 8 + g;
        split2(Wp[(2 * t) * ld + f], Wp[(2 * t + 1) * ld + f], bhi[nt][0], blo[nt][0]);
        split2(Wp[(8 + 2 * t) * ld + f], Wp[(9 + 2 * t) * ld + f], bhi[nt][1], blo[nt][1]);
    }
}

// Transpose of an 8 x 8 tile of 16-bit elements held as one register per lane.
__device__ __forceinline__ uint32_t trans8(uint32_t a)
{
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(a));
    return r;
}

// The adjoint and the weight gradient of 16 trajectories, k = T-1 .. 0:
//   G_k = [lambda_{k+1}; dJ/dy_k],  gw_k = G_k W,
//   lambda_k = gw_k[x] + sum_i p_{k,i} gw_k[block i, x],
//   dJ/dW += G_k^T w_k.
// Warps 0 and 1 carry the adjoint of 8 trajectories each and leave G_k, split,
// in shared memory; the other warps add up the gradient, an n-tile (8 of
// the 48 features) each, a chunk of kC steps behind them, so that the gradient's products, splits and
// transposes take no part in the serial chain.  Both operands of a gradient
// product come as row fragments (rows are trajectories) and it contracts over
// the rows: each 8 x 8 tile is transposed in registers.  The accumulators run
// over all steps of the 16 trajectories (gpart[block][16][48], added up in
// FP64 by launch_reduce): sums in other parts were measured and differ from
// these by up to 7e-5, the rounding of a 1,000-step FP32 tensor-core sum.
// One block per SM is asked for: the registers that the gradient's warps may
// take then are what lets four steps overlap (820 trajectories of 1,000
// samples 173 us, 201 with 79 registers).
template <int NP>
constexpr int kAdjWarps = 2 + 2 * (1 + NP);

template <int NP>
struct AdjStage {
    float h[kC][2][kFrag];     // x_k and the residuals' part of G_k
    float u[kC][16][16];       // inputs at their columns (zero elsewhere)
    float p[kC][16][2];
};

template <int NP>
__global__ void __launch_bounds__(32 * kAdjWarps<NP>, 1) adj_kernel(const float* __restrict__ Wp, Dims d,
                                                            const float* __restrict__ u,
                                                            const float* __restrict__ p, int n_traj, int T,
                                                            const float* __restrict__ hist,
                                                            float* __restrict__ gpart)
{
    __shared__ __align__(16) AdjStage<NP> sm[kStages];
    __shared__ __align__(16) float sG[2][kC][2][kFrag];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, wl = threadIdx.x >> 5;
    const int first = blockIdx.x * 16, n_chunk = (T + kC - 1) / kC;
    const bool is_adj = wl < 2;
    {   // rows beyond the data stay zero
        float* z = reinterpret_cast<float*>(sm);
        for (int i = threadIdx.x; i < (int)(sizeof(sm) / sizeof(float)); i += blockDim.x) z[i] = 0.f;
    }
    __syncthreads();
    // the inputs that this lane copies next, and down to which k0
    const int u_row = min(first + 8 * ((wl - 2) & 1) + g, n_traj - 1);
    const float* u_next = u + ((ptrdiff_t)u_row * T + (T - 1 - t)) * d.nu;
    const int u_from = first + 8 * (wl - 2) + g < n_traj ? t : INT_MAX;
    // chunk c holds steps T - 1 - c kC - q for q = 0, 1, ..; fetched in order
    auto fetch = [&](int c) {
        AdjStage<NP>& S = sm[c % kStages];
        const int k0 = T - 1 - c * kC;
        if (is_adj) {  // the history of a warp's rows, and their p, a step per lane
            const int tr = first + 8 * wl + g;
            if (tr < n_traj) {
                const float* src = hist + ((size_t)tr * T + k0) * 16 + 4 * t;
#pragma unroll
                for (int q = 0; q < kC; ++q)
                    if (k0 - q >= 0) copy_async<16>(&S.h[q][wl][4 * lane], src - q * 16);
                if (k0 - t >= 0)
#pragma unroll
                    for (int j = 0; j < NP; ++j)
                        copy_async<4>(&S.p[t][8 * wl + g][j], p + ((size_t)tr * T + (k0 - t)) * NP + j);
            }
        } else if (wl < 4) {  // the inputs of 8 rows, a step per lane
            if (k0 >= u_from) copy_row(&S.u[t][8 * (wl - 2) + g][d.nx], u_next, d.nu);
            u_next -= kC * d.nu;
        }
        copy_commit();
    };
    // zero scheduling beyond the data, as the free run takes it
    float pm[2], ips[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        pm[j] = j < NP ? d.pm[j] : 0.f;
#pragma unroll
        for (int r = 0; r < 2; ++r) ips[r][j] = j < NP && first + 8 * r + g < n_traj ? d.inv_ps[j] : 0.f;
    }
    constexpr int NT = 2 + 2 * NP;
    fetch(0);
    fetch(1);
    if (is_adj) {
        bool is_x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) is_x[j] = 8 * (j >> 1) + 2 * t + (j & 1) < d.nx;
        float ip[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) ip[j] = wl ? ips[1][j] : ips[0][j];
        uint32_t bhi[NT][2], blo[NT][2];
        load_bwd_frags<NT>(Wp, bhi, blo, g, t);
        float lam[4] = {0, 0, 0, 0};  // lambda_T = 0
        auto step = [&](const AdjStage<NP>& S, float* out, int q) {
            const float4 v = *reinterpret_cast<const float4*>(&S.h[q][wl][4 * lane]);
            const float2 pv = *reinterpret_cast<const float2*>(S.p[q][8 * wl + g]);
            const float pp[2] = {(pv.x - pm[0]) * ip[0], (pv.y - pm[1]) * ip[1]};
            // rows 0-7 the high, rows 8-15 the low parts (as in the free run)
            uint32_t a[4];
            split2(is_x[0] ? lam[0] : v.x, is_x[1] ? lam[1] : v.y, a[0], a[1]);
            split2(is_x[2] ? lam[2] : v.z, is_x[3] ? lam[3] : v.w, a[2], a[3]);
            *reinterpret_cast<uint4*>(out + (q * 2 + wl) * kFrag + 4 * lane) = make_uint4(a[0], a[1], a[2], a[3]);
            float2 gw[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                float c0[4], c1[4];
                mma16816_0(c0, a, bhi[nt][0], bhi[nt][1]);
                mma16816_0(c1, a, blo[nt][0], blo[nt][1]);
                gw[nt] = add2(make_float2(c0[0], c0[1]), add2(make_float2(c1[0], c1[1]), make_float2(c0[2], c0[3])));
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 l = gw[h];
#pragma unroll
                for (int m = 0; m < NP; ++m) {
                    l.x = fmaf(pp[m], gw[h + 2 + 2 * m].x, l.x);
                    l.y = fmaf(pp[m], gw[h + 2 + 2 * m].y, l.y);
                }
                lam[2 * h] = l.x;  // columns beyond the state are never used
                lam[2 * h + 1] = l.y;
            }
        };
        for (int c = 0; c <= n_chunk; ++c) {
            copy_wait<1>();
            __syncthreads();
            if (c < n_chunk) {
                fetch(c + 2);  // the stage last read two chunks ago
                const AdjStage<NP>& S = sm[c % kStages];
                float* out = &sG[c & 1][0][0][0];
                if ((c + 1) * kC <= T) {
#pragma unroll
                    for (int q = 0; q < kC; ++q) step(S, out, q);
                } else {
                    for (int q = 0; c * kC + q < T; ++q) step(S, out, q);
                }
            }
        }
        return;
    }
    const int kt = (wl - 2) >> 1, h = (wl - 2) & 1;  // scheduling block and half of the features of this warp
    const bool scaled = kt > 0;
    float pk = 0.f, ik[2] = {1.f, 1.f};
    if (scaled) {
        pk = kt == 1 ? pm[0] : pm[1];
        ik[0] = kt == 1 ? ips[0][0] : ips[0][1];
        ik[1] = kt == 1 ? ips[1][0] : ips[1][1];
    }
    // where this lane's two columns of z_k lie in a stage, in x_k or in u, as
    // steps and groups of 8 rows are as far apart in both, and their factors
    int at[2];
    float2 f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int c = 8 * h + 2 * t + j - d.nx;
        at[j] = c < 0 ? 4 * lane + 2 * h + j : kC * 2 * kFrag + 16 * g + 8 * h + 2 * t + j;
        (j ? f.y : f.x) = c < 0 ? 1.f : c < d.nu ? d.inv_su[c] : 0.f;
    }
    static_assert(offsetof(AdjStage<NP>, u) == kC * 2 * kFrag * sizeof(float) && sizeof(AdjStage<NP>::u) == sizeof(AdjStage<NP>::h),
                  "u follows h, steps and rows as far apart");
    float acc[4] = {0, 0, 0, 0};
    auto step = [&](auto paired, const AdjStage<NP>& S, const float* in, int q) {
        const uint4 ga = *reinterpret_cast<const uint4*>(in + (q * 2) * kFrag + 4 * lane);
        const uint4 gb = *reinterpret_cast<const uint4*>(in + (q * 2 + 1) * kFrag + 4 * lane);
        auto z = [&](int r) {
            const float* s = &S.h[0][0][0] + (2 * q + r) * kFrag;
            const float2 v = decltype(paired)::value ? *reinterpret_cast<const float2*>(s + at[0]) : make_float2(s[at[0]], s[at[1]]);
            return mul2(v, f);
        };
        float2 za = z(0), zb = z(1);
        if (scaled) {
            const float pa = (S.p[q][g][kt - 1] - pk) * ik[0], pb = (S.p[q][8 + g][kt - 1] - pk) * ik[1];
            za = mul2(za, make_float2(pa, pa));
            zb = mul2(zb, make_float2(pb, pb));
        }
        // A = G^T: (outputs 0-7 | 8-15) x (rows 0-7 | 8-15), in the order 00, 10, 01, 11
        const uint32_t ahi[4] = {trans8(ga.x), trans8(ga.z), trans8(gb.x), trans8(gb.z)};
        const uint32_t alo[4] = {trans8(ga.y), trans8(ga.w), trans8(gb.y), trans8(gb.w)};
        uint32_t ha, la, hb, lb;
        split2(za.x, za.y, ha, la);
        split2(zb.x, zb.y, hb, lb);
        const uint32_t b0h = trans8(ha), b1h = trans8(hb), b0l = trans8(la), b1l = trans8(lb);
        mma16816(acc, ahi, b0h, b1h);
        mma16816(acc, ahi, b0l, b1l);
        mma16816(acc, alo, b0h, b1h);
    };
    auto run = [&](auto paired) {
        for (int c = 0; c <= n_chunk; ++c) {
            copy_wait<1>();
            __syncthreads();
            if (c < n_chunk) fetch(c + 2);
            if (c == 0) continue;
            const AdjStage<NP>& S = sm[(c - 1) % kStages];
            const float* in = &sG[(c - 1) & 1][0][0][0];
            if (c * kC <= T) {
#pragma unroll
                for (int q = 0; q < kC; ++q) step(paired, S, in, q);
            } else {
                for (int q = 0; (c - 1) * kC + q < T; ++q) step(paired, S, in, q);
            }
        }
    };
    // both columns of every lane in one of the two: all warps of an even state, and the half of an odd one without its end
    if (d.nx % 2 == 0 || d.nx / 8 != h) run(std::true_type{});
    else run(std::false_type{});
    // acc: (o = g, f = 8 h + 2t), (g, +1), (g + 8, 2t), (g + 8, 2t + 1) of block kt
    constexpr int ld = kFB * kMaxKT;
    float* out = gpart + (size_t)blockIdx.x * kWN;
#pragma unroll
    for (int q = 0; q < 4; ++q) out[(g + 8 * (q >> 1)) * ld + kt * kFB + 8 * h + 2 * t + (q & 1)] = acc[q];
    if constexpr (NP + 1 < kMaxKT) {  // the blocks that this model does not have
        constexpr int n = (kMaxKT - 1 - NP) * kFB;
        if (wl == 2)
            for (int i = lane; i < kO * n; i += 32) out[(i / n) * ld + (1 + NP) * kFB + i % n] = 0.f;
    }
}

// FP32 values of N doubles on the integer pipe.  A conversion instruction
// takes 16 cycles of an SM's FP64 pipe whichever way it converts: with the
// inputs converted once per row here, the outputs' conversions (one in four
// lanes each) are all that this pipe is left with, 64 cycles per warp of 16
// runs and period, beside as many issue slots.  Gives what the instruction
// gives: to nearest (ties to even); zeros keep their sign; what is neither
// zero nor a normal FP32 number is left to the instruction (a branch no warp
// takes otherwise).
template <int N>
__device__ __forceinline__ void to_float(const double* x, float* r)
{
    bool other[N], any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const unsigned hi = (unsigned)__double2hiint(x[i]), lo = (unsigned)__double2loint(x[i]), m = hi & 0x7fffffffu;
        const bool normal = m - 0x38100000u < 0x0fe00000u, zero = (m | lo) == 0u;
        unsigned f = __funnelshift_l(lo, m - 0x38000000u, 3);
        f += ((lo & 0x1fffffffu) + 0x0fffffffu + (f & 1u)) >> 29;
        r[i] = __uint_as_float((normal ? f : 0u) | (hi & 0x80000000u));
        other[i] = !normal && !zero;
        any |= other[i];
    }
    if (__any_sync(0xffffffffu, any)) {
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (other[i]) r[i] = (float)x[i];
    }
}

struct BodyPar {
    float inv_m, inv_J, dt;      // substep dt = Ts / n_sub
    float n, n_half;             // n_sub and n_sub (n_sub + 1) / 2
    float kp, kd;                // PD gains J w^2 and 2 xi J w
};

// Closed loop of 8 RG runs per warp (Sections 5.1.1, 5.4): per period the PD
// torque (Eq. 28, zero-order hold), the surrogate step with p = [fill,
// thetadot], and n_sub kick-then-drift substeps of the body under the held
// forces, summed in closed form: v += n dt a, x += n dt v + dt^2 a n(n+1)/2.
// The body state (FP32) is replicated in the four lanes of each row.  A chunk
// of kC periods of the inputs passes through shared memory: the four lanes of
// a row copy one period each, three chunks ahead, and convert it once for all
// four.  65,536 runs of 500 periods (n_x 12, n_p 2): 2.60 -> 0.92 ms, 2.8 TB/s;
// bound by the 297 instructions of a warp's period (50 % of the issue slots,
// 44 % of the FP64 pipe for the outputs) at 14 to 16 warps per SM, and by the
// period's chain for few runs.
// wide: out is 16-byte aligned, so that three lanes store a row's sample.
template <bool LOW, int NP, int RG>
__global__ void __launch_bounds__(32, RG == 2 ? 16 : 1) closed_loop_kernel(const float* __restrict__ Wp, Dims d, int B, int T,
                                                         const double* __restrict__ F, const double* __restrict__ tau,
                                                         const double* __restrict__ ref,
                                                         const double* __restrict__ fill, BodyPar bp,
                                                         double* __restrict__ out, int wide)
{
    __shared__ double raw[kStages][kC][RG][8][4];            // F_x, F_y, tau, theta_ref
    __shared__ __align__(16) float4 in[kC][RG][8];
    const int lane = threadIdx.x, g = lane >> 2, t = lane & 3, first = blockIdx.x * 8 * RG;
    for (int i = lane; i < kStages * kC * RG * 32; i += 32) (&raw[0][0][0][0][0])[i] = 0.0;  // rows beyond B stay zero
    __syncwarp();
    uint32_t bhi[kMaxKT][2][2], blo[kMaxKT][2][2];
    load_fwd_frags(Wp, bhi, blo, 1 + NP, g, t);
    bool is_x[4];
    float fu[4];
    int uq[4];  // the input at a column, 3 where none lies
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int q = 8 * (j >> 1) + 2 * t + (j & 1) - d.nx;
        is_x[j] = q < 0;
        uq[j] = q >= 0 && q < min(d.nu, 3) ? q : 3;
        fu[j] = uq[j] < 3 ? d.inv_su[uq[j]] : 0.f;
    }
    // lane and register of the loads F_x, F_y, T_b: columns n_x, n_x + 1, n_x + 2 of D
    int src[3];
    bool up[3], odd[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int c = d.nx + j;
        src[j] = (lane & ~3) + ((c & 7) >> 1);
        up[j] = c >= 8;
        odd[j] = c & 1;
    }
    float pp[RG][2];
    bool valid[RG];
#pragma unroll
    for (int r = 0; r < RG; ++r) {
        const int run = first + 8 * r + g;
        valid[r] = run < B;
        // scheduling clamped to the range it was identified on
        const float fl = valid[r] ? (float)fill[run] : 0.f;
        pp[r][0] = NP > 0 ? (fminf(fmaxf(fl, d.plo[0]), d.phi[0]) - d.pm[0]) * d.inv_ps[0] : 0.f;
        pp[r][1] = 0.f;
    }
    const int n_chunk = (T + kC - 1) / kC;
    auto fetch = [&](int c) {
        const int k = c * kC + t;
        if (k < T) {
#pragma unroll
            for (int r = 0; r < RG; ++r)
                if (valid[r]) {
                    const size_t o = (size_t)(first + 8 * r + g) * T + k;
                    double* dst = raw[c % kStages][t][r][g];
                    copy_async<8>(dst, F + 2 * o);
                    copy_async<8>(dst + 1, F + 2 * o + 1);
                    copy_async<8>(dst + 2, tau + o);
                    copy_async<8>(dst + 3, ref + o);
                }
        }
        copy_commit();
    };
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c) fetch(c);
    float s[RG][4] = {}, bs[RG][6] = {};  // surrogate state; r_x r_y theta v_x v_y omega
    const float ndt = bp.n * bp.dt, hdt2 = bp.n_half * bp.dt * bp.dt;
    double* o0 = out + (size_t)(first + g) * T * 6 + 2 * t;
    auto step = [&](int q, int k) {
        float z[8], uu[RG][3];
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r >= RG) {
                z[2 * r] = z[2 * r + 1] = z[4 + 2 * r] = z[5 + 2 * r] = 0.f;
                continue;
            }
            const float4 v = in[q][r][g];
            // the sample before the period: lane t stores components 2t, 2t + 1
            const double a = (double)(t == 0 ? bs[r][0] : t == 1 ? bs[r][2] : bs[r][4]);
            const double b = (double)(t == 0 ? bs[r][1] : t == 1 ? bs[r][3] : bs[r][5]);
            if (valid[r] && t < 3) {
                double* o = o0 + ((size_t)(8 * r) * T + k) * 6;
                if (wide) {
                    *reinterpret_cast<double2*>(o) = make_double2(a, b);
                } else {
                    o[0] = a;
                    o[1] = b;
                }
            }
            // rounding written out, so that a run gives the same in either row split
            const float tc = fmaf(bp.kp, v.w - bs[r][2], -__fmul_rn(bp.kd, bs[r][5]));
            uu[r][0] = v.x;
            uu[r][1] = v.y;
            uu[r][2] = v.z + tc;
            if (NP > 1) pp[r][1] = (fminf(fmaxf(bs[r][5], d.plo[1]), d.phi[1]) - d.pm[1]) * d.inv_ps[1];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float u = 0.f;
                if (LOW || j >= 2)
                    u = (uq[j] == 0 ? uu[r][0] : uq[j] == 1 ? uu[r][1] : uq[j] == 2 ? uu[r][2] : 0.f) * fu[j];
                z[4 * (j >> 1) + 2 * r + (j & 1)] = LOW || j >= 2 ? s[r][j] + u : s[r][j];  // one of the two is zero
            }
        }
        float D[8];
        product<NP, RG>(D, z, pp, bhi, blo);
#pragma unroll
        for (int r = 0; r < RG; ++r) {
            float load[3];  // sloshing loads: the first three outputs, in physical units
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float hi = odd[j] ? D[5 + 2 * r] : D[4 + 2 * r];
                float v = hi;
                if (LOW) v = up[j] ? hi : (odd[j] ? D[1 + 2 * r] : D[2 * r]);
                load[j] = __shfl_sync(0xffffffffu, v, src[j]) * d.sy[j];
            }
            const float ax = (uu[r][0] + load[0]) * bp.inv_m, ay = (uu[r][1] + load[1]) * bp.inv_m;
            const float aw = (uu[r][2] + load[2]) * bp.inv_J;
            bs[r][0] += fmaf(hdt2, ax, __fmul_rn(ndt, bs[r][3]));
            bs[r][1] += fmaf(hdt2, ay, __fmul_rn(ndt, bs[r][4]));
            bs[r][2] += fmaf(hdt2, aw, __fmul_rn(ndt, bs[r][5]));
            bs[r][3] += ndt * ax;
            bs[r][4] += ndt * ay;
            bs[r][5] += ndt * aw;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float v = D[4 * (j >> 1) + 2 * r + (j & 1)];
                s[r][j] = (LOW || j >= 2) ? (is_x[j] ? v : 0.f) : v;
            }
        }
    };
    for (int c = 0; c < n_chunk; ++c) {
        copy_wait<kStages - 2>();
        fetch(c + kStages - 1);
#pragma unroll
        for (int r = 0; r < RG; ++r) {  // the period this lane copied
            float v[4];
            to_float<4>(raw[c % kStages][t][r][g], v);
            in[t][r][g] = make_float4(v[0], v[1], v[2], v[3]);
        }
        __syncwarp();
        if ((c + 1) * kC <= T) {
#pragma unroll
            for (int q = 0; q < kC; ++q) step(q, c * kC + q);
        } else {
            for (int q = 0; c * kC + q < T; ++q) step(q, c * kC + q);
        }
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Row groups per warp of the serial passes: one while a warp per group still
// finds a scheduler of its own (152 SMs x 4), two beyond.
static int row_groups(int n_traj) { return groups_for(n_traj) <= 608 ? 1 : 2; }

int serial_warps(int n_traj) { return (groups_for(n_traj) + row_groups(n_traj) - 1) / row_groups(n_traj); }

template <class F>
static void by_np(int np, F&& f)
{
    if (np == 0) f(std::integral_constant<int, 0>{});
    else if (np == 1) f(std::integral_constant<int, 1>{});
    else f(std::integral_constant<int, 2>{});
}

cudaError_t launch_forward(int mode, const float* Wp, const Dims& d, const float* u, const float* p, const float* y,
                           int n_traj, int T, float* y_out, float* hist, double* loss_part, float grad_scale,
                           cudaStream_t st)
{
    const int warps = serial_warps(n_traj);
    by_np(d.np, [&](auto np) {
        constexpr int NP = decltype(np)::value;
        auto go = [&](auto kernel) {
            kernel<<<warps, 32, 0, st>>>(Wp, d, u, p, y, n_traj, T, y_out, hist, loss_part, grad_scale);
        };
        const bool low = d.nx < 8, one = row_groups(n_traj) == 1;
        if (mode == 0) {
            if (one) low ? go(fwd_kernel<0, true, NP, 1>) : go(fwd_kernel<0, false, NP, 1>);
            else low ? go(fwd_kernel<0, true, NP, 2>) : go(fwd_kernel<0, false, NP, 2>);
        } else {
            if (one) low ? go(fwd_kernel<1, true, NP, 1>) : go(fwd_kernel<1, false, NP, 1>);
            else low ? go(fwd_kernel<1, true, NP, 2>) : go(fwd_kernel<1, false, NP, 2>);
        }
    });
    return cudaGetLastError();
}

cudaError_t launch_backward(const float* Wp, const Dims& d, const float* u, const float* p, int n_traj, int T,
                            const float* hist, float* gpart, cudaStream_t st)
{
    by_np(d.np, [&](auto np) {
        constexpr int NP = decltype(np)::value;
        adj_kernel<NP><<<grad_parts(n_traj), 32 * kAdjWarps<NP>, 0, st>>>(Wp, d, u, p, n_traj, T, hist, gpart);
    });
    return cudaGetLastError();
}

cudaError_t launch_closed_loop(const float* Wp, const Dims& d, int B, int T, const double* F, const double* tau,
                               const double* ref, const double* fill, const BodyParHost& h, double* out,
                               cudaStream_t st)
{
    const BodyPar bp{h.inv_m, h.inv_J, h.dt, h.n, h.n_half, h.kp, h.kd};
    const int wide = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    by_np(d.np, [&](auto np) {
        constexpr int NP = decltype(np)::value;
        auto go = [&](auto kernel) {
            kernel<<<serial_warps(B), 32, 0, st>>>(Wp, d, B, T, F, tau, ref, fill, bp, out, wide);
        };
        if (row_groups(B) == 1) d.nx < 8 ? go(closed_loop_kernel<true, NP, 1>) : go(closed_loop_kernel<false, NP, 1>);
        else d.nx < 8 ? go(closed_loop_kernel<true, NP, 2>) : go(closed_loop_kernel<false, NP, 2>);
    });
    return cudaGetLastError();
}

}  // namespace lpv
