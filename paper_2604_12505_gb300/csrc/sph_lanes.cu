// sph_lanes.cu -- the density and force pass of a step with four lanes per
// particle, for tanks that fill the GPU a few warps deep.
//
// With a thread per particle the passes of such a tank are long loops in few
// warps, on a chain of staging rounds: a step takes 26 us from 4,000 to 25,000
// particles alike (40 at the paper's smoothing length, with more neighbours).
// Here a 4x4 tile has 512 threads instead of 128, so the loops are a quarter as
// long and the staging takes a quarter of the rounds: 19 to 22 us (25 to 29).
// Bound by the chain of a step still: staging rounds through L2, the ghosts
// after the body's update, three launches.
// The staged tile, its order and its record are those of density_kernel<4,4>;
// the sums add in its order (sph_lanes.cuh), and a tile's force sums run over
// the same 128 places in the same tree: results equal bit for bit.  The
// neighbour record holds a particle's three runs of candidates instead of its
// neighbours: all are evaluated again, and no bits are looked up.
#include <climits>

#include "sph_common.cuh"
#include "sph_launch.h"
#include "sph_tile.cuh"
#include "sph_lanes.cuh"

namespace sph {

namespace {

constexpr int kLanes = 4;
using Sh = Shape<4, 4>;
constexpr int kPlaces = Sh::THREADS;           // particles at once
constexpr int kThreads = kPlaces * kLanes;

// The runs of staged ghosts within clip of a particle, in the order of
// for_staged_ghosts; lane r looks in row r of the 3x3 ghost cells.
__device__ __forceinline__ Runs ghost_runs(const TankDev& T, const GhostStage<>& gs, bool on, float x, float y, float bc,
                                           float bs, float brx, float bry, float clip, int sub)
{
    int gx, gy, a = 0, b = 0;
    float ex, ey;
    if (on && ghost_cell(T, x, y, bc, bs, brx, bry, gx, gy, ex, ey) && sub < 3) {
        const int x0 = max(gx - 1, 0), x1 = min(gx + 1, T.G - 1), yy = gy - 1 + sub;
        const int X0 = gs.box[0], X1 = gs.box[1], Y0 = gs.box[2], Y1 = gs.box[3];
        const float ylo = T.g_orig + (float)yy * T.g_cell;
        const bool away = yy > 0 && yy < T.G - 1 && (ylo > ey + clip || ylo + T.g_cell < ey - clip);
        if (x0 <= x1 && x0 >= X0 && x1 <= X1 && yy >= Y0 && yy <= Y1 && !away) {
            const int r = yy - Y0, base = gs.base[r];
            a = base + gs.tab[r][x0 - X0];
            b = base + gs.tab[r][x1 + 1 - X0];
            if (x0 > 0 && x1 < T.G - 1) {
                a = lower_bx(gs, a, b, ex - clip);
                b = lower_bx(gs, a, b, ex + clip);
            }
        }
    }
    return lane_runs<kLanes>(pack_run(a, b));
}

__global__ void __launch_bounds__(kThreads, 2) density_lanes_kernel(SimDev S, int chained)
{
    __shared__ Stage<4, 4, false, false> sm;
    __shared__ GhostStage<> gs;
    const int4 td = S.tiles[blockIdx.x];
    const TankDev T = S.tank[td.x];
    const int cx0 = td.y, cy0 = td.z;
    const int sub = threadIdx.x & (kLanes - 1), mine = threadIdx.x / kLanes;
    const int first = (threadIdx.x & ~31) / kLanes;  // the warp's first place
    // as in density_pass: staged and summed over the fluid before the dependency
    int buf;
    if (chained) {
        buf = __ldcg(&S.run->next_buf);
    } else {
        pdl_wait();
        buf = (int)(S.run->step & 1);
    }
    const int nbuf = buf ^ 1;
    for (int c = threadIdx.x; c < 16; c += kThreads) {
        const int ix = cx0 + c % 4, iy = cy0 + c / 4;
        if (ix < T.G && iy < T.G) S.count[nbuf][T.cell_base + iy * T.G + ix] = 0;
    }
    const bool staged = stage_tile<4, 4, false>(S, T, buf, cx0, cy0, sm);
    save_stage(sm, staged, stage_record<4, 4>(S, blockIdx.x));
    const int n_own = staged ? sm.own_row[4] : 0;
    if (n_own == 0) {
        if (chained && blockIdx.x == 0) pdl_wait();
        return;
    }
    for (int p = 0; first + p < n_own; p += kPlaces) {  // by whole warps
        const int t = mine + p;
        const bool on = t < n_own;
        const int e = own_index(on ? t : 0, sm);
        const float4 pi = sm.pv[e];
        const float2 li = sm.plo[e];
        int a = 0, z = 0;
        if (on && sub < 3) {
            const int cl = sm.cell[e] + (sub - 1) * Sh::SX - 1;
            a = lower_x(sm, sm.start[cl], sm.start[cl + 1], pi.x - T.clip);
            z = lower_x(sm, sm.start[cl + 2], sm.start[cl + 3], pi.x + T.clip);
            if (t < Sh::MAXOWN) S.nbm[(size_t)blockIdx.x * (3 * Sh::MAXOWN) + t + sub * Sh::MAXOWN] = pack_run(a, z);
        }
        const Runs R = lane_runs<kLanes>(pack_run(a, z));
        const float Sf = fluid_sum<kLanes>(T, R, e, pi, li, sm.pv, sm.plo, sub);
        if (on && sub == 0) sm.key_in[t] = __float_as_uint(__fmul_rn(Sf, T.cW));
    }
    if (chained) pdl_wait();
    const BodyDev& b = S.body[td.x];
    const float bc = b.fc, bs = b.fs, brx = b.frx, bry = b.fry;
    const GhostFrame fr = ghost_frame(b);
    const int gmode = stage_ghosts<true>(S, T, bc, bs, brx, bry, fr, sm, n_own, gs, NoTangent{});
    for (int p = 0; first + p < n_own; p += kPlaces) {
        const int t = mine + p;
        const bool on = t < n_own;
        const int e = own_index(on ? t : 0, sm);
        const float4 pi = sm.pv[e];
        const float2 li = sm.plo[e];
        float Sg = 0.f;
        if (gmode == kGhostsStaged) {
            const Runs Q = ghost_runs(T, gs, on, pi.x, pi.y, bc, bs, brx, bry, T.clip, sub);
            Sg = ghost_sum<kLanes>(T, Q, pi, li, gs.gp, sub);
        } else if (gmode == kGhostsGlobal) {  // more ghosts than are staged: one lane alone
            if (on && sub == 0)
                for_ghosts(S, T, pi.x, pi.y, bc, bs, brx, bry, [&](int g) {
                    float4 gp, gv;
                    ghost_world(fr, __ldg(S.gB + g), gp, gv);
                    S.gpos[g] = gp;
                    S.gvel[g] = gv;
                    const float2 d = sep_fg(pi, li, gp);
                    const float r2 = dist2(d.x, d.y);
                    if (r2 < T.R2) Sg = fmaf(T.cW, ghost_bracket(T, r2), Sg);
                });
        }
        if (on && sub == 0) {
            const float rho = __fmul_rn(T.m, __fmaf_rn(T.gamma1, Sg, __uint_as_float(sm.key_in[t])));  // Eq. 14
            const float P = __fmul_rn(T.k, __fsub_rn(rho, T.rho0));                                     // Eq. 11
            S.rhoP[sm.slot[e]] = make_float2(rho, __fdiv_rn(P, __fmul_rn(rho, rho)));
        }
    }
    pdl_trigger();
}

__global__ void __launch_bounds__(kThreads, 2) force_lanes_kernel(SimDev S)
{
    __shared__ Stage<4, 4, true, false> sm;
    __shared__ GhostStage<> gs;
    __shared__ Red scratch[kPlaces / 32];
    __shared__ float part[5][kPlaces];  // wall force and torque, position sums of each place
    __shared__ unsigned pairs_all;
    pdl_trigger();
    const int4 td = S.tiles[blockIdx.x];
    const int tank = td.x;
    const TankDev T = S.tank[tank];
    const int sub = threadIdx.x & (kLanes - 1), mine = threadIdx.x / kLanes;
    const int first = (threadIdx.x & ~31) / kLanes;
    pdl_wait();
    const long long step = S.run->step;
    const int buf = (int)(step & 1), nbuf = buf ^ 1;
    if (blockIdx.x == 0 && threadIdx.x == 0) S.run->next_buf = nbuf;
    if (threadIdx.x == 0) pairs_all = 0u;
    const bool sample = (step % T.outer_every) == 0;
    const float damp = 1.0f - S.run->damping;
    if (!stage_from_record<kThreads, 4, 4, false>(S, tank, buf, stage_record<4, 4>(S, blockIdx.x), sm)) return;
    const int n_own = sm.own_row[4];
    if (n_own == 0) return;
    BodyDev& b = S.body[tank];
    const float bc = b.fc, bs = b.fs, brx = b.frx, bry = b.fry;
    const int gmode = stage_ghosts<false>(S, T, bc, bs, brx, bry, GhostFrame{}, sm, n_own, gs, NoTangent{});
    const float ox = b.fo_next[0], oy = b.fo_next[1];  // origin of the next grid
    int flags = 0, wall = 0;
    unsigned pairs = 0;
    WallSum W{0.f, 0.f, 0.f};
    float cxs = 0.f, cys = 0.f;
    for (int p = 0; first + p < n_own; p += kPlaces) {  // by whole warps
        const int t = mine + p;
        const bool on = t < n_own;
        const int e = own_index(on ? t : 0, sm);
        const float4 pi = sm.pv[e];
        const float2 li = sm.plo[e], ri = sm.rho[e];
        unsigned run = 0u;
        if (on && sub < 3) {
            if (t < Sh::MAXOWN) {
                run = S.nbm[(size_t)blockIdx.x * (3 * Sh::MAXOWN) + t + sub * Sh::MAXOWN];
            } else {
                const int cl = sm.cell[e] + (sub - 1) * Sh::SX - 1;
                run = pack_run(sm.start[cl], sm.start[cl + 3]);
            }
        }
        float ax = 0.f, ay = 0.f;
        const Runs R = lane_runs<kLanes>(run);
        pairs += (unsigned)fluid_forces<kLanes>(T, R, e, pi, li, ri, sm.pv, sm.plo, sm.rho, sub, ax, ay);
        BothSum B{W, ax, ay, T.inv_m};
        int met = 0;
        if (gmode == kGhostsStaged) {
            const Runs Q = ghost_runs(T, gs, on, pi.x, pi.y, bc, bs, brx, bry, T.hclip, sub);
            met = ghost_forces<kLanes>(T, Q, pi, li, ri, gs.gp, gs.gv, sub, B);
        } else if (gmode == kGhostsGlobal) {
            if (on && sub == 0)
                for_ghosts(S, T, pi.x, pi.y, bc, bs, brx, bry, [&](int g) {
                    const float2 d = sep_fg(pi, li, __ldg(S.gpos + g));
                    const float r2 = dist2(d.x, d.y);
                    if (!(r2 < T.h2)) return;
                    ++met;
                    if (!(r2 > 0.f)) return;
                    const float4 gv = __ldg(S.gvel + g);
                    B.add(ghost_force(T, pi, ri, gv, d, r2), d, make_float2(gv.z, gv.w));
                });
            B = B.of<kLanes>(0);
        }
        W = B;
        wall |= met > 0;
        pairs += (unsigned)met;
        if (on) {
            cxs += pi.x;
            cys += pi.y;
        }
        if (on && sub == 0) {
            ax = B.ax + T.grav_x;
            ay = B.ay + T.grav_y;
            // kick then drift, and the next grid, as in force_kernel
            const float2 vl = velocity_lo(S, buf, sm, e);
            float2 kx = two_sum(pi.z, fmaf(T.dt, ax, vl.x)), ky = two_sum(pi.w, fmaf(T.dt, ay, vl.y));
            if (damp != 1.0f) {
                const float hx = kx.x * damp, hy = ky.x * damp;
                kx = two_sum(hx, fmaf(kx.x, damp, -hx) + kx.y * damp);
                ky = two_sum(hy, fmaf(ky.x, damp, -hy) + ky.y * damp);
            }
            const float2 dx2 = two_sum(pi.x, fmaf(T.dt, kx.x, fmaf(T.dt, kx.y, li.x)));
            const float2 dy2 = two_sum(pi.y, fmaf(T.dt, ky.x, fmaf(T.dt, ky.y, li.y)));
            const float x = dx2.x, y = dy2.x;
            if (!(isfinite(x) && isfinite(y) && isfinite(kx.x) && isfinite(ky.x))) flags |= SPH_FLAG_NAN;
            bool out = false;
            const int ccx = cell_coord(x, ox, T.inv_cell, T.G, &out);
            const int ccy = cell_coord(y, oy, T.inv_cell, T.G, &out);
            const float ex = x - (ox + T.Wf), ey = y - (oy + T.Wf);
            if (out || fmaf(ex, ex, ey * ey) > T.cover2) flags |= SPH_FLAG_ESCAPED;
            const int cell = T.cell_base + ccy * T.G + ccx;
            const int slot = atomicAdd(&S.count[nbuf][cell], 1);
            if ((unsigned)slot < (unsigned)kCap) {
                S.pv[nbuf][cell * kCap + slot] = make_float4(x, y, kx.x, ky.x);
                S.lo[nbuf][cell * kCap + slot] = make_float4(dx2.y, dy2.y, kx.y, ky.y);
                S.pid[nbuf][cell * kCap + slot] = sm.pid[e];
            } else {
                flags |= SPH_FLAG_CELL_FULL;
            }
        }
    }
    if (flags) atomicOr(&b.flags, flags);
    if (sub == 0) {
        part[0][mine] = W.fx;
        part[1][mine] = W.fy;
        part[2][mine] = W.t;
        part[3][mine] = cxs;
        part[4][mine] = cys;
    }
    pairs = __reduce_add_sync(0xffffffffu, pairs);
    if ((threadIdx.x & 31) == 0 && pairs) atomicAdd(&pairs_all, pairs);
    // the tile's sums as force_kernel takes them: 128 places, a tree of four warps
    const bool any_wall = __syncthreads_or(wall) != 0;
    if (threadIdx.x >= kPlaces) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Red r{{part[0][threadIdx.x], 0.f}, {part[1][threadIdx.x], 0.f}, {part[2][threadIdx.x], 0.f},
          {part[3][threadIdx.x], 0.f}, {part[4][threadIdx.x], 0.f}, 0ull};
    r = warp_reduce(r, any_wall, sample);
    if (lane == 0) scratch[warp] = r;
    asm volatile("bar.sync 1, %0;" ::"n"(kPlaces) : "memory");
    if (warp) return;
    const F2 z{0.f, 0.f};
    r = lane < kPlaces / 32 ? scratch[lane] : Red{z, z, z, z, z, 0ull};
    r = warp_reduce(r, any_wall, sample, kPlaces / 64);
    auto all = [](F2 v) { return F2{__shfl_sync(0xffffffffu, v.hi, 0), __shfl_sync(0xffffffffu, v.lo, 0)}; };
    const F2 fx = all(r.fx), fy = all(r.fy), tq = all(r.t), cx = all(r.cx), cy = all(r.cy);
    const F2 q = lane == 0 ? fx : lane == 1 ? fy : lane == 2 ? tq : lane == 3 ? cx : cy;
    if ((lane < 3 && any_wall) || (lane >= 3 && lane < 5 && sample)) fix_add(&b.acc[lane], q);
    if (lane == 5 && pairs_all) atomicAdd(&b.pairs, (unsigned long long)pairs_all);
}

}  // namespace

cudaError_t launch_lanes(const SimDev& S, int n_tiles, int phase, cudaStream_t st, bool pdl, int chained)
{
    if (phase == 0) return launch(density_lanes_kernel, n_tiles, kThreads, st, pdl, S, chained);
    return launch(force_lanes_kernel, n_tiles, kThreads, st, pdl, S);
}

}  // namespace sph
