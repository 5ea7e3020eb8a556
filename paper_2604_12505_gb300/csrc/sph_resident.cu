// sph_resident.cu -- many steps of small tanks in one launch.
//
// A tank of up to 2,128 particles leaves most of the GPU idle, and a step of
// three launches is a chain of L2 round trips and, with a thread per particle,
// of long loops in few warps (25 us for 938 particles, 44 for the paper's
// 2,024; with four lanes per particle 19 and 25).  Here a cluster of CTAs
// keeps one tank's state in its shared memory from step to step, with four
// lanes per particle: 11 and 16 to 18 us.  The 4x4-cell tiles of the step kernels are
// dealt out to the CTAs (by particle count, when the kernel starts); a CTA
// holds the particles of its tiles and of the cells around them, sends a
// particle's new state to every CTA that will need it, and its density to
// those that hold it as a neighbour, through distributed shared memory.  A
// step is
//   sort      the received particles by cell, each cell by (x, index)
//   density   Eqs. 14, 11 of the own particles
//   -- cluster barrier: densities of the neighbours' particles --
//   force     Eqs. 10, 12, 16-19, kick then drift, new states sent
//   -- cluster barrier: new states, fluid force and torque sums --
//   body      Eq. 20 and the controller, by one warp of every CTA alike
// The body's update and the next sort overlap; what of it needs no fluid force
// is done beside the force pass.
//
// The arithmetic is that of density_kernel<4,4>, force_kernel<4,4> and
// body_kernel, in their order: the lanes of a particle evaluate sixteen
// candidates at once, four each, and then add them up one lane after the other,
// a tile's force sums run over the same lanes in the same tree, and the tank's
// sums are integers.  Results equal theirs bit for bit, so a tank gives the
// same whether it runs here or in a batch that does not fit.  Where the
// compiler could contract a product and a sum in more than one way, the
// rounding is written out.
//
// What bounds it: latency, and the fullest CTA.  Of a step's 37,000 cycles
// (the paper's tank, 4 to 5 warps a scheduler at work), the sort and the ghosts
// take 4,500, the density 10,000, the force 11,000, the sums 4,000 and the
// barriers with the wait for the fullest CTA 7,500.  Not faster: one lane per particle
// (87,000 cycles, long chains in few warps); a broadcast of every candidate to
// all four lanes (60,000, bound by the shuffles); 24 warps of 80 registers
// (2 % and -7 %); the neighbours in reach listed by the density pass for the
// force pass (force loop 6,800 -> 4,700 cycles, density loop 3,900 -> 5,000).
//
// Every buffer is sized for all of the tank's particles in one CTA: wherever
// the fluid goes, nothing overflows.  That bounds the tanks this kernel takes
// (resident_fits).  A tile with more particles around it than the step kernels
// stage raises SPH_FLAG_STAGE_FULL as it does there, so that a tank is not
// accepted or refused by the length of the call.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "sph_body.cuh"
#include "sph_common.cuh"
#include "sph_lanes.cuh"
#include "sph_launch.h"
#include "sph_tile.cuh"

namespace sph {

namespace {

constexpr int kThreads = 640, kWarps = kThreads / 32;
constexpr int kLanes = 4;           // lanes per particle
constexpr int kSlots = kThreads / kLanes;  // particles that a pass takes at once
constexpr int kSortThreads = kThreads - 32;  // the last warp updates the body meanwhile
constexpr int kTile = 4;            // cells per tile side, as the default tile of the step kernels
constexpr int kTileThreads = 128;   // threads that a tile has there: own particle t is summed by thread t % 128
constexpr int kStage = Shape<kTile, kTile>::MAXS;  // particles that a tile stages there, with its halo
constexpr int kMine = 4;            // particles of a sorting thread
constexpr unsigned short kNone = 0xffff;
constexpr unsigned kOwn = 1u << 31;

// The largest tank, by what the shared memory of an SM holds if all of the
// fluid gathers in one CTA's tiles: particles, ghosts, cells along a side.
constexpr int kMaxFluid = 2128, kMaxGhosts = 704, kMaxG = 30;
constexpr int kMaxTiles = (kMaxG + kTile - 1) / kTile * ((kMaxG + kTile - 1) / kTile);
// The grid is padded by a cell all round, so that a stencil never leaves it.
constexpr int kMaxCells = (kMaxG + 2) * (kMaxG + 2);
static_assert(kMaxFluid <= kMine * kSortThreads && kMaxFluid < kNone, "the sort's threads and 16-bit indices");

struct Mem {
    float4 in_pv[kMaxFluid];         // received, by particle index: state, low parts (and cell)
    float4 in_lo[kMaxFluid];
    float4 s_pv[kMaxFluid];          // sorted
    float4 g_b[kMaxGhosts];          // ghosts: body frame, world position, velocity and arm
    float4 g_p[kMaxGhosts];
    float4 g_v[kMaxGhosts];
    float2 s_plo[kMaxFluid];
    union {
        float2 s_rho[kMaxFluid];     // (rho, P / rho^2)
        unsigned long long key[kMaxFluid];  // before: the sort's keys
        Red red[4 * kMaxTiles];      // after: the tiles' force sums
    };
    union {
        float2 r_rho[kMaxFluid];     // received densities, by particle index
        float2 w_xy[kMaxFluid];      // after they are taken over: the own particles' force on the body
    };
    float w_t[kMaxFluid];            // and torque
    unsigned cnt[kMaxCells];
    unsigned hold[kMaxCells];        // the CTAs that hold a cell's particles; kOwn: this one owns it
    unsigned short gstart[kMaxG * kMaxG + 1];
    unsigned short start[kMaxCells + 1];   // sorted particles before each cell, and own ones
    unsigned short ostart[kMaxCells + 1];
    unsigned short in_cell[kMaxFluid];     // kNone: not received
    unsigned short own[kMaxFluid];         // sorted index of each own particle
    unsigned short s_id[kMaxFluid];
    unsigned short s_cell[kMaxFluid];
    unsigned short weight[kMaxTiles];
    unsigned char owner[kMaxTiles];
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cta_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// The address of another CTA's shared memory in this cluster.
__device__ __forceinline__ unsigned remote(unsigned local, int rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void put(unsigned at, float4 v)
{
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}
__device__ __forceinline__ void put(unsigned at, float2 v)
{
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(at), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void put(unsigned at, unsigned short v)
{
    asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(at), "h"(v) : "memory");
}
__device__ __forceinline__ void put(unsigned at, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(at), "l"(v) : "memory");
}
// All CTAs of the cluster: what was written before, to any of them, is seen after.
__device__ __forceinline__ void cluster_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void sort_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kSortThreads) : "memory"); }

// First indices in [lo0, hi0) and [lo1, hi1) of a list sorted by x whose x is
// not below v0, v1.
__device__ __forceinline__ void lower(const float4* l, int& lo0, int hi0, float v0, int& lo1, int hi1, float v1)
{
    while (hi0 - lo0 > 31 && l[lo0 + 31].x < v0) lo0 += 32;
    while (hi1 - lo1 > 31 && l[lo1 + 31].x < v1) lo1 += 32;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        if (lo0 + s <= hi0 && l[lo0 + s - 1].x < v0) lo0 += s;
        if (lo1 + s <= hi1 && l[lo1 + s - 1].x < v1) lo1 += s;
    }
}

// What the tile passes read of the body, as the body record holds it:
// cos, sin, r', rdot', thetadot' and the origin of the next grid, each as
// (hi, lo), at the place of its output in the body's update.
struct Frame {
    float2 v[10];
    __device__ GhostFrame ghosts() const { return {v[8], v[9], v[0], v[1], v[3].x, v[4].x, v[5].x}; }
};

static_assert(sizeof(TankDev) % 4 == 0 && sizeof(TankDev) / 4 <= kThreads, "one word per thread");

template <int CL>
struct Shared {
    TankDev T;
    RunDev run;
    Frame frame;
    // the body, by output of its update: its state, the plan of the update;
    // in shared memory, as registers of the whole CTA are short
    double state[10], anchor[2], tau_c;
    BodyPlan plan[10];
    double* y;                             // this step's sample, or null
    unsigned long long sums[CL][5];        // per CTA: fluid force, torque, position sums
    unsigned long long part[5];            // this CTA's
    int n_tile;                            // own tiles
    unsigned short at[kMaxTiles];          // own tiles: first cell,
    unsigned short row[kMaxTiles][kTile + 1];   // particles before each of their rows,
    unsigned char across[kMaxTiles];       // cells across
    unsigned char down[kMaxTiles];         // and down
    unsigned scan[32];
    int most;                              // particles of the fullest own tile
    float damp;
    int flags;
};
static_assert(sizeof(Mem) + sizeof(Shared<16>) + 256 <= 227 * 1024, "the shared memory of an SM");

}  // namespace

bool resident_fits(int n_f, int n_g, int G) { return n_f <= kMaxFluid && n_g <= kMaxGhosts && G <= kMaxG; }

template <int CL>
__global__ void __launch_bounds__(kThreads, 1) resident_kernel(SimDev S, int n_steps)
{
    extern __shared__ __align__(16) unsigned char mem[];
    Mem& M = *reinterpret_cast<Mem*>(mem);
    __shared__ Shared<CL> sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cta_rank(), tank = blockIdx.x / CL;
    if (tid < (int)(sizeof(TankDev) / 4)) reinterpret_cast<int*>(&sh.T)[tid] = reinterpret_cast<const int*>(S.tank + tank)[tid];
    if (tid == 0) {
        sh.run = *S.run;
        sh.n_tile = 0;
        sh.flags = 0;
        sh.damp = 1.0f - S.run->damping;
    }
    __syncthreads();
    const TankDev& T = sh.T;
    const int G = T.G, P = G + 2, nt = (G + kTile - 1) / kTile, n_g = T.n_g;
    const int cells = P * P, tiles = nt * nt;
    float4 *const in_pv = M.in_pv, *const in_lo = M.in_lo, *const s_pv = M.s_pv, *const g_b = M.g_b, *const g_p = M.g_p, *const g_v = M.g_v;
    float2 *const s_plo = M.s_plo, *const s_rho = M.s_rho, *const r_rho = M.r_rho, *const w_xy = M.w_xy;
    float *const w_t = M.w_t;
    unsigned long long *const key = M.key;
    Red *const red = M.red;
    unsigned *const cnt = M.cnt, *const hold = M.hold;
    unsigned short *const gstart = M.gstart, *const start = M.start, *const ostart = M.ostart, *const in_cell = M.in_cell, *const own = M.own, *const s_id = M.s_id, *const s_cell = M.s_cell, *const weight = M.weight;
    unsigned char *const owner = M.owner;

    const RunDev& run = sh.run;
    const long long step_first = run.step;
    int buf = (int)(step_first & 1);

    // ------------------------------------------------------------------
    // start: ghosts, cell counts, the tiles' owners, this CTA's particles
    // ------------------------------------------------------------------
    for (int g = tid; g < n_g; g += kThreads) g_b[g] = __ldg(S.gB + T.ghost_base + g);
    for (int c = tid; c <= G * G; c += kThreads) gstart[c] = (unsigned short)(__ldg(S.gstart + T.gcell_base + c) - T.ghost_base);
    for (int c = tid; c < cells; c += kThreads) {
        const int x = c % P - 1, y = c / P - 1;
        const bool in = x >= 0 && x < G && y >= 0 && y < G;
        cnt[c] = in ? min(max(__ldcg(S.count[buf] + T.cell_base + y * G + x), 0), kCap) : 0;
    }
    for (int e = tid; e < T.n_f; e += kThreads) in_cell[e] = kNone;
    __syncthreads();
    for (int i = tid; i < tiles; i += kThreads) {  // particles of each tile
        int n = 0;
        for (int r = 0; r < kTile; ++r)
            for (int q = 0; q < kTile; ++q) {
                const int x = (i % nt) * kTile + q, y = (i / nt) * kTile + r;
                if (x < G && y < G) n += cnt[(y + 1) * P + x + 1];
            }
        weight[i] = (unsigned short)n;
    }
    __syncthreads();
    // The tiles in order, cut into CL parts of at most `cap` particles each, the
    // smallest cap of the 32 that the lanes try: the same in every CTA.
    if (warp == 0) {
        int total = 0, most = 0;
        for (int i = lane; i < tiles; i += 32) {
            total += weight[i];
            most = max(most, (int)weight[i]);
        }
        total = __reduce_add_sync(0xffffffffu, total);
        most = max(__reduce_max_sync(0xffffffffu, most), (total + CL - 1) / CL);
        const int cap = most + (lane * most + 15) / 16;  // the last: nearly 3 times the mean, always enough
        int part = 0, in = 0;
        for (int i = 0; i < tiles; ++i) {
            if (in + weight[i] > cap) {
                ++part;
                in = 0;
            }
            in += weight[i];
        }
        const int best = __ffs(__ballot_sync(0xffffffffu, part < CL)) - 1;
        if (lane == best) {
            part = in = 0;
            for (int i = 0; i < tiles; ++i) {
                if (in + weight[i] > cap) {
                    ++part;
                    in = 0;
                }
                in += weight[i];
                owner[i] = (unsigned char)part;
            }
        }
    }
    __syncthreads();
    // own tiles; the CTAs that hold a cell's particles are the owners of the
    // tiles that the cells around it lie in
    for (int i = tid; i < tiles; i += kThreads)
        if (owner[i] == rank) {
            const int j = atomicAdd(&sh.n_tile, 1), x = (i % nt) * kTile, y = (i / nt) * kTile;
            sh.at[j] = (unsigned short)((y + 1) * P + x + 1);
            sh.across[j] = (unsigned char)min(kTile, G - x);
            sh.down[j] = (unsigned char)min(kTile, G - y);
        }
    for (int c = tid; c < cells; c += kThreads) {
        const int x = c % P - 1, y = c / P - 1;
        unsigned h = 0u;
        if (x >= 0 && x < G && y >= 0 && y < G) {
            const int x0 = max(x - 1, 0) / kTile, x1 = min(x + 1, G - 1) / kTile;
            const int y0 = max(y - 1, 0) / kTile, y1 = min(y + 1, G - 1) / kTile;
            h = (1u << owner[y0 * nt + x0]) | (1u << owner[y0 * nt + x1]) | (1u << owner[y1 * nt + x0]) |
                (1u << owner[y1 * nt + x1]);
            if (owner[(y / kTile) * nt + x / kTile] == rank) h |= kOwn;
        }
        hold[c] = h;
    }
    __syncthreads();
    for (int u = tid; u < cells * kCap; u += kThreads) {  // a cell's particles, if held
        const int c = u / kCap, q = u - c * kCap;
        if (q >= (int)cnt[c] || !(hold[c] >> rank & 1u)) continue;
        const int gs = (T.cell_base + (c / P - 1) * G + c % P - 1) * kCap + q;
        const int id = __ldcg(S.pid[buf] + gs) - T.pid_base;
        in_pv[id] = __ldcg(S.pv[buf] + gs);
        in_lo[id] = __ldcg(S.lo[buf] + gs);
        in_cell[id] = (unsigned short)c;
    }
    __syncthreads();
    for (int c = tid; c < cells; c += kThreads) cnt[c] = 0;
    // the body: a lane of the last warp holds output l of its update (body_plan)
    const bool body_warp = warp == kWarps - 1;
    const bool ctrl_on = run.ctrl_on != 0, body_fixed = run.body_fixed != 0;
    const BodyDev& b0 = S.body[tank];
    if (body_warp) {
        if (lane < 6) sh.state[lane] = reinterpret_cast<const double*>(&b0)[lane];
        if (lane == 8) sh.state[8] = b0.c;
        if (lane == 9) sh.state[9] = b0.s;
        if (lane == 10) sh.tau_c = b0.tau_c;
        if (lane == 0)
            sh.frame = Frame{{b0.drx, b0.dry, {0.f, 0.f}, {b0.fvx, 0.f}, {b0.fvy, 0.f}, {b0.fw, 0.f}, {b0.fo_next[0], 0.f},
                              {b0.fo_next[1], 0.f}, b0.dc, b0.ds}};
    }
    unsigned pairs_sum = 0;  // of this thread: at most a tank's pairs a step, by the steps of a launch
    cluster_sync();  // every CTA has read the state, and may be written to

    // sorted index of particle t of own tile i
    auto tile_at = [&](int i, int t) {
        const unsigned short* r = sh.row[i];
        int q = 0;
#pragma unroll
        for (int k = 1; k < kTile; ++k) q += t >= (int)r[k];
        return (int)start[(int)sh.at[i] + q * P] + t - (int)r[q];
    };
    const int sub = lane & (kLanes - 1);
    // The sorted particles around a particle in cell c, clipped to the support.
    auto stencil = [&](bool on, int c, float x) {
        int a = 0, z = 0;
        if (on && sub < 3) {
            const int cl = c + (sub - 1) * P - 1;
            a = start[cl];
            z = start[cl + 2];
            lower(s_pv, a, start[cl + 1], x - T.clip, z, start[cl + 3], x + T.clip);
        }
        return lane_runs<kLanes>(pack_run(a, z));
    };
    // The ghosts within clip, as for_staged_ghosts visits them.
    auto ghost_rows = [&](bool on, float xi, float yi, float clip) {
        const Frame& F = sh.frame;
        int gx, gy, a = 0, b = 0;
        float ex, ey;
        const bool any = on && ghost_cell(T, xi, yi, F.v[8].x, F.v[9].x, F.v[0].x, F.v[1].x, gx, gy, ex, ey);
        if (any && sub < 3) {
            const int x0 = max(gx - 1, 0), x1 = min(gx + 1, G - 1), yy = gy - 1 + sub;
            if (x0 <= x1 && yy >= 0 && yy <= G - 1) {
                const float ylo = T.g_orig + (float)yy * T.g_cell;
                const bool away = yy > 0 && yy < G - 1 && (ylo > ey + clip || ylo + T.g_cell < ey - clip);
                if (!away) {
                    a = gstart[yy * G + x0];
                    b = gstart[yy * G + x1 + 1];
                    if (x0 > 0 && x1 < G - 1) {
                        int z = a;
                        lower(g_b, a, b, ex - clip, z, b, ex + clip);
                        b = z;
                    }
                }
            }
        }
        return lane_runs<kLanes>(pack_run(a, b));
    };

    const unsigned a_pv = smem_addr(in_pv), a_lo = smem_addr(in_lo), a_cell = smem_addr(in_cell), a_rho = smem_addr(r_rho);
    const int oe = T.outer_every;
    int phase = (int)(step_first % oe);  // 0 at a sample
    // the next sample's place among the run's
    long long n_sample = (step_first + oe - 1) / oe - (run.step0 + oe - 1) / oe;

    for (int k = 0; k < n_steps; ++k) {
        const bool sample = phase == 0;
        // --------------------------------------------------------------
        // sort by cell and (x, index); the last warp updates the body
        // --------------------------------------------------------------
        if (!body_warp) {
            if (tid < 5) sh.part[tid] = 0ull;
            int c_in[kMine], slot[kMine];
#pragma unroll
            for (int q = 0; q < kMine; ++q) {
                const int e = tid + q * kSortThreads;
                c_in[q] = e < T.n_f ? in_cell[e] : kNone;
            }
#pragma unroll
            for (int q = 0; q < kMine; ++q)
                if (c_in[q] != kNone) slot[q] = (int)atomicAdd(&cnt[c_in[q]], 1u);
            sort_sync();
            // running sums over the cells: all in the low half, own in the high
            constexpr int kPer = 2;
            unsigned before = 0;
            for (int c0 = 0; c0 < cells; c0 += kPer * kSortThreads) {
                unsigned v[kPer], sum = 0;
#pragma unroll
                for (int q = 0; q < kPer; ++q) {
                    const int c = c0 + kPer * tid + q;
                    v[q] = 0;
                    if (c < cells) {
                        v[q] = cnt[c] | (hold[c] & kOwn ? cnt[c] << 16 : 0u);
                        cnt[c] = 0;
                    }
                    sum += v[q];
                }
                unsigned incl = sum;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (lane == 31) sh.scan[warp] = incl;
                sort_sync();
                const unsigned w = lane < kWarps - 1 ? sh.scan[lane] : 0u;
                unsigned at = before + incl - sum + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
                before += __reduce_add_sync(0xffffffffu, w);
#pragma unroll
                for (int q = 0; q < kPer; ++q) {
                    const int c = c0 + kPer * tid + q;
                    if (c <= cells) {
                        start[c] = (unsigned short)(at & 0xffffu);
                        ostart[c] = (unsigned short)(at >> 16);
                    }
                    at += v[q];
                }
                sort_sync();
            }
            if (tid == 0) {
                start[cells] = (unsigned short)(before & 0xffffu);
                ostart[cells] = (unsigned short)(before >> 16);
            }
#pragma unroll
            for (int q = 0; q < kMine; ++q)
                if (c_in[q] != kNone) {
                    const int e = tid + q * kSortThreads;
                    key[start[c_in[q]] + slot[q]] = (unsigned long long)order_key(in_pv[e].x) << 16 | (unsigned)e;
                }
            sort_sync();
            const int n_in = (int)start[cells];
            for (int q = tid; q < n_in; q += kSortThreads) {
                const unsigned long long ke = key[q];
                const int e = (int)(ke & 0xffffu), c = in_cell[e], a = start[c], z = start[c + 1];
                const float4 p = in_pv[e], lo = in_lo[e];
                int d = a;
                for (int j = a; j < z; ++j) d += key[j] < ke;
                if (z - a > kCap) atomicOr(&sh.flags, SPH_FLAG_CELL_FULL);
                s_pv[d] = p;
                s_plo[d] = make_float2(lo.x, lo.y);
                s_id[d] = (unsigned short)e;
                s_cell[d] = (unsigned short)c;
                in_cell[e] = kNone;
                if (hold[c] & kOwn) own[ostart[c] + d - a] = (unsigned short)d;
            }
        }
        __syncthreads();
        // --------------------------------------------------------------
        // ghosts (Eq. 21), then the density of the own particles (Eqs. 14, 11)
        // --------------------------------------------------------------
        const int n_in = (int)start[cells], n_own = (int)ostart[cells];
        for (int g = tid; g < n_g; g += kThreads) ghost_world(sh.frame.ghosts(), g_b[g], g_p[g], g_v[g]);
        if (tid == 0) {
            sh.most = 0;
        }
        __syncthreads();
        // the rows of the own tiles, for their sums
        if (const int i = kThreads - 1 - tid; i < sh.n_tile) {
            int acc = 0, around = 0;
            const int at = sh.at[i], wide = sh.across[i], high = sh.down[i];
#pragma unroll
            for (int r = -1; r <= kTile; ++r) {
                const int c = at + r * P;
                if (r >= 0) sh.row[i][r] = (unsigned short)acc;
                if (r >= 0 && r < high) acc += (int)start[c + wide] - (int)start[c];
                if (r <= high) around += (int)start[c + wide + 1] - (int)start[c - 1];
            }
            // a tank that the step kernels cannot stage is refused here too
            if (acc > 0 && around > kStage) atomicOr(&sh.flags, SPH_FLAG_STAGE_FULL);
            if (acc > kTileThreads) atomicMax(&sh.most, acc);
        }
        const int first = warp * (32 / kLanes);  // the warp's first particle, and this lane's
        const int mine = tid / kLanes;
        auto keep = [](unsigned* p, const Runs& R) {
            p[0] = (unsigned)R.o0 | (unsigned)R.n0 << 16;
            p[1] = (unsigned)(R.o1 + R.n0) | (unsigned)(R.n1 - R.n0) << 16;
            p[2] = (unsigned)(R.o2 + R.n1) | (unsigned)(R.n - R.n1) << 16;
        };
        unsigned kept[6];  // the first pass's runs, of particles and of ghosts, for the force
        for (int p = 0; first + p < n_own; p += kSlots) {  // by whole warps
            const bool on = mine + p < n_own;
            const int e = on ? own[mine + p] : 0;
            const int c = s_cell[e];
            const float4 pi = s_pv[e];
            const float2 li = s_plo[e];
            const Runs R = stencil(on, c, pi.x);
            if (p == 0) keep(kept, R);
            float Sf = fluid_sum<kLanes>(T, R, e, pi, li, s_pv, s_plo, sub);
            Sf = __fmul_rn(Sf, T.cW);
            const Runs Q = ghost_rows(on, pi.x, pi.y, T.clip);
            if (p == 0) keep(kept + 3, Q);
            const float Sg = ghost_sum<kLanes>(T, Q, pi, li, g_p, sub);
            const float rho = __fmul_rn(T.m, __fmaf_rn(T.gamma1, Sg, Sf));       // Eq. 14
            const float Pr = __fmul_rn(T.k, __fsub_rn(rho, T.rho0));              // Eq. 11
            const float2 v = make_float2(rho, __fdiv_rn(Pr, __fmul_rn(rho, rho)));
            if (on && sub == 0) {
                s_rho[e] = v;
                unsigned to = hold[c] & ~(kOwn | 1u << rank);
                while (to) {
                    const int r = __ffs(to) - 1;
                    to &= to - 1;
                    put(remote(a_rho + 8u * s_id[e], r), v);
                }
            }
        }
        cluster_sync();
        for (int e = tid; e < n_in; e += kThreads)
            if (!(hold[s_cell[e]] & kOwn)) s_rho[e] = r_rho[s_id[e]];
        __syncthreads();
        // --------------------------------------------------------------
        // force, kick then drift; the new states to whoever will need them
        // --------------------------------------------------------------
        const float damp = sh.damp;
        int flags = 0;
        for (int p = 0; first + p < n_own; p += kSlots) {
            const bool on = mine + p < n_own;
            const int e = on ? own[mine + p] : 0;
            const float4 pi = s_pv[e];
            const float2 li = s_plo[e], ri = s_rho[e];
            const Runs R = p == 0 ? unpack_runs(kept[0], kept[1], kept[2]) : stencil(on, s_cell[e], pi.x);
            float ax = 0.f, ay = 0.f;
            int nff = fluid_forces<kLanes>(T, R, e, pi, li, ri, s_pv, s_plo, s_rho, sub, ax, ay);
            BothSum W{{0.f, 0.f, 0.f}, ax, ay, T.inv_m};
            const Runs Q = p == 0 ? unpack_runs(kept[3], kept[4], kept[5]) : ghost_rows(on, pi.x, pi.y, T.clip);
            nff += ghost_forces<kLanes>(T, Q, pi, li, ri, g_p, g_v, sub, W);
            ax = W.ax;
            ay = W.ay;
            pairs_sum += (unsigned)nff;
            if (on && sub == 0) {
                w_xy[e] = make_float2(W.fx, W.fy);
                w_t[e] = W.t;
            }
            ax += T.grav_x;
            ay += T.grav_y;
            // kick then drift (Section 3.4) on the two-float state
            const unsigned short id = s_id[e];
            const float2 vl = make_float2(in_lo[id].z, in_lo[id].w);
            float2 kx = two_sum(pi.z, fmaf(T.dt, ax, vl.x)), ky = two_sum(pi.w, fmaf(T.dt, ay, vl.y));
            if (damp != 1.0f) {  // relaxation: scale the two-float velocity
                const float hx = kx.x * damp, hy = ky.x * damp;
                kx = two_sum(hx, fmaf(kx.x, damp, -hx) + kx.y * damp);
                ky = two_sum(hy, fmaf(ky.x, damp, -hy) + ky.y * damp);
            }
            const float2 dx2 = two_sum(pi.x, fmaf(T.dt, kx.x, fmaf(T.dt, kx.y, li.x)));
            const float2 dy2 = two_sum(pi.y, fmaf(T.dt, ky.x, fmaf(T.dt, ky.y, li.y)));
            const float x = dx2.x, y = dy2.x;
            if (on && !(isfinite(x) && isfinite(y) && isfinite(kx.x) && isfinite(ky.x))) flags |= SPH_FLAG_NAN;
            const float ox = sh.frame.v[6].x, oy = sh.frame.v[7].x;
            bool out = false;
            const int ccx = cell_coord(x, ox, T.inv_cell, G, &out);
            const int ccy = cell_coord(y, oy, T.inv_cell, G, &out);
            const float ex = x - (ox + T.Wf), ey = y - (oy + T.Wf);
            if (on && (out || fmaf(ex, ex, ey * ey) > T.cover2)) flags |= SPH_FLAG_ESCAPED;
            const float4 pv = make_float4(x, y, kx.x, ky.x), lo = make_float4(dx2.y, dy2.y, kx.y, ky.y);
            const unsigned short ncell = (unsigned short)((ccy + 1) * P + ccx + 1);
            __syncwarp();  // the low parts are read
            for (unsigned to = on ? hold[ncell] & ~kOwn : 0u; to; to &= to - 1) {  // a lane for each part
                const int r = __ffs(to) - 1;
                if (sub == 0) put(remote(a_pv + 16u * id, r), pv);
                if (sub == 1) put(remote(a_lo + 16u * id, r), lo);
                if (sub == 2) put(remote(a_cell + 2u * id, r), ncell);
            }
        }
        // the body's update as far as the fluid force is not needed
        if (body_warp) {
            const double* q = sh.state;
            const double rx = q[0], ry = q[1], th = q[2], vx = q[3], vy = q[4], w = q[5], c = q[8], sn = q[9];
            double* y = nullptr;
            double tau_c = sh.tau_c;
            double ux = 0.0, uy = 0.0, ut = 0.0, ref = 0.0;
            if (run.u) {
                const double* up = run.u + tank * run.u_tank_stride + 3 * (step_first + k - run.step0);
                ux = up[0];
                uy = up[1];
                ut = up[2];
            }
            if (run.theta_ref && sample) ref = run.theta_ref[tank * run.ref_stride + n_sample];
            if (sample) {
                y = run.y ? run.y + tank * run.y_tank_stride + n_sample * SPH_NY : nullptr;
                if (y && rank == 0 && lane < 6) y[lane] = pick(lane, 0, rx, ry, th, vx, vy, w);
                if (ctrl_on) {
                    const double cJ = run.ctrl_J, cw = run.ctrl_w, cxi = run.ctrl_xi;
                    const double Jc = cJ > 0.0 ? cJ : T.J_body;
                    tau_c = Jc * cw * cw * (ref - th) - 2.0 * cxi * Jc * cw * w;
                }
            }
            const double tau = ut + (ctrl_on ? tau_c : 0.0);
            const BodyPlan plan = body_plan(T, lane, 0, body_fixed, rx, ry, th, vx, vy, w, c, sn, ux, uy, tau);
            if (lane < 10) sh.plan[lane] = plan;
            if (lane < 2) sh.anchor[lane] = lane ? ry : rx;  // the position before the step
            if (lane == 0) {
                sh.tau_c = tau_c;
                sh.y = y;
            }
            __syncwarp();
        }
        if (flags) atomicOr(&sh.flags, flags);
        __syncthreads();
        // A tile thread's sum runs on from its particle t to its next, t + 128:
        // where both met ghosts, the later one's is taken again from there.
        for (int t0 = kTileThreads; t0 < sh.most; t0 += kTileThreads) {
            for (int i = 0, job = 0; i < sh.n_tile; ++i)
                for (int t1 = t0; t1 < min((int)sh.row[i][kTile], t0 + kTileThreads); t1 += 32 / kLanes, ++job) {
                    if (job % kWarps != warp) continue;
                    const int t = t1 + lane / kLanes;
                    bool on = t < (int)sh.row[i][kTile];
                    int e = 0;
                    WallSum W{0.f, 0.f, 0.f};
                    if (on) {
                        const int before = tile_at(i, t - kTileThreads);
                        e = tile_at(i, t);
                        W.fx = w_xy[before].x;
                        W.fy = w_xy[before].y;
                        W.t = w_t[before];
                        on = W.fx != 0.f || W.fy != 0.f || W.t != 0.f;
                    }
                    if (!__any_sync(0xffffffffu, on)) continue;
                    const float4 pi = s_pv[e];
                    ghost_forces<kLanes>(T, ghost_rows(on, pi.x, pi.y, T.hclip), pi, s_plo[e], s_rho[e], g_p, g_v, sub, W);
                    if (on && sub == 0) {
                        w_xy[e] = make_float2(W.fx, W.fy);
                        w_t[e] = W.t;
                    }
                }
            __syncthreads();
        }
        // the tiles' sums in the tree of their four warps, then as integers
        for (int j = warp; j < 4 * sh.n_tile; j += kWarps) {
            const int i = j >> 2, n = sh.row[i][kTile], t = (j & 3) * 32 + lane;
            if ((j & 3) * 32 >= n) continue;
            const F2 z{0.f, 0.f};
            Red acc{z, z, z, z, z, 0ull};
            if (t < n) {
                const int last = tile_at(i, t + (n - 1 - t) / kTileThreads * kTileThreads);
                const float2 w = w_xy[last];
                acc.fx.hi = w.x;
                acc.fy.hi = w.y;
                acc.t.hi = w_t[last];
                if (sample)
                    for (int q = t; q < n; q += kTileThreads) {
                        const float4 p = s_pv[tile_at(i, q)];
                        acc.cx.hi += p.x;
                        acc.cy.hi += p.y;
                    }
            }
            const bool wall = __any_sync(0xffffffffu, acc.fx.hi != 0.f || acc.fy.hi != 0.f || acc.t.hi != 0.f);
            // warp_reduce, as a loop: its code is executed once a step
            for (int o = 16; o > 0 && wall; o >>= 1) {
                acc.fx = f2_add(acc.fx, shfl_down_f2(acc.fx, o));
                acc.fy = f2_add(acc.fy, shfl_down_f2(acc.fy, o));
                acc.t = f2_add(acc.t, shfl_down_f2(acc.t, o));
            }
            for (int o = 16; o > 0 && sample; o >>= 1) {
                acc.cx = f2_add(acc.cx, shfl_down_f2(acc.cx, o));
                acc.cy = f2_add(acc.cy, shfl_down_f2(acc.cy, o));
            }
            if (lane == 0) red[j] = acc;
        }
        __syncthreads();
        for (int q = tid; q < 5 * sh.n_tile; q += kThreads) {
            const int i = q / 5, c = q - 5 * i, n = sh.row[i][kTile];
            if (n == 0 || (c >= 3 && !sample)) continue;
            const F2 z{0.f, 0.f};
            auto r = [&](int w) { return w * 32 < n ? (&red[4 * i + w].fx)[c] : z; };
            const F2 v = f2_add(f2_add(r(0), r(2)), f2_add(r(1), r(3)));
            const long long x = __float2ll_rn(v.hi * kFixScale) + __float2ll_rn(v.lo * kFixScale);
            if (x) atomicAdd(&sh.part[c], (unsigned long long)x);
        }
        __syncthreads();
        if (tid < 5 * CL) put(remote(smem_addr(&sh.sums[rank][tid % 5]), tid / 5), sh.part[tid % 5]);
        cluster_sync();
        // --------------------------------------------------------------
        // the body (Eq. 20, Eq. 28): every CTA alike, the first one samples
        // --------------------------------------------------------------
        if (body_warp) {
            double vq = 0.0;
            if (lane < 5) {
                unsigned long long sum = 0ull;
#pragma unroll
                for (int r = 0; r < CL; ++r) sum += sh.sums[r][lane];
                vq = (double)(long long)sum * kFixUnit;
            }
            const double Fx = __shfl_sync(0xffffffffu, vq, 0), Fy = __shfl_sync(0xffffffffu, vq, 1);
            const double Tq = __shfl_sync(0xffffffffu, vq, 2), Cx = __shfl_sync(0xffffffffu, vq, 3);
            const double Cy = __shfl_sync(0xffffffffu, vq, 4);
            double* const y = sh.y;
            const double v = body_apply(sh.plan[lane < 10 ? lane : 0], lane, 0, body_fixed, Fx, Fy, Tq);
            if (y && rank == 0 && lane >= 6 && lane < SPH_NY) {
                double o = sel3(lane - 6, Fx, Fy, Tq);
                if (lane >= 9) o = T.n_f ? (lane == 9 ? Cx : Cy) / T.n_f : 0.0;
                y[lane] = o;
            }
            if (!body_fixed && lane < 10) sh.state[lane] = v;
            const float hi = (float)v, lo = (float)(v - (double)hi);
            if (lane < 10) sh.frame.v[lane] = make_float2(hi, lo);
        }
        buf ^= 1;
        n_sample += sample;
        if (++phase == oe) phase = 0;
    }
    __syncthreads();
    // ------------------------------------------------------------------
    // end: the state back into the grid of the next step's buffer
    // ------------------------------------------------------------------
    for (int c = rank * kThreads + tid; c < G * G; c += CL * kThreads) S.count[buf][T.cell_base + c] = 0;
    cluster_sync();
    for (int e = tid; e < T.n_f; e += kThreads) {
        const int c = in_cell[e];
        if (c == kNone || !(hold[c] & kOwn)) continue;
        const int gc = T.cell_base + (c / P - 1) * G + (c % P - 1);
        const int q = atomicAdd(&S.count[buf][gc], 1);
        if ((unsigned)q < (unsigned)kCap) {
            S.pv[buf][gc * kCap + q] = in_pv[e];
            S.lo[buf][gc * kCap + q] = in_lo[e];
            S.pid[buf][gc * kCap + q] = T.pid_base + e;
        } else {
            atomicOr(&sh.flags, SPH_FLAG_CELL_FULL);
        }
    }
    unsigned long long pairs = pairs_sum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) pairs += __shfl_down_sync(0xffffffffu, pairs, o);
    BodyDev& b = S.body[tank];
    if (lane == 0 && pairs) atomicAdd(&b.pairs, pairs);
    __syncthreads();
    if (tid == 0 && sh.flags) atomicOr(&b.flags, sh.flags);
    if (rank == 0 && body_warp && n_steps > 0) {
        if (!body_fixed && (lane < 6 || lane == 8 || lane == 9)) reinterpret_cast<double*>(&b)[lane < 6 ? lane : lane - 2] = sh.state[lane];
        if (lane < 2) b.anchor[buf][lane] = sh.anchor[lane];
        if (lane == 0) {
            const Frame& F = sh.frame;
            b.dc = F.v[8];
            b.ds = F.v[9];
            b.drx = F.v[0];
            b.dry = F.v[1];
            b.fc = F.v[8].x;
            b.fs = F.v[9].x;
            b.frx = F.v[0].x;
            b.fry = F.v[1].x;
            b.fvx = F.v[3].x;
            b.fvy = F.v[4].x;
            b.fw = F.v[5].x;
            b.fo_next[0] = F.v[6].x;
            b.fo_next[1] = F.v[7].x;
            b.tau_c = sh.tau_c;
        }
    }
}

__global__ void advance_kernel(RunDev* run, int n)
{
    run->step += n;
    run->next_buf = (int)(run->step & 1);
}

namespace {

struct Launch {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    Launch(int B, int CL, cudaStream_t st)
    {
        cfg.gridDim = dim3(B * CL);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = sizeof(Mem);
        cfg.stream = st;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = CL;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
};

}  // namespace

// CTAs per tank: sixteen (the most a cluster can have) while the GPU holds all
// tanks at once, else eight, else none: tanks that wait for a place lose to the
// step kernels (64 of the paper's tanks take those 72 us a step, 12 tanks 35,
// in clusters of eight 22).
cudaError_t prepare_resident(int B, int& cluster)
{
    cudaError_t e = cudaFuncSetAttribute(resident_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Mem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(resident_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Mem));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(resident_kernel<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    int at_once[2] = {};
    const Launch l16(B, 16, nullptr), l8(B, 8, nullptr);
    e = cudaOccupancyMaxActiveClusters(&at_once[0], resident_kernel<16>, &l16.cfg);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&at_once[1], resident_kernel<8>, &l8.cfg);
    cluster = at_once[0] >= B ? 16 : at_once[1] >= B ? 8 : 0;
    return e;
}

cudaError_t launch_resident(const SimDev& S, int cluster, int n_steps, cudaStream_t st)
{
    const Launch l(S.B, cluster, st);
    cudaError_t e = cluster == 16 ? cudaLaunchKernelEx(&l.cfg, resident_kernel<16>, S, n_steps)
                                  : cudaLaunchKernelEx(&l.cfg, resident_kernel<8>, S, n_steps);
    if (e != cudaSuccess) return e;
    advance_kernel<<<1, 1, 0, st>>>(S.run, n_steps);  // after every tank has read where the run stands
    return cudaGetLastError();
}

}  // namespace sph
