// Two time steps in one pass over memory (A/B pattern, FP32 storage).
//
// The one-step kernels stream at the copy bandwidth, so a step cannot get
// faster unless its populations cross DRAM less often.  Here a block owns a
// tile of columns and marches along z: it computes step 1 on the tile and a
// halo of one cell around it, keeps those post-collision values in shared
// memory only, and computes step 2 from them, so that two steps read and
// write every population once.  The halo (32 x 24 cells in step 1 for 30 x 22
// in step 2) is computed again by the neighbouring tiles.  Bitwise the same
// results as two one-step launches.
//
// A warp is one row of 32 columns.  An iteration is: step 1 of plane s from
// registers into shared memory; the loads of plane s + 1 are issued; one
// barrier; step 2 of plane s - 1 from shared memory to the other grid, which
// covers the latency of those loads.
//
// Shared memory holds what step 1 leaves, already streamed in y (a value is
// stored in the row that reads it), in rings over planes: directions with c_z
// = +1 for planes s - 3 ... s, c_z = 0 for s - 2 ... s, c_z = -1 for s - 1 and
// s (a slower warp may still read for step 2 of plane s - 2): 57 values for each
// column of the tile's inner rows.  With walls a value that crosses one is stored
// where its reflection is read, which may be plane s + 1 of c_z = -1: 62.
//
// What bounds it: latency at 24 warps per SM.  It uses 0.63 of the issue slots (413
// instructions a cell and step) and two thirds of the copy bandwidth; the largest
// stall is the wait for the next plane's loads (3.2 warps per issue), whose number the
// registers cap, and the barrier of each plane follows (0.9).  A step, one-step
// kernel -> this one: periodic 256^3 364 -> 289 us, 192^3 155 -> 131; walled
// channel 512x256x256 739 -> 585.  Measured on the way: the loads issued after the
// barrier 328 us at 256^3; 28 rows (72 registers) spill the prefetched plane, 364;
// two rows a thread with packed arithmetic and 16 warps 495, with the plane staged
// by cp.async 532: too few warps to cover the phases.
#pragma once

#include "lbm_step.cuh"

namespace lbm {

constexpr int PAIR_LANES = 32;           // columns of a tile row in step 1, one warp
constexpr int PAIR_TX = PAIR_LANES - 2;  // and in step 2
constexpr int PAIR_SMS = 152;            // one block per SM

// Two FP32 numbers for this GPU's packed instructions (one add, multiply or fma
// of two independent pairs), which have the arithmetic rate of the scalar ones at
// half the issue slots (15.5 against 30.9 thousand billion thread instructions
// per second).  Each component is rounded as the scalar operation rounds it;
// negating an operand costs nothing.
struct __align__(8) F2 {
    float x, y;
    F2() = default;
    __host__ __device__ __forceinline__ F2(float a, float b) : x(a), y(b) {}
    __host__ __device__ explicit __forceinline__ F2(float a) : x(a), y(a) {}
};
__device__ __forceinline__ float2 raw(F2 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ F2 pair_of(float2 a) { return F2(a.x, a.y); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.x, -a.y); }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return pair_of(__fadd2_rn(raw(a), raw(b))); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return pair_of(__fadd2_rn(raw(a), raw(-b))); }
__device__ __forceinline__ F2 &operator+=(F2 &a, F2 b) { return a = a + b; }
__device__ __forceinline__ F2 mul(F2 a, F2 b) { return pair_of(__fmul2_rn(raw(a), raw(b))); }
__device__ __forceinline__ F2 mad(F2 a, F2 b, F2 c) { return pair_of(__ffma2_rn(raw(a), raw(b), raw(c))); }

// The collision of FP32 storage (collide_lean with the one-rounding update and
// the compensated momentum, rho0 = 1) with packed instructions: the x and y face
// pairs, and the two edge pairs of each plane, are the two components (edges (k, k
// + 1) = (3, 4) of the xy plane, (5, 6) of xz, (7, 8) of yz).  Bitwise the same
// results, about 170 instead of 237 operations.
struct RelaxPacked {
    Relax<float> r;
    F2 hp, hm, Kf, Ke, Af, Ae, half_a, force[4];  // each twice, or by the two components
};

static inline RelaxPacked to_packed(const Relax<float> &r)
{
    RelaxPacked p;
    p.r = r;
    p.hp = F2(r.hp);
    p.hm = F2(r.hm);
    p.Kf = F2(r.Kf);
    p.Ke = F2(r.Ke);
    p.Af = F2(r.Af);
    p.Ae = F2(r.Ae);
    p.half_a = F2(r.half_a[0], r.half_a[1]);
    p.force[0] = F2(r.force[0], r.force[1]);
    for (int i = 1; i < 4; ++i) p.force[i] = F2(r.force[2 * i + 1], r.force[2 * i + 2]);
    return p;
}

__device__ __forceinline__ void relax_pairs(F2 &gp, F2 &gm, F2 nsym, F2 nasym, F2 force, const RelaxPacked &p)
{
    const F2 b = mad(p.hm, nasym, -force);
    gp = gp - mad(p.hp, nsym, b);
    gm = gm - mad(p.hp, nsym, -b);
}

__device__ __forceinline__ void collide_packed(float g[Q], const RelaxPacked &p)
{
    const Relax<float> &r = p.r;
    F2 fp(g[1], g[3]), fm(g[2], g[4]);  // faces along x and y
    F2 ep[3], em[3];                    // edges of the xy, xz, yz planes
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        ep[i] = F2(g[7 + 4 * i], g[9 + 4 * i]);
        em[i] = F2(g[8 + 4 * i], g[10 + 4 * i]);
    }
    const F2 sf = fp + fm, df = fp - fm;
    const float sz = g[5] + g[6], dz = g[5] - g[6];
    F2 se[3], de[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        se[i] = ep[i] + em[i];
        de[i] = ep[i] - em[i];
    }
    const float drho = g[0] + (((sf.x + sf.y) + (sz + se[0].x)) + ((se[0].y + se[1].x) + (se[1].y + se[2].x)) + se[2].y);
    F2 u = df, du(0.f, 0.f);  // along x and y, and what rounding u drops
    float uz = dz, duz = 0.f;
    two_sum_acc(u, du, F2(de[0].x, de[0].x));
    two_sum_acc(u, du, F2(de[0].y, -de[0].y));
    two_sum_acc(u, du, F2(de[1].x, de[2].x));
    two_sum_acc(u, du, F2(de[1].y, de[2].y));
    two_sum_acc(u, du, p.half_a);
    two_sum_acc(uz, duz, de[1].x);
    two_sum_acc(uz, duz, -de[1].y);
    two_sum_acc(uz, duz, de[2].x);
    two_sum_acc(uz, duz, -de[2].y);
    two_sum_acc(uz, duz, r.half_a[2]);
    const F2 u2 = mul(u, u);
    const float uz2 = mul(uz, uz), uu = (u2.x + u2.y) + uz2;
    const float base = mad(-1.5f, uu, drho);
    const float Bf = mad(r.wf, base, -mul(r.kf, uu));
    g[0] = mad(-r.wp, g[0] - mad(r.w0, base, mul(r.k0, uu)), g[0]);
    // faces
    const F2 nsym = mad(F2(-2.f), mad(p.Kf, u2, F2(Bf)), sf), nasym = mad(-p.Af, u, df) - du;
    relax_pairs(fp, fm, nsym, nasym, p.force[0], p);
    g[1] = fp.x;
    g[3] = fp.y;
    g[2] = fm.x;
    g[4] = fm.y;
    const float nsz = mad(-2.f, mad(r.Kf, uz2, Bf), sz), naz = mad(-r.Af, uz, dz) - duz;
    const float bz = mad(r.hm, naz, -r.force[2]);
    g[5] = g[5] - mad(r.hp, nsz, bz);
    g[6] = g[6] - mad(r.hp, nsz, -bz);
    // edges of the planes xy, xz, yz; the axis normal to each is z, y, x
    const float a[3] = {u.x, u.x, u.y}, c[3] = {u.y, uz, uz}, n2[3] = {uz2, u2.y, u2.x};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const F2 cu(a[i] + c[i], a[i] - c[i]);
        const float Be = mad(r.we, base, mul(r.ke, n2[i]));
        const F2 ns = mad(F2(-2.f), mad(p.Ke, mul(cu, cu), F2(Be)), se[i]), na = mad(-p.Ae, cu, de[i]);
        relax_pairs(ep[i], em[i], ns, na, p.force[i + 1], p);
        g[7 + 4 * i] = ep[i].x;
        g[9 + 4 * i] = ep[i].y;
        g[8 + 4 * i] = em[i].x;
        g[10 + 4 * i] = em[i].y;
    }
}

struct Lat19 {
    static constexpr int NQ = Q;
    using Consts = RelaxPacked;
    // 24 rows leave 80 registers a thread, 20 leave 96, which the wall logic needs
    template <bool WALLS> static constexpr int warps = WALLS ? 20 : 24;
    static __host__ __device__ constexpr int cx(int q) { return CX(q); }
    static __host__ __device__ constexpr int cy(int q) { return CY(q); }
    static __host__ __device__ constexpr int cz(int q) { return CZ(q); }
    // The walled kernel spills with the packed collision (channel 617 against 585 us).
    template <bool RHO0, bool WALLS, bool MRT>
    static __device__ __forceinline__ void collide(float g[Q], const RelaxPacked &p)
    {
        if constexpr (!WALLS && !MRT && !RHO0) collide_packed(g, p);
        else collide_any<float, RHO0, MRT, true>(g, p.r);
    }
};

// Shared-memory slots of a lattice: directions are grouped by c_z, each group
// a ring over planes.
template <typename L, bool WALLS>
struct PairRing {
    static __host__ __device__ constexpr int opp(int q) { return q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1); }
    static __host__ __device__ constexpr int count(int cz, int below)
    {
        int n = 0;
        for (int q = 0; q < below; ++q) n += L::cz(q) == cz;
        return n;
    }
    static constexpr int NP = count(1, L::NQ), N0 = count(0, L::NQ), NM = count(-1, L::NQ);
    static constexpr int RP = 4, R0 = 3, RM = WALLS ? 3 : 2;  // planes in each ring
    static constexpr int SLOTS = RP * NP + R0 * N0 + RM * NM;
    // slot of direction q when its group's ring stands at plane position 0
    static __host__ __device__ constexpr int first(int q)
    {
        return L::cz(q) > 0 ? count(1, q) : (L::cz(q) == 0 ? RP * NP + count(0, q) : RP * NP + R0 * N0 + count(-1, q));
    }
};

// Rows of a tile in step 1, one warp each.
template <typename L, bool WALLS> constexpr int pair_warps = L::template warps<WALLS>;

template <typename L, bool WALLS> constexpr int pair_smem()
{
    return PairRing<L, WALLS>::SLOTS * (pair_warps<L, WALLS> - 2) * PAIR_LANES * 4;
}

struct PairTiles {
    int tx, ty;  // columns a tile writes (at most PAIR_TX x rows - 2)
    int len;     // planes a block writes
};

template <typename L> struct PairPlanes {
    float *p[L::NQ];
};

template <typename L, bool RHO0, bool WALLS, bool MRT>
__global__ void __launch_bounds__(pair_warps<L, WALLS> *PAIR_LANES, 1)
    k_pair(PairPlanes<L> src, PairPlanes<L> dst, Geo g, typename L::Consts p, PairTiles t)
{
    using Ring = PairRing<L, WALLS>;
    constexpr int NQ = L::NQ;
    constexpr int W = pair_warps<L, WALLS>;
    constexpr int COLS = (W - 2) * PAIR_LANES;
    extern __shared__ float sh[];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int x0 = blockIdx.x * t.tx, y0 = blockIdx.y * t.ty, z0 = blockIdx.z * t.len;
    const int wx = min(t.tx, g.nx - x0), wy = min(t.ty, g.ny - y0), wz = min(t.len, g.nz - z0);
    const int xr = x0 - 1 + lane, yr = y0 - 1 + row;
    // step 1 covers the tile and its halo (beyond a wall there is no cell), step 2 the tile
    const bool in1 = lane <= wx + 1 && row <= wy + 1 && !(WALLS && g.wall_x && (xr < 0 || xr >= g.nx)) &&
                     !(WALLS && g.wall_y && (yr < 0 || yr >= g.ny));
    const bool in2 = lane >= 1 && lane <= wx && row >= 1 && row <= wy;
    // wrapped columns and rows around the cell, in bytes (any offset a thread forms is in range, see pair_runs)
    unsigned xs[3], ys[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        xs[i] = (unsigned)((xr - 1 + i + 2 * g.nx) % g.nx) * 4u;
        ys[i] = (unsigned)((yr - 1 + i + 2 * g.ny) % g.ny) * (unsigned)g.nx * 4u;
    }
    const bool bxm = WALLS && g.wall_x && xr == 0, bxp = WALLS && g.wall_x && xr == g.nx - 1;
    const bool bym = WALLS && g.wall_y && yr == 0, byp = WALLS && g.wall_y && yr == g.ny - 1;
    const bool edge_xy = __any_sync(0xffffffffu, bxm || bxp || bym || byp);
    const long long nxy = (long long)g.nx * g.ny * 4;
    // rows of shared memory are the tile's rows 1 ... W - 2
    float *const col = sh + (row - 1) * PAIR_LANES + lane;
    const bool up = row < W - 2, own = row >= 1 && row <= W - 2, down = row >= 2;  // rows row + 1, row, row - 1 exist

    auto plane_exists = [&](int s0) { return !(WALLS && g.wall_z && (s0 < 0 || s0 >= g.nz)); };
    auto at = [](const float *base, long long plane, unsigned off) {
        return *reinterpret_cast<const float *>(reinterpret_cast<const char *>(base) + plane + off);
    };
    float f[NQ];  // populations that stream into this thread's cell of the next plane
    auto load = [&](int s0) {  // s0 may lie one plane outside the lattice
        if (!in1 || !plane_exists(s0)) return;
        const int s = s0 < 0 ? s0 + g.nz : (s0 >= g.nz ? s0 - g.nz : s0);
        const long long zs[3] = {(s == 0 ? g.nz - 1 : s - 1) * nxy, s * nxy, (s == g.nz - 1 ? 0 : s + 1) * nxy};
        const bool bzm = WALLS && g.wall_z && s == 0, bzp = WALLS && g.wall_z && s == g.nz - 1;
        if (WALLS && (edge_xy || bzm || bzp)) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int cx = L::cx(q), cy = L::cy(q), cz = L::cz(q);
                const bool w = (cx > 0 && bxm) || (cx < 0 && bxp) || (cy > 0 && bym) || (cy < 0 && byp) ||
                               (cz > 0 && bzm) || (cz < 0 && bzp);
                f[q] = w ? at(src.p[Ring::opp(q)], zs[1], ys[1] + xs[1])
                         : at(src.p[q], zs[1 - cz], ys[1 - cy] + xs[1 - cx]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                f[q] = at(src.p[q], zs[1 - L::cz(q)], ys[1 - L::cy(q)] + xs[1 - L::cx(q)]);
        }
    };

    asm volatile("griddepcontrol.wait;" ::: "memory");  // launched early, see step_begin
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    load(z0 - 1);
    int kp = 0, k0 = 0, km = 0;  // ring positions of plane s
    for (int it = 0; it < wz + 2; ++it) {
        const int s = z0 - 1 + it;
        // ---- step 1 of plane s
        if (in1 && plane_exists(s)) {
            L::template collide<RHO0, WALLS, MRT>(f, p);
            const bool bzm = WALLS && g.wall_z && s == 0, bzp = WALLS && g.wall_z && s == g.nz - 1;
            if (WALLS && (edge_xy || bzm || bzp)) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int cx = L::cx(q), cy = L::cy(q), cz = L::cz(q), o = Ring::opp(q);
                    const bool w = (cx > 0 && bxp) || (cx < 0 && bxm) || (cy > 0 && byp) || (cy < 0 && bym) ||
                                   (cz > 0 && bzp) || (cz < 0 && bzm);
                    const int k = cz > 0 ? kp * Ring::NP : (cz == 0 ? k0 * Ring::N0 : km * Ring::NM);
                    // a value that crosses a wall arrives at the own cell in the opposite direction: it is
                    // stored where that direction is read for this cell (column x + c_x, plane s + c_z)
                    const int ko = cz > 0 ? (km == 2 ? 0 : km + 1) * Ring::NM
                                          : (cz == 0 ? k0 * Ring::N0 : ((kp + 3) & 3) * Ring::NP);
                    if (w ? in2 : (cy > 0 ? up : (cy == 0 ? own : down)))
                        col[w ? (ko + Ring::first(o)) * COLS + cx
                              : (k + Ring::first(q)) * COLS + cy * PAIR_LANES] = f[q];
                }
            } else {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int cy = L::cy(q), cz = L::cz(q);
                    const int k = cz > 0 ? kp * Ring::NP : (cz == 0 ? k0 * Ring::N0 : km * Ring::NM);
                    if (cy > 0 ? up : (cy == 0 ? own : down))
                        col[(k + Ring::first(q)) * COLS + cy * PAIR_LANES] = f[q];
                }
            }
        }
        if (it + 1 < wz + 2) load(s + 1);
        __syncthreads();
        // ---- step 2 of plane s - 1
        if (it >= 2 && in2) {
            const int jp = (kp + 2) & 3, j0 = k0 == 0 ? 2 : k0 - 1;  // planes s - 2 and s - 1
            float h[NQ];
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int cz = L::cz(q);
                const int k = cz > 0 ? jp * Ring::NP : (cz == 0 ? j0 * Ring::N0 : km * Ring::NM);
                h[q] = col[(k + Ring::first(q)) * COLS - L::cx(q)];
            }
            L::template collide<RHO0, WALLS, MRT>(h, p);
            const long long zd = (s - 1) * nxy;
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                *reinterpret_cast<float *>(reinterpret_cast<char *>(dst.p[q]) + zd + (ys[1] + xs[1])) = h[q];
        }
        kp = (kp + 1) & 3;
        k0 = k0 == 2 ? 0 : k0 + 1;
        km = km == Ring::RM - 1 ? 0 : km + 1;
    }
}

// Tiles for a lattice.  The blocks of one launch run in waves of PAIR_SMS, and
// each computes step 1 of two planes more than it writes; iterations: those of
// all waves one after the other, which the planes per block minimise.
static inline PairTiles pair_tiles(const Geo &g, int out_rows, dim3 &grid, long long &iterations)
{
    PairTiles t{};
    const int ntx = (g.nx + PAIR_TX - 1) / PAIR_TX, nty = (g.ny + out_rows - 1) / out_rows;
    t.tx = (g.nx + ntx - 1) / ntx;
    t.ty = (g.ny + nty - 1) / nty;
    const long long tiles = (long long)ntx * nty;
    iterations = -1;
    for (int c = 1; c <= g.nz; ++c) {
        const int len = (g.nz + c - 1) / c;
        const int nc = (g.nz + len - 1) / len;
        const long long k = (tiles * nc + PAIR_SMS - 1) / PAIR_SMS * (len + 2);
        if (iterations < 0 || k < iterations) {
            iterations = k;
            t.len = len;
            grid = dim3((unsigned)ntx, (unsigned)nty, (unsigned)nc);
        }
        if (len < 8) break;
    }
    return t;
}

// Whether two steps go through k_pair.  It addresses a plane by 32-bit byte offsets
// and forms wrapped coordinates as int, up to three edges long: a plane of 2^30 cells or
// more, an edge above 2^29, or more tile rows than a grid may have are stepped singly
// whatever is asked (`always`).  Otherwise where its iterations take less time than two
// one-step launches, which run at `glups` from DRAM.  An iteration takes `us`, with walls
// `us_walls` and the more the fewer waves overlap (D3Q19: 2.7 to 2.95 us, MRT 3.05 to
// 3.2; with walls 3.0 in one wave, 2.7 in four, 2.4 in eight; D3Q27 with walls 4.3, 3.7
// in three, 3.1 in nine; MRT with walls and rho0 = rho 3.7 in one wave.  With one figure for all, walled 1000x64x64 ran 98 us a step in
// pairs, 91 singly; D3Q27 116x160x279 208 and 171).  Not with walls on x, whose ends put
// half of the warps on the wall path (closed box 256x192x160: 172 against 210 us), nor
// for lattices whose grids stay in L2 (both below 200 MB; 96^3: 20 us a step against 22).
struct PairTimes {
    double us, us_walls, us_walls_per_wave, glups;
};
template <typename L>
static inline bool pair_runs(const Geo &g, bool always, const PairTimes &t)
{
    if ((long long)g.nx * g.ny >= 1LL << 30 || g.nx > 1 << 29 || g.ny > 1 << 29) return false;
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
    dim3 grid;
    long long iterations;
    pair_tiles(g, (walls ? pair_warps<L, true> : pair_warps<L, false>) - 2, grid, iterations);
    if (grid.y > 65535) return false;
    const long long waves = ((long long)grid.x * grid.y * grid.z + PAIR_SMS - 1) / PAIR_SMS;
    const double us = walls ? t.us_walls + t.us_walls_per_wave / waves : t.us;
    return always ||
           (!g.wall_x && g.ncell * 8 * L::NQ >= 200000000 && iterations * us < 2.0 * (double)g.ncell / (t.glups * 1e3));
}

template <typename L, bool RHO0, bool WALLS, bool MRT>
static cudaError_t launch_pair_k(const PairPlanes<L> &S, const PairPlanes<L> &D, const Geo &g,
                                 const typename L::Consts &p, cudaStream_t stream)
{
    constexpr int smem = pair_smem<L, WALLS>();
    static_assert(smem <= 227 * 1024, "tile does not fit shared memory");
    auto k = k_pair<L, RHO0, WALLS, MRT>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    dim3 grid;
    long long iterations;
    const PairTiles t = pair_tiles(g, pair_warps<L, WALLS> - 2, grid, iterations);
    launch_step_kernel(k, true, grid, pair_warps<L, WALLS> * PAIR_LANES, stream, smem, S, D, g, p, t);
    return cudaGetLastError();
}

template <typename L>
static PairPlanes<L> pair_planes(const void *base, long long ncell)
{
    PairPlanes<L> r;
    for (int q = 0; q < L::NQ; ++q) r.p[q] = (float *)const_cast<void *>(base) + (long long)q * ncell;
    return r;
}

}  // namespace lbm
