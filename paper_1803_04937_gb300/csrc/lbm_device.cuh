// Device-side building blocks of the D3Q19 library: the lattice, storage
// conversions, lattice geometry (periodic wrap and half-way bounce-back), the
// gather / scatter patterns of the A/B and AA propagation schemes, and the
// collision of Eq. 15 (SRT) or its TRT split, written in shifted variables
// g_q = f_q - w_q.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "lbm_launch.h"

namespace lbm {

constexpr int Q = 19;

// D3Q19 velocity set of Sec. 2.3 in this library's order: q = 0 rest, then
// nine pairs (q, q+1) with c_{q+1} = -c_q: three faces, six edges.
__host__ __device__ constexpr int CX(int q)
{
    constexpr int t[Q] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[q];
}
__host__ __device__ constexpr int CY(int q)
{
    constexpr int t[Q] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[q];
}
__host__ __device__ constexpr int CZ(int q)
{
    constexpr int t[Q] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[q];
}
__host__ __device__ constexpr int OPP(int q) { return q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1); }
__host__ __device__ constexpr int NORM2(int q) { return CX(q) * CX(q) + CY(q) * CY(q) + CZ(q) * CZ(q); }
// weights 1/3, 1/18, 1/36 (Sec. 2.3)
template <typename R>
__host__ __device__ constexpr R WQ(int q)
{
    return NORM2(q) == 0 ? R(1) / R(3) : (NORM2(q) == 1 ? R(1) / R(18) : R(1) / R(36));
}

// ---------------------------------------------------------------- storage

template <typename T> struct Storage;
template <> struct Storage<double> {
    using R = double;
    static __device__ __forceinline__ R load(const double *p) { return *p; }
    static __device__ __forceinline__ void store(double *p, R v) { *p = v; }
};
template <> struct Storage<float> {
    using R = float;
    static __device__ __forceinline__ R load(const float *p) { return *p; }
    static __device__ __forceinline__ void store(float *p, R v) { *p = v; }
};
template <> struct Storage<__half> {
    using R = float;
    static __device__ __forceinline__ R load(const __half *p) { return __half2float(*p); }
    static __device__ __forceinline__ void store(__half *p, R v) { *p = __float2half_rn(v); }
};
template <> struct Storage<__nv_bfloat16> {
    using R = float;
    static __device__ __forceinline__ R load(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, R v) { *p = __float2bfloat16_rn(v); }
};

// ---------------------------------------------------------------- geometry


struct Geo {
    int nx, ny, nz;
    int wall_x, wall_y, wall_z;  // 1: half-way bounce-back walls at both ends
    long long ncell;             // plane stride of the SoA grid, nx * ny * nz
};

// Quotient and remainder by a divisor fixed per launch: for 0 <= n < 2^31,
// n / d = (n * ceil(2^(31 + l) / d)) >> (31 + l) with 2^l >= d (the factor's
// error, below d, is multiplied by n < 2^31 and stays below 2^(31 + l)).
struct Divider {
    unsigned d, mul;
    int shift;

    Divider() = default;
    explicit Divider(int divisor) : d((unsigned)divisor)
    {
        int l = 0;
        while ((1LL << l) < divisor) ++l;
        shift = 31 + l;
        mul = (unsigned)(((1ULL << shift) + d - 1) / d);
    }
    __device__ __forceinline__ int div(int n, int &rem) const
    {
        const int quo = (int)(((unsigned long long)(unsigned)n * mul) >> shift);
        rem = n - quo * (int)d;
        return quo;
    }
};

// A box of lattice rows, y in [y0, y0 + rows), z from z0 on, walked as one
// sequence of work items (cells, or groups of neighbouring cells) in memory
// order, so that a block holds as many items as it has threads whatever the
// length of a row: with one block row per lattice row, a lattice four cells
// long kept 4 of 32 lanes busy (4x96x96 FP64: 93 us a step), one of 40 quads 40
// of 64 (160^3 FP16: 64 us).  The two divisions cost a few of about 500
// instructions.
struct Box {
    unsigned count;  // items
    int y0, z0;
    Divider per_row, rows;  // items in a row, rows in a plane of the box
    int y_walled = 0;       // wall rows only: rows of the faces normal to y, which come first
    Divider planes{1};      // ... and planes of a y face
    int y_last = 0, z_last = 0;
    int nz = 0;             // planes of the box
    bool waits = true;      // step_begin waits for the launch before (false: it had ended before this one began)

    Box() = default;
    Box(int items_per_row, int y0_, int y1, int z0_, int planes_)
        : count((unsigned)((long long)items_per_row * (y1 - y0_) * planes_)), y0(y0_), z0(z0_),
          per_row(items_per_row), rows(y1 - y0_), nz(planes_)
    {
    }
    // item i: its place in the row, y and z
    __device__ __forceinline__ void at(unsigned i, int &item, int &y, int &z) const
    {
        int yr;
        z = z0 + rows.div(per_row.div((int)i, item), yr);
        y = y0 + yr;
    }

    // the same from a thread's place in a grid of blocks that are rectangles of
    // rows; false for a thread outside the box
    __device__ __forceinline__ bool at_block(int &item, int &y, int &z) const
    {
        item = blockIdx.x * blockDim.x + threadIdx.x;
        const unsigned yr = blockIdx.y * blockDim.y + threadIdx.y;
        y = y0 + (int)yr;
        z = z0 + (int)blockIdx.z;
        return item < (int)per_row.d && yr < rows.d;
    }
    // Threads along x of such blocks, 128, 64 or 32 of `threads`, with the fewest
    // idle lanes at the end of a row, the larger on ties; 0: take the items as one
    // sequence, because more than 1/8 of the lanes would be idle or the grid would
    // have too many rows; or because four cells an item past the row's end would pass
    // 2^31 - 1.
    int block_x(int threads) const
    {
        const int n = (int)per_row.d;
        if (n > (1 << 29) - 128) return 0;
        int bx = 0, idle = 0;
        for (int c = 128; c >= 32; c /= 2) {
            const int w = (n + c - 1) / c * c - n;
            if (c <= threads && (!bx || w < idle)) {
                bx = c;
                idle = w;
            }
        }
        const long long by = threads / bx;
        return 8LL * idle > n || (rows.d + by - 1) / by > 65535 ? 0 : bx;
    }

    // The rows at walls normal to y or z: rows y = 0 and ny - 1 over all z, then
    // planes z = 0 and nz - 1 over the other y.
    static Box wall_rows(int items_per_row, const Geo &g)
    {
        const int ylo = g.wall_y ? 1 : 0, yhi = g.wall_y ? g.ny - 1 : g.ny;
        Box b;
        b.y0 = ylo;
        b.z0 = 0;
        b.per_row = Divider(items_per_row);
        b.rows = Divider(yhi > ylo ? yhi - ylo : 1);
        b.planes = Divider(g.nz);
        b.y_last = g.ny - 1;
        b.z_last = g.nz - 1;
        b.y_walled = g.wall_y ? (g.ny > 1 ? 2 : 1) * g.nz : 0;
        const long long z_walled = g.wall_z && yhi > ylo ? (long long)(g.nz > 1 ? 2 : 1) * (yhi - ylo) : 0;
        b.count = (unsigned)(items_per_row * (b.y_walled + z_walled));
        return b;
    }
    __device__ __forceinline__ void at_wall(unsigned i, int &item, int &y, int &z) const
    {
        const int row = per_row.div((int)i, item);
        if (row < y_walled) {
            y = planes.div(row, z) ? y_last : 0;
        } else {
            int yr;
            z = rows.div(row - y_walled, yr) ? z_last : 0;
            y = y0 + yr;
        }
    }
};

// The rows of a lattice with walls in one launch: the first blocks take the rows at
// walls normal to y or z (which cost more and so start first), the others the rows
// between them, as one sequence of items or (bx_log2 >= 0) in blocks that are rectangles of
// rows.  Every row is in exactly one block's part, and which part a block has is
// uniform in it.
struct WalledBox {
    Box walls, inner;
    unsigned wall_blocks;
    int bx_log2;                  // -1: inner is one sequence
    Divider blocks_x, blocks_y;   // rectangles along x and y

    // rectangles: where the shape of the inner rows fills them (Box::block_x)
    WalledBox(int items_per_row, int items_per_wall_row, const Geo &g, int threads, bool rectangles)
        : walls(Box::wall_rows(items_per_wall_row, g))
    {
        const int ylo = g.wall_y ? 1 : 0, yhi = g.wall_y ? g.ny - 1 : g.ny;
        const int zlo = g.wall_z ? 1 : 0, zhi = g.wall_z ? g.nz - 1 : g.nz;
        const bool some = yhi > ylo && zhi > zlo;
        inner = some ? Box(items_per_row, ylo, yhi, zlo, zhi - zlo) : Box(items_per_row, 0, 1, 0, 0);
        wall_blocks = (walls.count + threads - 1) / threads;
        const int bx = rectangles && some ? inner.block_x(threads) : 0;
        bx_log2 = bx == 0 ? -1 : (bx == 128 ? 7 : (bx == 64 ? 6 : 5));
        blocks_x = Divider(bx ? (int)((inner.per_row.d + bx - 1) / bx) : 1);
        blocks_y = Divider(bx ? (int)((inner.rows.d + threads / bx - 1) / (threads / bx)) : 1);
    }
    unsigned blocks(int threads) const
    {
        return wall_blocks + (bx_log2 < 0 ? (inner.count + threads - 1) / threads : blocks_x.d * blocks_y.d * (unsigned)inner.nz);
    }
    __device__ __forceinline__ bool at_walls() const { return blockIdx.x < wall_blocks; }
    // this thread's item in the sequence of its block's part
    __device__ __forceinline__ unsigned wall_item() const { return blockIdx.x * blockDim.x + threadIdx.x; }
    __device__ __forceinline__ unsigned inner_item() const { return (blockIdx.x - wall_blocks) * blockDim.x + threadIdx.x; }
    // ... and its item, y and z in a rectangle; y may lie past the box, item past the row
    __device__ __forceinline__ void inner_rectangle(int &item, int &y, int &z) const
    {
        int ix, iy;
        z = inner.z0 + blocks_y.div(blocks_x.div((int)(blockIdx.x - wall_blocks), ix), iy);
        item = (ix << bx_log2) + (int)(threadIdx.x & ((1u << bx_log2) - 1));
        y = inner.y0 + iy * (int)(blockDim.x >> bx_log2) + (int)(threadIdx.x >> bx_log2);
    }
};

// Launches of consecutive steps overlap their start with the end of the one
// before (programmatic dependent launch): a step's blocks may be scheduled once
// all blocks of the launch before have passed step_begin, that is once it needs
// no more slots, and wait there for its completion, which also makes visible what
// it wrote.  Every launch that may start early waits for itself: another launch's
// wait orders its blocks, but publishes no memory to them.
__device__ __forceinline__ void step_begin(const Box &box)
{
    if (box.waits) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void step_begin(const WalledBox &box) { step_begin(box.inner); }

// One lattice cell with its wrapped neighbour coordinates and the wall flags
// of its six faces (true when the neighbour across that face is beyond a wall).
struct Cell {
    int x, y, z;
    int xm, xp, ym, yp, zm, zp;
    bool bxm, bxp, bym, byp, bzm, bzp;
    int nx, nxy;

    __device__ __forceinline__ Cell(int x_, int y_, int z_, const Geo &g) : x(x_), y(y_), z(z_)
    {
        xm = x == 0 ? g.nx - 1 : x - 1;
        xp = x == g.nx - 1 ? 0 : x + 1;
        ym = y == 0 ? g.ny - 1 : y - 1;
        yp = y == g.ny - 1 ? 0 : y + 1;
        zm = z == 0 ? g.nz - 1 : z - 1;
        zp = z == g.nz - 1 ? 0 : z + 1;
        bxm = g.wall_x && x == 0;
        bxp = g.wall_x && x == g.nx - 1;
        bym = g.wall_y && y == 0;
        byp = g.wall_y && y == g.ny - 1;
        bzm = g.wall_z && z == 0;
        bzp = g.wall_z && z == g.nz - 1;
        nx = g.nx;
        nxy = g.nx * g.ny;
    }
    __device__ __forceinline__ int self() const { return (z * nxy) + y * nx + x; }

    // Cell x + s*c_q (s = +1: push target, s = -1: pull source).  Sets
    // `wall` when the link crosses a bounce-back wall.
    template <int S>
    __device__ __forceinline__ int along(int q, bool &wall) const
    {
        const int cx = S * CX(q), cy = S * CY(q), cz = S * CZ(q);
        int xs = cx == 0 ? x : (cx > 0 ? xp : xm);
        int ys = cy == 0 ? y : (cy > 0 ? yp : ym);
        int zs = cz == 0 ? z : (cz > 0 ? zp : zm);
        bool w = false;
        if (cx > 0) w |= bxp;
        if (cx < 0) w |= bxm;
        if (cy > 0) w |= byp;
        if (cy < 0) w |= bym;
        if (cz > 0) w |= bzp;
        if (cz < 0) w |= bzm;
        wall = w;
        return zs * nxy + ys * nx + xs;
    }
};

// State layouts.  The canonical state is f_q(x, t) after streaming, before
// collision.  How it sits in memory:
//   AB      : grid[q][x - c_q] (the previous step's post-collision value that
//             streams into x); through a wall, grid[qbar][x].
//   AA_EVEN : grid[q][x] (after an even number of AA steps).
//   AA_ODD  : grid[qbar][x - c_q]; through a wall grid[q][x] (after an odd
//             number of AA steps).
enum Layout { AB = 0, AA_EVEN = 1, AA_ODD = 2 };

// Where post-collision values of a step go:
//   AB_NEXT : grid[q][x]                 (pull scheme, next step gathers them)
//   AA_EVEN : grid[qbar][x]
//   AA_ODD  : grid[q][x + c_q]; through a wall grid[qbar][x]
// and, to write a canonical state f_q(x) into a grid so that the AB gather
// returns it: AB_CANON : grid[q][x - c_q]; through a wall grid[qbar][x].
enum Dest { D_AB_NEXT = 0, D_AA_EVEN = 1, D_AA_ODD = 2, D_AB_CANON = 3 };

template <int D, typename T, typename R>
__device__ __forceinline__ void scatter(T *grid, const Cell &c, long long ncell, const R g[Q])
{
    const int self = c.self();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long off;
        if (D == D_AB_NEXT) {
            off = (long long)q * ncell + self;
        } else if (D == D_AA_EVEN) {
            off = (long long)OPP(q) * ncell + self;
        } else if (D == D_AA_ODD) {
            bool wall;
            int dst = c.template along<1>(q, wall);
            off = wall ? (long long)OPP(q) * ncell + self : (long long)q * ncell + dst;
        } else {
            bool wall;
            int dst = c.template along<-1>(q, wall);
            off = wall ? (long long)OPP(q) * ncell + self : (long long)q * ncell + dst;
        }
        Storage<T>::store(grid + off, g[q]);
    }
}

// ---------------------------------------------------------------- reductions

// Sum over the block (blockDim.x a multiple of 32, at most 1024 threads);
// the result is valid in thread 0.  Fixed order: deterministic.
__device__ __forceinline__ double block_sum(double v, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    v = 0.0;
    if (warp == 0) {
        const int nw = blockDim.x >> 5;
        v = lane < nw ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;
}

// ---------------------------------------------------------------- physics

// Per-launch collision constants (prepared on the host).
template <typename R>
struct Coll {
    R omega_p;        // 1 / tau
    R omega_m;        // 1 / tau-  (= omega_p for SRT)
    R kappa;          // 0: D3Q19-S (Eq. 14), 1: D3Q19-I (Eq. 22)
    R half_a[3];      // a / 2, the velocity shift of Eq. 17
    R force[9];       // (1 - omega_m / 2) F_q for the first member q = 2k+1 of pair k
    int rho0_is_rho;  // 0: rho0 = 1, 1: rho0 = rho
};

// Macroscopic quantities of the shifted populations: drho = rho - 1,
// u from rho0 u = j + a/2 (Eq. 16, Eq. 17), and rho0.
template <typename R>
static inline Coll<R> to_coll(const CollBoth &c)
{
    Coll<R> p;
    p.omega_p = R(c.omega_p);
    p.omega_m = R(c.omega_m);
    p.kappa = R(c.kappa);
    for (int i = 0; i < 3; ++i) p.half_a[i] = R(c.half_a[i]);
    for (int k = 0; k < 9; ++k) p.force[k] = R(c.force[k]);
    p.rho0_is_rho = c.rho0_is_rho;
    return p;
}

template <typename R>
__device__ __forceinline__ void macro(const R g[Q], const Coll<R> &p, R &drho, R &rho0, R u[3])
{
    R s = g[0];
    R jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        s += g[q];
        if (CX(q) > 0) jx += g[q];
        if (CX(q) < 0) jx -= g[q];
        if (CY(q) > 0) jy += g[q];
        if (CY(q) < 0) jy -= g[q];
        if (CZ(q) > 0) jz += g[q];
        if (CZ(q) < 0) jz -= g[q];
    }
    drho = s;
    rho0 = p.rho0_is_rho ? R(1) + s : R(1);
    R inv = p.rho0_is_rho ? R(1) / rho0 : R(1);
    u[0] = (jx + p.half_a[0]) * inv;
    u[1] = (jy + p.half_a[1]) * inv;
    u[2] = (jz + p.half_a[2]) * inv;
}

// Equilibrium of pair k (q = 2k+1 and its opposite) in shifted form:
//   geq_q = sym + asym,  geq_qbar = sym - asym,
// with the standard part w (drho + rho0 (9/2 (c.u)^2 - 3/2 u^2)), asym =
// 3 w rho0 c.u, plus kappa * rho0 * Delta_q where D3Q19-I = D3Q19-S + Delta:
//   face along axis a:   Delta = -(u^2 - u_a^2) / 12
//   edge in plane (a,b): Delta = u_c^2 / 24   (c the third axis)
// (the difference of Eq. 22 and Eq. 14 written per velocity group; both
// equilibria run the same instructions and differ only in kappa).
template <typename R, int q>
__device__ __forceinline__ void pair_equilibrium(const R u[3], R uu, R drho, R rho0, R kappa, R &sym, R &asym)
{
    constexpr int cx = CX(q), cy = CY(q), cz = CZ(q);
    const R w = WQ<R>(q);
    R cu = R(cx) * u[0] + R(cy) * u[1] + R(cz) * u[2];
    R delta;
    if (NORM2(q) == 1) {
        R ua = cx != 0 ? u[0] : (cy != 0 ? u[1] : u[2]);
        delta = (ua * ua - uu) * (R(1) / R(12));
    } else {
        R uc = cx == 0 ? u[0] : (cy == 0 ? u[1] : u[2]);
        delta = uc * uc * (R(1) / R(24));
    }
    sym = w * (drho + rho0 * (R(4.5) * cu * cu - R(1.5) * uu)) + kappa * rho0 * delta;
    asym = w * rho0 * R(3) * cu;
}

template <typename R>
__device__ __forceinline__ R rest_equilibrium(R uu, R drho, R rho0, R kappa)
{
    return WQ<R>(0) * (drho - rho0 * R(1.5) * uu) + kappa * rho0 * uu * (R(1) / R(6));
}

// ---------------------------------------------------------------- lean collision (step kernels)

// Products and fused multiply-adds of the collision, written out (plain
// products are never left to be contracted), so that every kernel rounds a
// cell's update alike.
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mad(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return fma(a, b, c); }

template <typename R> __device__ __forceinline__ R third() { return R(1.0f / 3.0f); }
template <> __device__ __forceinline__ double third<double>() { return 1.0 / 3.0; }

// Per-launch constants of the collision, folded so that a cell update needs
// few instructions.  With P = rho0 (1, or rho when rho0 = rho) and base =
// drho - 3/2 P u^2, the symmetric (even) equilibrium part of a pair is
//   faces along a:     wf base - kf u^2 + Kf u_a^2
//   edges normal to c: we base + ke u_c^2 + Ke (c.u)^2
//   rest:              w0 base + k0 u^2
// (kappa = 0: D3Q19-S; kappa = 1 adds the D3Q19-I corrections Delta), and the
// antisymmetric part is A/2 (c.u) with A = 6 w P.  The factors that carry P
// are stored for P = 1 and scaled per cell when rho0 = rho.
template <typename R>
struct Relax {
    R hp, hm, wp;    // omega+ / 2, omega- / 2, omega+
    R w0, wf, we;    // 1/3, 1/18, 1/36
    R k0, kf, ke;    // kappa / 6, kappa / 12, kappa / 24
    R Kf, Ke;        // 9/2 wf + kappa / 12, 9/2 we
    R Af, Ae;        // 6 wf, 6 we  (twice the antisymmetric coefficient)
    R half_a[3];     // a / 2
    R force[9];      // (1 - omega- / 2) F_q, q = 2k+1
    R hb, h4;        // MRT: (omega+ - omega_bulk) / 2, (omega+ - omega_4) / 2
};

template <typename R>
static inline Relax<R> to_relax(const CollBoth &c)
{
    const double wp = c.omega_p, wm = c.omega_m, k = c.kappa;
    const double w0 = 1.0 / 3.0, wf = 1.0 / 18.0, we = 1.0 / 36.0;
    Relax<R> r;
    r.hp = R(0.5 * wp);
    r.hm = R(0.5 * wm);
    r.wp = R(wp);
    r.w0 = R(w0);
    r.wf = R(wf);
    r.we = R(we);
    r.k0 = R(k / 6.0);
    r.kf = R(k / 12.0);
    r.ke = R(k / 24.0);
    r.Kf = R(4.5 * wf + k / 12.0);
    r.Ke = R(4.5 * we);
    // The equilibrium's first moment is (Af + 4 Ae) u per axis; with the
    // weights rounded to R it would be u (1 + eps), and the antisymmetric
    // relaxation would then grow the momentum by omega- eps every step (2000
    // FP32 steps: ~1e-4).  Af is chosen so that Af + 4 Ae = 1 exactly in R
    // (1 - 4 Ae is exact by Sterbenz's lemma).
    r.Ae = R(1.0 / 6.0);
    r.Af = R(1) - R(4) * r.Ae;
    for (int i = 0; i < 3; ++i) r.half_a[i] = R(c.half_a[i]);
    for (int i = 0; i < 9; ++i) r.force[i] = R(c.force[i]);
    r.hb = R(0.5 * (wp - c.omega_bulk));
    r.h4 = R(0.5 * (wp - c.omega_4));
    return r;
}

// Error-free sum (Knuth's TwoSum): hi + lo tracks hi + v exactly, hi holding
// the rounded sum and lo the accumulated rounding errors.
template <typename R>
__device__ __forceinline__ void two_sum_acc(R &hi, R &lo, R v)
{
    const R s = hi + v;
    const R bv = s - hi;
    lo += (hi - (s - bv)) + (v - bv);
    hi = s;
}

// Double-float numbers: an unevaluated sum hi + lo of two floats.  Sums of
// FP32 terms built with error-free transformations (TwoSum) keep about 48
// bits, as many as FP64 sums of the same FP32 terms would, and run on the FP32
// pipe.
struct DF {
    float hi, lo;
};

__device__ __forceinline__ DF df_add(DF a, DF b)
{
    const float s = a.hi + b.hi;
    const float bv = s - a.hi;
    float e = (a.hi - (s - bv)) + (b.hi - bv);
    e += a.lo + b.lo;
    const float hi = s + e;
    return DF{hi, e - (hi - s)};
}

__device__ __forceinline__ DF df_warp_sum(DF a)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const DF b{__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o)};
        a = df_add(a, b);
    }
    return a;
}

// c_q . u of a lattice direction (c: its components, -1, 0 or 1) without the
// products by 0 and +-1, which the compiler may not drop by itself.
template <typename R>
__device__ __forceinline__ R along(int cx, int cy, int cz, const R u[3])
{
    R r = cx ? (cx > 0 ? u[0] : -u[0]) : (cy ? (cy > 0 ? u[1] : -u[1]) : (cz > 0 ? u[2] : -u[2]));
    if (cx && cy) r = cy > 0 ? r + u[1] : r - u[1];
    if ((cx || cy) && cz) r = cz > 0 ? r + u[2] : r - u[2];
    return r;
}

// Moments and symmetric-equilibrium bases of one cell, shared by the step and
// the adjoint.  s[k], d[k]: sum and difference of pair
// k (q = 2k+1, q + 1).
//
// COMP (rho0 = 1 only): the momentum is summed with TwoSum, and du = (j +
// a/2) - u, the part of the exact velocity that rounding u drops, is kept.
// The antisymmetric relaxation moves the momentum by -omega- (j + a/2 - u)
// per step (zero in exact arithmetic); with a rounded u, that is -omega- du
// every step, and in a flow that changes slowly (a channel accelerated from
// rest by a body force) these errors add up coherently: FP32 storage, 5000
// steps, 1x256x1 channel column in emulation: 1.9e-5 of max|u| against the
// FP64 oracle.  neq() subtracts du from the face pair of each axis, which
// makes the momentum balance exact again; what remains is the storage
// rounding (same emulation: 9e-7).
template <typename R, bool RHO0_IS_RHO, bool COMP = false>
struct CellEq {
    R s[9], d[9];
    R u[3], u2[3], uu, P;
    R du[3];
    R Bf, Be[3], eq0;
    R Kf, Ke, Af, Ae;

    __device__ __forceinline__ CellEq(const R g[Q], const Relax<R> &p)
    {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            s[k] = g[2 * k + 1] + g[2 * k + 2];
            d[k] = g[2 * k + 1] - g[2 * k + 2];
        }
        const R drho = g[0] + (((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7])) + s[8]);
        // momentum: pair k < 3 is the face pair of axis k (c = +e_k) and starts the sum
        R j[3] = {d[0], d[1], d[2]};
        if (RHO0_IS_RHO || !COMP) {
#pragma unroll
            for (int k = 3; k < 9; ++k) {
                const int q = 2 * k + 1;
                if (CX(q) != 0) j[0] = CX(q) > 0 ? j[0] + d[k] : j[0] - d[k];
                if (CY(q) != 0) j[1] = CY(q) > 0 ? j[1] + d[k] : j[1] - d[k];
                if (CZ(q) != 0) j[2] = CZ(q) > 0 ? j[2] + d[k] : j[2] - d[k];
            }
        }
        if (RHO0_IS_RHO) {
            P = R(1) + drho;
            const R inv = R(1) / P;
#pragma unroll
            for (int i = 0; i < 3; ++i) u[i] = mul(j[i] + p.half_a[i], inv);
        } else if (COMP) {
            R lo[3] = {R(0), R(0), R(0)};
#pragma unroll
            for (int k = 3; k < 9; ++k) {
                const int q = 2 * k + 1;
                if (CX(q) != 0) two_sum_acc(j[0], lo[0], CX(q) > 0 ? d[k] : -d[k]);
                if (CY(q) != 0) two_sum_acc(j[1], lo[1], CY(q) > 0 ? d[k] : -d[k]);
                if (CZ(q) != 0) two_sum_acc(j[2], lo[2], CZ(q) > 0 ? d[k] : -d[k]);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                u[i] = j[i];
                two_sum_acc(u[i], lo[i], p.half_a[i]);
                du[i] = lo[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) u[i] = j[i] + p.half_a[i];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) u2[i] = mul(u[i], u[i]);
        uu = (u2[0] + u2[1]) + u2[2];
        R k0 = p.k0, kf = p.kf, ke = p.ke;
        Kf = p.Kf;
        Ke = p.Ke;
        Af = p.Af;
        Ae = p.Ae;
        R h = R(-1.5);  // -3/2 P
        if (RHO0_IS_RHO) {
            k0 = mul(k0, P); kf = mul(kf, P); ke = mul(ke, P);
            Kf = mul(Kf, P); Ke = mul(Ke, P); Af = mul(Af, P); Ae = mul(Ae, P);
            h = mul(h, P);
        }
        const R base = mad(h, uu, drho);
        Bf = mad(p.wf, base, -mul(kf, uu));
#pragma unroll
        for (int i = 0; i < 3; ++i) Be[i] = mad(p.we, base, mul(ke, u2[i]));
        eq0 = mad(p.w0, base, mul(k0, uu));
    }

    // Non-equilibrium parts of pair k: s - 2 sym and d - 2 asym, each formed
    // by one fused multiply-add so that only the small result is rounded.
    template <int k>
    __device__ __forceinline__ void neq(R &nsym, R &nasym) const
    {
        constexpr int q = 2 * k + 1;
        const R cu = along(CX(q), CY(q), CZ(q), u);
        R sym, A;
        if (NORM2(q) == 1) {
            const int a = CX(q) ? 0 : (CY(q) ? 1 : 2);
            sym = mad(Kf, u2[a], Bf);
            A = Af;
        } else {
            const int c = CX(q) == 0 ? 0 : (CY(q) == 0 ? 1 : 2);
            sym = mad(Ke, mul(cu, cu), Be[c]);
            A = Ae;
        }
        nsym = mad(R(-2), sym, s[k]);
        nasym = mad(-A, cu, d[k]);
        if constexpr (COMP && !RHO0_IS_RHO && k < 3) nasym -= du[k];
    }
};

// One collision (Eq. 15, or its TRT split) of the shifted populations g in
// place: g -/+ (omega+/2)(s - 2 sym) -/+ (omega-/2)(d - 2 asym) +/- (1 -
// omega-/2) F for the two members of each pair; the same result as the
// textbook form g - omega+ (g+ - geq+) - omega- (g- - geq-) + (1 - omega-/2) F
// up to rounding order.  With ONE_ROUNDING the change of each population is
// formed first by one fma (small numbers, small rounding) and added to g in one
// operation: one rounding at the scale of g instead of two (measured on the
// 256^3 FP32 shear wave after 2000 steps: worst error against the FP64 oracle
// 1.1e-5 -> 3.7e-6).  The step kernels take it for FP32 and FP64 storage
// (one_rounding_v); with 16-bit storage the rounding at the store is 2^13 times
// coarser than FP32's, so the two-rounding form loses nothing there, and some
// 16-bit kernels run it faster (walled channel 512x256x256, BF16: 77.8 -> 79.8
// GLUPS; D3Q27 four cells, FP16: 59.6 -> 62.9).
template <typename T>
constexpr bool one_rounding_v = sizeof(T) >= 4;

// FP32 storage (FP32 arithmetic with the one-rounding update) also sums the
// momentum with compensation (CellEq, COMP): 16-bit storage rounds far more
// coarsely at the store, and FP64 arithmetic does not need it.
template <typename R, bool ONE_ROUNDING>
constexpr bool compensated_v = ONE_ROUNDING && std::is_same<R, float>::value;

template <typename R, bool RHO0_IS_RHO, bool ONE_ROUNDING, int k>
__device__ __forceinline__ void relax_pair(R g[Q], const CellEq<R, RHO0_IS_RHO, compensated_v<R, ONE_ROUNDING>> &e,
                                           const Relax<R> &p)
{
    constexpr int q = 2 * k + 1;
    R nsym, nasym;
    e.template neq<k>(nsym, nasym);
    const R b = mad(p.hm, nasym, -p.force[k]);
    if (ONE_ROUNDING) {
        g[q] = g[q] - mad(p.hp, nsym, b);
        g[q + 1] = g[q + 1] - mad(p.hp, nsym, -b);
    } else {
        g[q] = mad(-p.hp, nsym, g[q]) - b;
        g[q + 1] = mad(-p.hp, nsym, g[q + 1]) + b;
    }
}

template <typename R, bool RHO0_IS_RHO, bool ONE_ROUNDING>
__device__ __forceinline__ void collide_lean(R g[Q], const Relax<R> &p)
{
    const CellEq<R, RHO0_IS_RHO, compensated_v<R, ONE_ROUNDING>> e(g, p);
    g[0] = mad(-p.wp, g[0] - e.eq0, g[0]);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 0>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 1>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 2>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 3>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 4>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 5>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 6>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 7>(g, e, p);
    relax_pair<R, RHO0_IS_RHO, ONE_ROUNDING, 8>(g, e, p);
}

// MRT collision (Sec. 3.2-3.3) in population space.  The even part of the
// non-equilibrium (rest n0 and pair sums ns) has, in the monomial moment basis,
// the second-order moments P and the fourth-order moments Q_c = sum over the
// two edge pairs normal to axis c (xi_a^2 xi_b^2, {a,b,c} = {x,y,z}); its
// zeroth moment is zero.  Relaxing the deviator of P at omega+, the trace
// T = tr P at omega_bulk and Q at omega_4 equals relaxing everything at
// omega+ and adding back (omega+ - omega_bulk) times the population vector
// whose only non-zero moment is that trace (rest -T, faces T/3, edges 0),
// plus (omega+ - omega_4) times the vector whose only non-zero moments are
// the Q (rest sum Q, face a Q_a - sum Q, edges normal to c Q_c/2); these are
// the columns of the inverse moment matrix for those moments.  The odd part
// relaxes at omega- with the force, exactly as in collide_lean.
template <typename R, bool RHO0_IS_RHO, bool ONE_ROUNDING>
__device__ __forceinline__ void collide_mrt(R g[Q], const Relax<R> &p)
{
    const CellEq<R, RHO0_IS_RHO, compensated_v<R, ONE_ROUNDING>> e(g, p);
    R ns[9], na[9];
    e.template neq<0>(ns[0], na[0]);
    e.template neq<1>(ns[1], na[1]);
    e.template neq<2>(ns[2], na[2]);
    e.template neq<3>(ns[3], na[3]);
    e.template neq<4>(ns[4], na[4]);
    e.template neq<5>(ns[5], na[5]);
    e.template neq<6>(ns[6], na[6]);
    e.template neq<7>(ns[7], na[7]);
    e.template neq<8>(ns[8], na[8]);
    // pairs 3, 4 are the edges normal to z, 5, 6 to y, 7, 8 to x
    const R faces = (ns[0] + ns[1]) + ns[2];
    const R Qn[3] = {ns[7] + ns[8], ns[5] + ns[6], ns[3] + ns[4]};
    const R Qsum = (Qn[0] + Qn[1]) + Qn[2];
    const R T = mad(R(2), Qsum, faces);
    const R bT = mul(p.hb, T);       // (omega+ - omega_bulk) T / 2
    const R bQ = mul(p.h4, Qsum);    // (omega+ - omega_4) sum Q / 2
    const R face0 = mad(bT, third<R>(), -bQ);
    g[0] = mad(R(-2), bT - bQ, mad(-p.wp, g[0] - e.eq0, g[0]));
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int q = 2 * k + 1;
        R corr;  // (omega+ - omega_bulk) B / 2 + (omega+ - omega_4) G / 2 for this pair
        if (NORM2(q) == 1) {
            const int a = CX(q) ? 0 : (CY(q) ? 1 : 2);
            corr = mad(p.h4, Qn[a], face0);
        } else {
            const int c = CX(q) == 0 ? 0 : (CY(q) == 0 ? 1 : 2);
            corr = mul(mul(R(0.5f), p.h4), Qn[c]);
        }
        const R a1 = mad(p.hp, ns[k], -corr);
        const R b = mad(p.hm, na[k], -p.force[k]);
        if (ONE_ROUNDING) {
            g[q] = g[q] - (a1 + b);
            g[q + 1] = g[q + 1] - (a1 - b);
        } else {
            g[q] = (g[q] - a1) - b;
            g[q + 1] = (g[q + 1] - a1) + b;
        }
    }
}

// Step collision: the lean SRT/TRT update, or MRT.
template <typename R, bool RHO0_IS_RHO, bool MRT, bool ONE_ROUNDING>
__device__ __forceinline__ void collide_any(R g[Q], const Relax<R> &p)
{
    if constexpr (MRT)
        collide_mrt<R, RHO0_IS_RHO, ONE_ROUNDING>(g, p);
    else
        collide_lean<R, RHO0_IS_RHO, ONE_ROUNDING>(g, p);
}

// Shifted equilibrium geq_q = feq_q(rho, u) - w_q for all q (lbm_init).
template <typename R>
__device__ __forceinline__ void equilibrium_all(R rho, const R u[3], const Coll<R> &p, R g[Q])
{
    R drho = rho - R(1);
    R rho0 = p.rho0_is_rho ? rho : R(1);
    R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    g[0] = rest_equilibrium(uu, drho, rho0, p.kappa);
#define LBM_EQ_PAIR(k)                                                              \
    {                                                                               \
        R s_, a_;                                                                   \
        pair_equilibrium<R, 2 * k + 1>(u, uu, drho, rho0, p.kappa, s_, a_);         \
        g[2 * k + 1] = s_ + a_;                                                     \
        g[2 * k + 2] = s_ - a_;                                                     \
    }
    LBM_EQ_PAIR(0) LBM_EQ_PAIR(1) LBM_EQ_PAIR(2) LBM_EQ_PAIR(3) LBM_EQ_PAIR(4)
    LBM_EQ_PAIR(5) LBM_EQ_PAIR(6) LBM_EQ_PAIR(7) LBM_EQ_PAIR(8)
#undef LBM_EQ_PAIR
}

}  // namespace lbm
