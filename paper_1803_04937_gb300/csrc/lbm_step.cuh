// Fused stream + collide time step (Eq. 15; D3Q19-S / D3Q19-I equilibria;
// SRT / TRT; periodic or half-way bounce-back; Buick-Greated force): kernel
// templates, instantiated per storage precision in lbm_step_<prec>.cu.
//
// Each thread gathers the populations that stream into its cell(s), collides
// them in registers (FP32, or FP64 for FP64 storage) and stores the
// post-collision values.  Structure-of-arrays storage gives coalesced accesses
// along x for every population.  Algorithmic traffic: 19 loads + 19 stores
// per cell.
//
// Address arithmetic is kept to one 32-bit index per access: the base pointer
// of each population plane comes from the kernel parameters (a table of 19
// pointers) and the nine source/target row offsets (y +- 1, z +- 1, wrapped)
// are formed once per thread.  WALLS = false compiles the periodic lattice
// without any bounce-back logic.
//
// Three thread mappings, each over the lattice as one sequence of cells, pairs or
// quads (Box):
//  - one cell per thread (any nx; the FP32 and FP64 default): scalar loads;
//    the +-x populations are read one element off alignment, which L1/L2
//    absorb without extra DRAM traffic.
//  - two neighbouring cells per thread (nx even): every population is read
//    and written as an aligned pair (half2 / bfloat162 / float2 / double2);
//    a +-x shifted pair is assembled from the own pair and one element of the
//    neighbouring lane's pair (warp shuffle), with one scalar access at the
//    ends of the warp's part of a row.  (16-bit A/B steps form it from two words
//    by a funnel shift instead, k_ab2w.)
//  - four cells per thread (16-bit storage, nx % 4 == 0; the 16-bit default):
//    8-byte quads of raw 16-bit codes; a +-x shifted window is formed from the
//    aligned quad and its aligned neighbour quad by funnel shifts (load4w).
#pragma once

#include <type_traits>
#include <utility>

#include "lbm_device.cuh"
#include "lbm_launch.h"

namespace lbm {

template <typename T> struct Planes {
    T *p[Q];
};

template <typename T>
static inline Planes<T> planes_of(void *base, long long ncell)
{
    Planes<T> r;
    for (int q = 0; q < Q; ++q) r.p[q] = (T *)base + (long long)q * ncell;
    return r;
}

// Per-thread lattice geometry: wrapped neighbour coordinates, the nine row
// offsets of the rows y + dy, z + dz (dy, dz in {-1, 0, 1}) and, with walls,
// the wall flags of the six faces of the cell(s).
template <bool WALLS>
struct Site {
    int x, xm, xp;      // x and its wrapped neighbours (first cell of the thread)
    int row[3][3];      // row[dy + 1][dz + 1] = ((z + dz) ny + (y + dy)) nx, wrapped
    int own;            // row[1][1]
    bool bxm, bxp, bym, byp, bzm, bzp;

    __device__ __forceinline__ Site(int x_, int y, int z, int span, const Geo &g)
    {
        x = x_;
        xm = x == 0 ? g.nx - 1 : x - 1;
        xp = x + span >= g.nx ? x + span - g.nx : x + span;  // first cell after the thread's span
        const int ym = y == 0 ? g.ny - 1 : y - 1;
        const int yp = y == g.ny - 1 ? 0 : y + 1;
        const int zm = z == 0 ? g.nz - 1 : z - 1;
        const int zp = z == g.nz - 1 ? 0 : z + 1;
        const int nxy = g.nx * g.ny;
        const int ys[3] = {ym, y, yp}, zs[3] = {zm, z, zp};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) row[a][b] = zs[b] * nxy + ys[a] * g.nx;
        own = row[1][1];
        if (WALLS) {
            bxm = g.wall_x && x == 0;
            bxp = g.wall_x && x + span >= g.nx;
            bym = g.wall_y && y == 0;
            byp = g.wall_y && y == g.ny - 1;
            bzm = g.wall_z && z == 0;
            bzp = g.wall_z && z == g.nz - 1;
        } else {
            bxm = bxp = bym = byp = bzm = bzp = false;
        }
    }

    // Does the link from the cell along s * c_q cross a y/z wall?
    template <int S>
    __device__ __forceinline__ bool wall_yz(int q) const
    {
        if (!WALLS) return false;
        const int cy = S * CY(q), cz = S * CZ(q);
        bool w = false;
        if (cy > 0) w |= byp;
        if (cy < 0) w |= bym;
        if (cz > 0) w |= bzp;
        if (cz < 0) w |= bzm;
        return w;
    }
    template <int S>
    __device__ __forceinline__ int row_along(int q) const
    {
        return row[S * CY(q) + 1][S * CZ(q) + 1];
    }
};

// For rows that touch no y/z wall: the y/z wall flags are constant false, so
// only the x-wall selects remain.
template <bool WALLS>
__device__ __forceinline__ void drop_yz(Site<WALLS> &s)
{
    s.bym = s.byp = s.bzm = s.bzp = false;
}

// An in-place step writes the locations it has read; left alone, the compiler
// keeps the 19 load addresses (64-bit each) alive through the collisions to
// reuse them for the stores, and spills.  Passing the offsets through an
// empty asm statement hides that equality, so the store addresses are formed
// again from the kernel-parameter base pointers after the collisions.
__device__ __forceinline__ void opaque(int &v) { asm volatile("" : "+r"(v)); }
template <bool WALLS>
__device__ __forceinline__ void opaque(Site<WALLS> &s)
{
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) opaque(s.row[a][b]);
    opaque(s.own);
    opaque(s.x);
    opaque(s.xm);
    opaque(s.xp);
}

// ---------------------------------------------------------------- pairs

template <typename T> struct Pair;
template <> struct Pair<float> {
    static __device__ __forceinline__ void load(const float *p, float &a, float &b)
    {
        float2 v = *reinterpret_cast<const float2 *>(p);
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void store(float *p, float a, float b)
    {
        *reinterpret_cast<float2 *>(p) = make_float2(a, b);
    }
};
template <> struct Pair<double> {
    static __device__ __forceinline__ void load(const double *p, double &a, double &b)
    {
        double2 v = *reinterpret_cast<const double2 *>(p);
        a = v.x;
        b = v.y;
    }
    static __device__ __forceinline__ void store(double *p, double a, double b)
    {
        *reinterpret_cast<double2 *>(p) = make_double2(a, b);
    }
};
template <> struct Pair<__half> {
    static __device__ __forceinline__ void load(const __half *p, float &a, float &b)
    {
        __half2 v = *reinterpret_cast<const __half2 *>(p);
        a = __low2float(v);
        b = __high2float(v);
    }
    static __device__ __forceinline__ void store(__half *p, float a, float b)
    {
        *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a, b);
    }
};
template <> struct Pair<__nv_bfloat16> {
    static __device__ __forceinline__ void load(const __nv_bfloat16 *p, float &a, float &b)
    {
        __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(p);
        a = __low2float(v);
        b = __high2float(v);
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, float a, float b)
    {
        *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
    }
};

// ---------------------------------------------------------------- one cell per thread

// Gather of the populations streaming into one cell.  SWAP = false: A/B
// layout (plane q at x - c_q; through a wall, plane qbar of the own cell);
// SWAP = true: AA odd layout (plane qbar at x - c_q; through a wall, plane q
// of the own cell).
template <bool SWAP, bool WALLS, typename T, typename R>
__device__ __forceinline__ void gather1(const Planes<T> &P, const Site<WALLS> &s, R f[Q])
{
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const int xs = cx == 0 ? s.x : (cx > 0 ? s.xm : s.xp);
        bool w = s.template wall_yz<-1>(q);
        if (WALLS) {
            if (cx > 0) w |= s.bxm;
            if (cx < 0) w |= s.bxp;
        }
        const T *src = SWAP ? P.p[OPP(q)] : P.p[q];
        const T *bnc = SWAP ? P.p[q] : P.p[OPP(q)];
        const T *a = w ? bnc + s.own + s.x : src + s.template row_along<-1>(q) + xs;
        f[q] = Storage<T>::load(a);
    }
}

// Gather, collision and stores of k_ab1 for one cell.
template <typename T, bool RHO0, bool WALLS, bool MRT>
__device__ __forceinline__ void ab1_body(const Planes<T> &src, const Planes<T> &dst, const Site<WALLS> &s,
                                         const Relax<typename Storage<T>::R> &p)
{
    using R = typename Storage<T>::R;
    R f[Q];
    gather1<false>(src, s, f);
    collide_any<R, RHO0, MRT, one_rounding_v<T>>(f, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) Storage<T>::store(dst.p[q] + s.own + s.x, f[q]);
}

template <typename T, bool RHO0, bool WALLS, bool MRT = false>
__global__ void __launch_bounds__(256) k_ab1(Planes<T> src, Planes<T> dst, Geo g, Relax<typename Storage<T>::R> p,
                                             Box box)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= box.count) return;
    int x, y, z;
    box.at(i, x, y, z);
    step_begin(box);
    if constexpr (WALLS) {
        // warps with no cell at a wall take the periodic body (uniform branch per warp)
        const Site<true> sw(x, y, z, 1, g);
        const bool touches = sw.bxm || sw.bxp || sw.bym || sw.byp || sw.bzm || sw.bzp;
        if (__any_sync(__activemask(), touches)) {
            ab1_body<T, RHO0, true, MRT>(src, dst, sw, p);
            return;
        }
    }
    ab1_body<T, RHO0, false, MRT>(src, dst, Site<false>(x, y, z, 1, g), p);
}

// Blocks per SM the one-cell AA steps are compiled for.  With the compensated
// momentum sum of FP32 storage the compiler's own choice for the odd step is
// 94 registers, two blocks of 256 threads per SM (FP32 AA pair 0.98 -> 0.83
// of the copy bandwidth at 256^3).  Measured for the FP32 SRT/TRT pair
// (even, odd blocks; 256^3 / 768^3): (5, 3) 0.932 / 0.943 (odd step 80
// registers, 16 bytes spilled; even 48, none), (6, 3) 0.911 / 0.924, (5, 2)
// 0.889 / 0.897, (6, 4) 0.859 / 0.871; (5, 3) is kept.
template <typename T, bool MRT>
constexpr int aa1_blocks(bool odd)
{
    return (std::is_same<T, float>::value && !MRT) ? (odd ? 3 : 5) : 1;
}

// AA even step: own cell only (read plane q, write plane qbar).  The store
// side takes its own copy of the plane table (the same pointers): given one
// table, the compiler keeps its 19 pointers in registers between the loads and
// the stores (80 instead of 40 registers; +1.5 % FP32, +2.8 % FP64 measured).
template <typename T, bool RHO0, bool MRT = false>
__global__ void __launch_bounds__(256, aa1_blocks<T, MRT>(false)) k_aa_even1(Planes<T> P, Planes<T> Pw, Geo g,
                                                                           Relax<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    const unsigned own = blockIdx.x * blockDim.x + threadIdx.x;
    if (own >= (unsigned)g.ncell) return;
    step_begin(box);
    R f[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q] = Storage<T>::load(P.p[q] + own);
    collide_any<R, RHO0, MRT, one_rounding_v<T>>(f, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) Storage<T>::store(Pw.p[OPP(q)] + own, f[q]);
}

// AA odd step: read plane qbar at x - c_q, write plane q at x + c_q (through
// a wall: read plane q / write plane qbar of the own cell).  Every location is
// read and written by exactly one thread.
template <typename T, bool RHO0, bool MRT, bool WALLS>
__device__ __forceinline__ void aa_odd1_body(const Planes<T> &P, const Site<WALLS> &s,
                                             const Relax<typename Storage<T>::R> &p)
{
    using R = typename Storage<T>::R;
    R f[Q];
    gather1<true>(P, s, f);
    collide_any<R, RHO0, MRT, one_rounding_v<T>>(f, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const int xt = cx == 0 ? s.x : (cx > 0 ? s.xp : s.xm);
        bool w = s.template wall_yz<1>(q);
        if (WALLS) {
            if (cx > 0) w |= s.bxp;
            if (cx < 0) w |= s.bxm;
        }
        T *a = w ? P.p[OPP(q)] + s.own + s.x : P.p[q] + s.template row_along<1>(q) + xt;
        Storage<T>::store(a, f[q]);
    }
}

template <typename T, bool RHO0, bool MRT = false>
__global__ void __launch_bounds__(256, aa1_blocks<T, MRT>(true)) k_aa_odd1(Planes<T> P, Geo g,
                                                                         Relax<typename Storage<T>::R> p, Box box)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= box.count) return;
    int x, y, z;
    box.at(i, x, y, z);
    step_begin(box);
    aa_odd1_body<T, RHO0, MRT>(P, Site<false>(x, y, z, 1, g), p);
}

// With walls (WalledBox); XWALLS: walls on x too.
template <typename T, bool RHO0, bool MRT, bool XWALLS>
__global__ void __launch_bounds__(256, aa1_blocks<T, MRT>(true)) k_aa_odd1_walls(Planes<T> P, Geo g,
                                                                               Relax<typename Storage<T>::R> p,
                                                                               WalledBox box)
{
    int x, y, z;
    if (box.at_walls()) {
        const unsigned i = box.wall_item();
        if (i >= box.walls.count) return;
        box.walls.at_wall(i, x, y, z);
        step_begin(box);
        aa_odd1_body<T, RHO0, MRT>(P, Site<true>(x, y, z, 1, g), p);
    } else {
        const unsigned i = box.inner_item();
        if (i >= box.inner.count) return;
        box.inner.at(i, x, y, z);
        step_begin(box);
        Site<XWALLS> s(x, y, z, 1, g);
        drop_yz(s);
        aa_odd1_body<T, RHO0, MRT>(P, s, p);
    }
}

// ---------------------------------------------------------------- two cells per thread

// The pair of a thread of a sequence of pairs (Box), and its place in the warp:
// head / last pair of the warp's part of a row (a warp may hold several rows'
// ends).  Threads past the end repeat the last pair and take part in the shuffles.
struct PairAt {
    int x0, y, z;
    bool active, head, last;

    __device__ __forceinline__ explicit PairAt(const Box &box) : PairAt(box, blockIdx.x * blockDim.x + threadIdx.x) {}
    __device__ __forceinline__ PairAt(const Box &box, unsigned i, bool wall_rows = false)
    {
        const int lane = threadIdx.x & 31;
        active = i < box.count;
        int xp;
        if (wall_rows) box.at_wall(active ? i : box.count - 1u, xp, y, z);
        else box.at(active ? i : box.count - 1u, xp, y, z);
        x0 = 2 * xp;
        head = lane == 0 || xp == 0;
        last = lane == 31 || xp + 1 == (int)box.per_row.d || i + 1 >= box.count;
    }
};

// Pair-wise gather for the cells (x0, x0 + 1), x0 even, nx even (layouts as
// in gather1).
template <bool SWAP, bool WALLS, typename T, typename R>
__device__ __forceinline__ void gather2(const Planes<T> &P, const Site<WALLS> &s, const PairAt &at, R f0[Q], R f1[Q])
{
    const int x0 = s.x;
    const bool active = at.active, last = at.last;
    // Phase 1: issue every load before any shuffle.  lo/hi: the own pair of
    // the source row (or, through a y/z wall, the own cell's reflected pair);
    // e: the element beyond the segment's edge for the +-x populations.
    R lo[Q], hi[Q], e[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<-1>(q);
        const T *src = SWAP ? P.p[OPP(q)] : P.p[q];
        const T *bnc = SWAP ? P.p[q] : P.p[OPP(q)];
        const int srow = s.template row_along<-1>(q);
        Pair<T>::load(w ? bnc + s.own + x0 : src + srow + x0, lo[q], hi[q]);
        e[q] = R(0);
        if (cx > 0) {  // pull from x - 1: lane 0 needs element x0 - 1
            const T *a = (WALLS && s.bxm) ? bnc + s.own + x0 : src + srow + s.xm;
            if (at.head && active && !w) e[q] = Storage<T>::load(a);
        } else if (cx < 0) {  // pull from x + 1: the segment's last lane needs element x0 + 2
            const T *a = (WALLS && s.bxp) ? bnc + s.own + x0 + 1 : src + srow + s.xp;
            if (last && active && !w) e[q] = Storage<T>::load(a);
        }
    }
    // Phase 2: assemble the shifted pairs.
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<-1>(q);
        if (cx == 0) {
            f0[q] = lo[q];
            f1[q] = hi[q];
        } else if (cx > 0) {
            R left = __shfl_up_sync(0xffffffffu, hi[q], 1);
            if (at.head) left = e[q];
            f0[q] = w ? lo[q] : left;
            f1[q] = w ? hi[q] : lo[q];
        } else {
            R right = __shfl_down_sync(0xffffffffu, lo[q], 1);
            if (last) right = e[q];
            f0[q] = w ? lo[q] : hi[q];
            f1[q] = w ? hi[q] : right;
        }
    }
}

template <typename T, bool RHO0, bool WALLS>
__global__ void __launch_bounds__(256, 4) k_ab2(Planes<T> src, Planes<T> dst, Geo g, Relax<typename Storage<T>::R> p,
                                                Box box)
{
    using R = typename Storage<T>::R;
    const PairAt at(box);
    const Site<WALLS> s(at.x0, at.y, at.z, 2, g);
    step_begin(box);
    R f0[Q], f1[Q];
    gather2<false>(src, s, at, f0, f1);
    if (!at.active) return;
    const int x0 = at.x0;
    collide_lean<R, RHO0, one_rounding_v<T>>(f0, p);
    collide_lean<R, RHO0, one_rounding_v<T>>(f1, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) Pair<T>::store(dst.p[q] + s.own + x0, f0[q], f1[q]);
}

template <typename T, bool RHO0>
__global__ void __launch_bounds__(256) k_aa_even2(Planes<T> P, Geo g, Relax<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    int own = 2 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if ((unsigned)own >= (unsigned)g.ncell) return;
    opaque(own);
    step_begin(box);
    R f0[Q], f1[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) Pair<T>::load(P.p[q] + own, f0[q], f1[q]);
    collide_lean<R, RHO0, one_rounding_v<T>>(f0, p);
    collide_lean<R, RHO0, one_rounding_v<T>>(f1, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) Pair<T>::store(P.p[OPP(q)] + own, f0[q], f1[q]);
}

// AA odd step, two cells per thread: gather plane qbar from x - c_q (pairs),
// collide, and write plane q at x + c_q.  A +-x shifted write is assembled
// into the aligned pair (x0, x0 + 1) of the target row from the own values and
// the neighbouring lane's (warp shuffle); the element that belongs to the
// neighbouring segment is written by the edge lane as a scalar.  Through a
// wall the value goes to plane qbar of the own cell.  Every location is
// written by exactly one thread, as in the one-cell kernel.
template <typename T, bool RHO0, bool WALLS>
__device__ __forceinline__ void aa_odd2_body(const Planes<T> &P, const Site<WALLS> &s, const PairAt &at,
                                             const Relax<typename Storage<T>::R> &p)
{
    using R = typename Storage<T>::R;
    const int x0 = at.x0;
    const bool active = at.active, head = at.head, last = at.last;
    R f0[Q], f1[Q];
    gather2<true>(P, s, at, f0, f1);
    if (active) {
        collide_lean<R, RHO0, one_rounding_v<T>>(f0, p);
        collide_lean<R, RHO0, one_rounding_v<T>>(f1, p);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<1>(q);
        T *dst = P.p[q];
        T *bnc = P.p[OPP(q)];
        const int trow = s.template row_along<1>(q);
        if (cx == 0) {
            if (active) Pair<T>::store(w ? bnc + s.own + x0 : dst + trow + x0, f0[q], f1[q]);
        } else if (cx > 0) {
            // element x0 of the target row receives cell x0 - 1, element x0 + 1 cell x0
            const R left = __shfl_up_sync(0xffffffffu, f1[q], 1);
            if (!active) continue;
            if (w) {
                Pair<T>::store(bnc + s.own + x0, f0[q], f1[q]);
                continue;
            }
            if (head)
                Storage<T>::store(dst + trow + x0 + 1, f0[q]);
            else
                Pair<T>::store(dst + trow + x0, left, f0[q]);
            if (last)  // cell x0 + 1 goes to x0 + 2: the next segment, the periodic image, or a wall
                Storage<T>::store((WALLS && s.bxp) ? bnc + s.own + x0 + 1 : dst + trow + s.xp, f1[q]);
        } else {
            // element x0 of the target row receives cell x0 + 1, element x0 + 1 cell x0 + 2
            const R right = __shfl_down_sync(0xffffffffu, f0[q], 1);
            if (!active) continue;
            if (w) {
                Pair<T>::store(bnc + s.own + x0, f0[q], f1[q]);
                continue;
            }
            if (last)
                Storage<T>::store(dst + trow + x0, f1[q]);
            else
                Pair<T>::store(dst + trow + x0, f1[q], right);
            if (head)  // cell x0 goes to x0 - 1: the previous segment, the periodic image, or a wall
                Storage<T>::store((WALLS && s.bxm) ? bnc + s.own + x0 : dst + trow + s.xm, f0[q]);
        }
    }
}

template <typename T, bool RHO0>
__global__ void __launch_bounds__(256, 2) k_aa_odd2(Planes<T> P, Geo g, Relax<typename Storage<T>::R> p, Box box)
{
    const PairAt at(box);
    const Site<false> s(at.x0, at.y, at.z, 2, g);
    step_begin(box);
    aa_odd2_body<T, RHO0>(P, s, at, p);
}

// With walls, as k_aa_odd1_walls.
template <typename T, bool RHO0, bool XWALLS>
__global__ void __launch_bounds__(256, 2) k_aa_odd2_walls(Planes<T> P, Geo g, Relax<typename Storage<T>::R> p,
                                                          WalledBox box)
{
    if (box.at_walls()) {
        const PairAt at(box.walls, box.wall_item(), true);
        const Site<true> s(at.x0, at.y, at.z, 2, g);
        step_begin(box);
        aa_odd2_body<T, RHO0>(P, s, at, p);
    } else {
        const PairAt at(box.inner, box.inner_item());
        Site<XWALLS> s(at.x0, at.y, at.z, 2, g);
        drop_yz(s);
        step_begin(box);
        aa_odd2_body<T, RHO0>(P, s, at, p);
    }
}

// ---------------------------------------------------------------- four cells per thread (16-bit storage)

// Raw 16-bit codes <-> float for the 16-bit storage types.
template <typename T> struct Bits16;
template <> struct Bits16<__half> {
    static __device__ __forceinline__ float to_float(unsigned int b)
    {
        return __half2float(__ushort_as_half((unsigned short)b));
    }
    static __device__ __forceinline__ unsigned int from_float(float v)
    {
        return __half_as_ushort(__float2half_rn(v));
    }
};
template <> struct Bits16<__nv_bfloat16> {
    static __device__ __forceinline__ float to_float(unsigned int b)
    {
        return __bfloat162float(__ushort_as_bfloat16((unsigned short)b));
    }
    static __device__ __forceinline__ unsigned int from_float(float v)
    {
        return __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
};

// Element c (0..3) of four 16-bit codes packed in a uint2, and its replacement.
template <int c>
__device__ __forceinline__ unsigned int quad_get(const uint2 &v)
{
    const unsigned int w = c < 2 ? v.x : v.y;
    return (c & 1) ? (w >> 16) : (w & 0xffffu);
}
template <int c>
__device__ __forceinline__ void quad_set(uint2 &v, unsigned int b)
{
    unsigned int &w = c < 2 ? v.x : v.y;
    w = (c & 1) ? ((w & 0x0000ffffu) | (b << 16)) : ((w & 0xffff0000u) | (b & 0xffffu));
}

// Phase 1, windowed: for every population the four inputs of the cells
// x0 .. x0 + 3 as one 8-byte window of raw 16-bit codes.  A +-x shifted
// window is assembled from the aligned quad and its aligned neighbour quad
// (x0 - 4 or x0 + 4, wrapped) by two funnel shifts, so no lane needs another
// lane's data; the neighbour quads are the lines the adjacent lanes load
// anyway (L1 hits; no extra DRAM traffic).  Through a y/z wall the window is
// the own cells' reflected quad; at an x wall the element beyond the wall is
// the own cell's reflected slot.  SWAP as in load4.
template <bool SWAP, bool WALLS, typename T>
__device__ __forceinline__ void load4w(const Planes<T> &P, const Site<WALLS> &s, const Geo &g, uint2 (&win)[Q])
{
    const int xs = s.x;
    const int xprev = xs == 0 ? g.nx - 4 : xs - 4;
    const int xnext = xs + 4 >= g.nx ? 0 : xs + 4;
    uint2 nb[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<-1>(q);
        const unsigned short *srcq = reinterpret_cast<const unsigned short *>(SWAP ? P.p[OPP(q)] : P.p[q]);
        const unsigned short *bncq = reinterpret_cast<const unsigned short *>(SWAP ? P.p[q] : P.p[OPP(q)]);
        const int srow = s.template row_along<-1>(q);
        const uint2 *pq = reinterpret_cast<const uint2 *>(w ? bncq + s.own + xs : srcq + srow + xs);
        const uint2 *pn = reinterpret_cast<const uint2 *>(srcq + srow + (cx > 0 ? xprev : xnext));
        const bool xwall = WALLS && ((cx > 0 && s.bxm) || (cx < 0 && s.bxp));
        if (xwall && !w) pn = reinterpret_cast<const uint2 *>(bncq + s.own + xs);
        // The in-place AA odd step (SWAP) takes non-coherent loads (FP16 0.797 -> 0.803,
        // BF16 0.774 -> 0.791 of the copy bandwidth at 256^3): the elements it uses of
        // a quad are its own cells' inputs, which only this thread writes, and only
        // after it has read them; the other elements of a neighbour quad may be stale
        // and are not used.  Such a launch must not start before the end of the one
        // whose results it reads (launch_step_kernel).
        win[q] = SWAP ? __ldg(pq) : *pq;
        if (cx != 0) nb[q] = w ? make_uint2(0u, 0u) : (SWAP ? __ldg(pn) : *pn);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<-1>(q);
        if (cx == 0 || w) continue;
        const uint2 c = win[q];
        uint2 n = nb[q];
        if (cx > 0) {
            // [x0 - 1, x0, x0 + 1, x0 + 2]: element 3 of the quad before (or the reflected x0)
            if (WALLS && s.bxm) n.y = n.x << 16;
            win[q].x = __funnelshift_l(n.y, c.x, 16);
            win[q].y = __funnelshift_l(c.x, c.y, 16);
        } else {
            // [x0 + 1, x0 + 2, x0 + 3, x0 + 4]: element 0 of the quad after (or the reflected x0 + 3)
            if (WALLS && s.bxp) n.x = n.y >> 16;
            win[q].x = __funnelshift_r(c.x, c.y, 16);
            win[q].y = __funnelshift_r(c.y, n.x, 16);
        }
    }
}

// Four collisions on windows: element c of every population's window is the
// input of cell c, and its result is written back into element c.
template <typename T, bool RHO0, bool MRT = false>
__device__ __forceinline__ void collide4(uint2 (&win)[Q], const Relax<float> &p)
{
#define LBM_AB4_CELL(c)                                                                      \
    {                                                                                        \
        float f[Q];                                                                          \
        _Pragma("unroll") for (int q = 0; q < Q; ++q) f[q] = Bits16<T>::to_float(quad_get<c>(win[q]));   \
        collide_any<float, RHO0, MRT, false>(f, p);                                          \
        _Pragma("unroll") for (int q = 0; q < Q; ++q) quad_set<c>(win[q], Bits16<T>::from_float(f[q]));  \
    }
    LBM_AB4_CELL(0) LBM_AB4_CELL(1) LBM_AB4_CELL(2) LBM_AB4_CELL(3)
#undef LBM_AB4_CELL
}

// A/B pull step for 16-bit storage, four cells (x0 .. x0 + 3) per thread,
// x0 a multiple of 4, nx a multiple of 4: every population is read and
// written as 8-byte quads, so the address work is shared by four cells.  The
// shifted inputs come from the aligned quad and its aligned neighbour by
// funnel shifts (load4w), so no lane waits for another; the four results are
// written back into the windows in place.  Replacing the earlier gather
// (neighbour elements by warp shuffles and a carry chain through the four
// cells) took this step from 0.88 to 1.04 of the measured copy bandwidth.
// Bitwise the same results as the one- and two-cell kernels.
// Loads, four collisions and stores of k_ab4 for one thread's quad.
template <typename T, bool RHO0, bool WALLS, bool MRT>
__device__ __forceinline__ void ab4_body(const Planes<T> &src, const Planes<T> &dst, const Site<WALLS> &s,
                                         const Geo &g, const Relax<float> &p)
{
    uint2 win[Q];
    load4w<false>(src, s, g, win);
    collide4<T, RHO0, MRT>(win, p);
#pragma unroll
    for (int q = 0; q < Q; ++q)
        *reinterpret_cast<uint2 *>(reinterpret_cast<unsigned short *>(dst.p[q]) + s.own + s.x) = win[q];
}

// Blocks per SM of the periodic step: five, but four where five leave BF16 short of
// registers (256^3: MRT 221 -> 209 us, rho0 = rho 215 -> 212; the others 7 to 20 % slower).
template <typename T, bool RHO0, bool MRT>
constexpr int ab4_blocks = std::is_same_v<T, __nv_bfloat16> && MRT != RHO0 ? 4 : 5;

template <typename T, bool RHO0, bool MRT = false>
__global__ void __launch_bounds__(128, ab4_blocks<T, RHO0, MRT>) k_ab4(Planes<T> src, Planes<T> dst, Geo g, Relax<float> p, Box box)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= box.count) return;  // no lane needs another lane's data
    int xq, y, z;
    box.at(i, xq, y, z);
    const Site<false> s(4 * xq, y, z, 4, g);
    step_begin(box);
    ab4_body<T, RHO0, false, MRT>(src, dst, s, g, p);
}

// With walls (WalledBox); XWALLS: walls on x too, whose selects cost the rows
// between the y and z walls little (the end quads' shifted windows take the
// reflected own quad).
template <typename T, bool RHO0, bool MRT, bool XWALLS>
__global__ void __launch_bounds__(128, 5) k_ab4_walls(Planes<T> src, Planes<T> dst, Geo g, Relax<float> p, WalledBox box)
{
    int xq, y, z;
    if (box.at_walls()) {
        const unsigned i = box.wall_item();
        if (i >= box.walls.count) return;
        box.walls.at_wall(i, xq, y, z);
        const Site<true> s(4 * xq, y, z, 4, g);
        step_begin(box);
        ab4_body<T, RHO0, true, MRT>(src, dst, s, g, p);
    } else {
        const unsigned i = box.inner_item();
        if (i >= box.inner.count) return;
        box.inner.at(i, xq, y, z);
        Site<XWALLS> s(4 * xq, y, z, 4, g);
        drop_yz(s);
        step_begin(box);
        ab4_body<T, RHO0, XWALLS, MRT>(src, dst, s, g, p);
    }
}

// A/B pull step for 16-bit storage whose rows hold pairs but not quads of cells
// (nx even): the same windows, of two codes in a 32-bit word.
// 190x131x97 FP16 42.8 -> 37.5 us against the shuffles of k_ab2, with walls on all
// axes 62.8 -> 37.9; blocks per SM 5 / 6 / 8: 37.5 / 39.3 / 38.1 us, with walls
// 39.6 / 37.9 / 44.2.
template <typename T, bool RHO0, bool WALLS>
__global__ void __launch_bounds__(128, WALLS ? 6 : 5) k_ab2w(Planes<T> src, Planes<T> dst, Geo g, Relax<float> p, Box box)
{
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= box.count) return;
    int xp, y, z;
    box.at(i, xp, y, z);
    const Site<WALLS> s(2 * xp, y, z, 2, g);
    step_begin(box);
    const int xprev = s.x == 0 ? g.nx - 2 : s.x - 2;
    const int xnext = s.x + 2 >= g.nx ? 0 : s.x + 2;
    unsigned win[Q], nb[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<-1>(q);
        const unsigned short *from = reinterpret_cast<const unsigned short *>(src.p[q]) + s.template row_along<-1>(q);
        const unsigned short *own = reinterpret_cast<const unsigned short *>(src.p[OPP(q)]) + s.own + s.x;
        win[q] = *reinterpret_cast<const unsigned *>(w ? own : from + s.x);
        if (cx != 0) {
            const bool xwall = WALLS && ((cx > 0 && s.bxm) || (cx < 0 && s.bxp));
            nb[q] = *reinterpret_cast<const unsigned *>(xwall ? own : from + (cx > 0 ? xprev : xnext));
        }
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        if (cx == 0 || s.template wall_yz<-1>(q)) continue;
        if (cx > 0)  // [x0 - 1, x0]: element 1 of the pair before (or the reflected x0)
            win[q] = __funnelshift_l(WALLS && s.bxm ? nb[q] << 16 : nb[q], win[q], 16);
        else         // [x0 + 1, x0 + 2]: element 0 of the pair after (or the reflected x0 + 1)
            win[q] = __funnelshift_r(win[q], WALLS && s.bxp ? nb[q] >> 16 : nb[q], 16);
    }
    float f[Q];
    unsigned low[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) f[q] = Bits16<T>::to_float(win[q] & 0xffffu);
    collide_lean<float, RHO0, false>(f, p);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        low[q] = Bits16<T>::from_float(f[q]);
        f[q] = Bits16<T>::to_float(win[q] >> 16);
        win[q] = low[q];
    }
    collide_lean<float, RHO0, false>(f, p);
#pragma unroll
    for (int q = 0; q < Q; ++q)
        *reinterpret_cast<unsigned *>(reinterpret_cast<unsigned short *>(dst.p[q]) + s.own + s.x) =
            (Bits16<T>::from_float(f[q]) << 16) | (win[q] & 0xffffu);
}

// AA even step for 16-bit storage, four cells per thread: own quads of plane
// q in, own quads of plane qbar out.  The stores take their own copy of the
// plane table (see k_aa_even1), which lets the step run five blocks per SM
// without spills (96 registers; with one table it needed 128).
template <typename T, bool RHO0, bool MRT = false>
__global__ void __launch_bounds__(128, 5) k_aa_even4(Planes<T> P, Planes<T> Pw, Geo g, Relax<float> p, Box box)
{
    int own = 4 * (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if ((unsigned)own >= (unsigned)g.ncell) return;
    opaque(own);  // (left to see through it, the compiler spills 96 bytes)
    step_begin(box);
    uint2 quad[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q)
        quad[q] = *reinterpret_cast<const uint2 *>(reinterpret_cast<const unsigned short *>(P.p[q]) + own);
    collide4<T, RHO0, MRT>(quad, p);
    int own_w = own;
    opaque(own_w);
#pragma unroll
    for (int q = 0; q < Q; ++q)
        *reinterpret_cast<uint2 *>(reinterpret_cast<unsigned short *>(Pw.p[OPP(q)]) + own_w) = quad[q];
}

// AA odd step for 16-bit storage, four cells per thread: gather plane qbar
// from x - c_q (as k_ab4 with the planes swapped), collide, and write plane q
// at x + c_q.  A +-x shifted write is assembled into the aligned quad
// (x0 .. x0 + 3) of the target row from three own results and one of the
// neighbouring lane (warp shuffle); at a segment's edge the lane writes the
// three own elements of the aligned quad and the edge lane writes the fourth
// result as a scalar into the neighbouring segment (or its periodic image, or
// through an x wall into plane qbar of the own cell).  Through a y/z wall the
// quad goes to plane qbar of the own cells.  Each location is written by one
// thread, and read (for a value that is used) only by that thread, as in the
// one-cell kernel.
// FORM: how the quads are walked (SEQUENCE_CACHED on periodic lattices only).  ROWS_OF_BLOCKS: in blocks that are rectangles
// of rows, whose rows a warp does not leave; the fastest from DRAM where rows fill
// them (step of a pair, 256^3: FP16 208 us against 227, BF16 212 against 229).
// SEQUENCE: as one sequence (192^3 FP16: 95 against 108 us, 160^3 60 against 74).
// SEQUENCE_CACHED: the same for lattices that stay in L2 (128^3 FP16 22.8 against
// 26.8 us); it differs in the branch before the loads, without which the compiler
// spreads them among the collisions: that saves its spills, but leaves too few
// loads in flight for DRAM (192^3 FP16: 99 us).
enum OddForm { ROWS_OF_BLOCKS, SEQUENCE, SEQUENCE_CACHED };
// With walls (WalledBox) the wall rows are stepped cell by cell, and the rows
// between them keep the x-wall selects also without walls on x (the flags are then
// false).  Both in one launch: a launch of its own for the wall rows after the other
// costs a small lattice a second launch (closed box 32^3 FP16, step of a pair: 5.3
// against 3.0 us; 96^3 15.6 against 11.7).  At four blocks per SM instead of five
// nothing spills, and the branch is wanted by the rectangles only (256^3 with rho0 =
// rho 262 us without it, 230 with; sequences of 192^3 FP16 93 us without, 105 with,
// at five blocks 100).
template <typename T, bool RHO0, bool WALLS, bool MRT = false, OddForm FORM = SEQUENCE>
__global__ void __launch_bounds__(128, MRT || WALLS ? 4 : 5)
    k_aa_odd4(Planes<T> P, Geo g, Relax<float> p, std::conditional_t<WALLS, WalledBox, Box> box)
{
    const int lane = threadIdx.x & 31;
    constexpr bool SEQ = FORM != ROWS_OF_BLOCKS;
    int xq, y, z;
    bool active, end;  // end: the last quad there is for a warp that is not full
    if constexpr (WALLS) {
        if (box.at_walls()) {
            const unsigned i = box.wall_item();
            if (i >= box.walls.count) return;
            int x;
            box.walls.at_wall(i, x, y, z);
            aa_odd1_body<T, RHO0, MRT>(P, Site<true>(x, y, z, 1, g), p);
            return;
        }
        if constexpr (SEQ) {
            const unsigned i = box.inner_item();
            active = i < box.inner.count;
            end = i + 1 >= box.inner.count;
            box.inner.at(active ? i : box.inner.count - 1u, xq, y, z);
        } else {
            box.inner_rectangle(xq, y, z);
            if (y >= box.inner.y0 + (int)box.inner.rows.d) return;  // uniform across the warp
            active = 4 * xq < g.nx;
            xq = active ? xq : 0;
            end = false;
        }
    } else if constexpr (SEQ) {
        const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
        active = i < box.count;
        end = i + 1 >= box.count;
        box.at(active ? i : box.count - 1u, xq, y, z);
    } else {
        const int x0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
        y = blockIdx.y * blockDim.y + threadIdx.y;
        z = blockIdx.z;
        if (y >= g.ny) return;  // uniform across the warp
        active = x0 < g.nx;
        xq = active ? x0 >> 2 : 0;
        end = false;
    }
    // a branch that the loads stay behind, with nothing to wait for, before the row
    // offsets (256^3 FP16: 241 us a step without it, 215 with; with rho0 = rho no faster)
    if constexpr (FORM == ROWS_OF_BLOCKS && MRT && !RHO0 && !WALLS) {
        if (box.waits) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    Site<WALLS> s(4 * xq, y, z, 4, g);
    drop_yz(s);
    // ends of the lanes' segment of a row (a warp of a sequence may hold several rows' ends)
    const bool head = lane == 0 || (SEQ && xq == 0);
    const bool last = lane == 31 || s.x + 4 >= g.nx || end;
    // ... and after them
    if constexpr (FORM == (WALLS ? ROWS_OF_BLOCKS : SEQUENCE)) step_begin(box);
    uint2 quad[Q];
    load4w<true>(P, s, g, quad);
    if (active) collide4<T, RHO0, MRT>(quad, p);
    Site<WALLS> sw = s;
    opaque(sw);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int cx = CX(q);
        const bool w = s.template wall_yz<1>(q);
        unsigned short *dst = reinterpret_cast<unsigned short *>(P.p[q]);
        unsigned short *bnc = reinterpret_cast<unsigned short *>(P.p[OPP(q)]);
        const int trow = sw.template row_along<1>(q);
        if (cx == 0) {
            if (active) *reinterpret_cast<uint2 *>(w ? bnc + sw.own + sw.x : dst + trow + sw.x) = quad[q];
        } else if (cx > 0) {
            // target elements x0 .. x0 + 3 receive cells x0 - 1 .. x0 + 2
            const unsigned int left = __shfl_up_sync(0xffffffffu, quad[q].y >> 16, 1);
            if (!active) continue;
            if (w) {
                *reinterpret_cast<uint2 *>(bnc + sw.own + sw.x) = quad[q];
                continue;
            }
            unsigned short *t = dst + trow + sw.x;
            if (head) {  // element x0 belongs to the previous segment's last cell
                t[1] = (unsigned short)(quad[q].x & 0xffffu);
                *reinterpret_cast<unsigned int *>(t + 2) = __byte_perm(quad[q].x, quad[q].y, 0x5432);
            } else {
                uint2 v;
                v.x = __byte_perm(left, quad[q].x, 0x5410);
                v.y = __byte_perm(quad[q].x, quad[q].y, 0x5432);
                *reinterpret_cast<uint2 *>(t) = v;
            }
            if (last)  // cell x0 + 3 goes to x0 + 4: the next segment, the periodic image, or a wall
                *((WALLS && s.bxp) ? bnc + sw.own + sw.x + 3 : dst + trow + sw.xp) = (unsigned short)(quad[q].y >> 16);
        } else {
            // target elements x0 .. x0 + 3 receive cells x0 + 1 .. x0 + 4
            const unsigned int rgt = __shfl_down_sync(0xffffffffu, quad[q].x & 0xffffu, 1);
            if (!active) continue;
            if (w) {
                *reinterpret_cast<uint2 *>(bnc + sw.own + sw.x) = quad[q];
                continue;
            }
            unsigned short *t = dst + trow + sw.x;
            if (last) {  // element x0 + 3 belongs to the next segment's first cell
                *reinterpret_cast<unsigned int *>(t) = __byte_perm(quad[q].x, quad[q].y, 0x5432);
                t[2] = (unsigned short)(quad[q].y >> 16);
            } else {
                uint2 v;
                v.x = __byte_perm(quad[q].x, quad[q].y, 0x5432);
                v.y = __byte_perm(quad[q].y, rgt, 0x5432);
                *reinterpret_cast<uint2 *>(t) = v;
            }
            if (head)  // cell x0 goes to x0 - 1: the previous segment, the periodic image, or a wall
                *((WALLS && s.bxm) ? bnc + sw.own + sw.x : dst + trow + sw.xm) = (unsigned short)(quad[q].x & 0xffffu);
        }
    }
}

// ---------------------------------------------------------------- dispatch

static inline unsigned blocks_for(long long items, int threads) { return (unsigned)((items + threads - 1) / threads); }

// Launches a step kernel; early: as a programmatic dependent of the stream's
// last launch (step_begin).  Kernels with non-coherent loads are not launched early.
template <typename... P, typename... A>
static void launch_step_kernel(void (*kernel)(P...), bool early, dim3 grid, dim3 threads, cudaStream_t stream,
                               int shared_bytes, A &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = threads;
    cfg.dynamicSmemBytes = (size_t)shared_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);  // its error is the caller's cudaGetLastError
}

// ... over a box, whose rows fill blocks of bx threads along x, or (bx = 0) as
// one sequence of items; the box is the kernel's last argument.
template <typename... P, typename... A>
static void launch_step_box(void (*kernel)(P...), bool early, Box box, int bx, int threads, cudaStream_t stream,
                            A &&...args)
{
    box.waits = early;
    if (bx == 0) {
        launch_step_kernel(kernel, early, blocks_for(box.count, threads), threads, stream, 0, std::forward<A>(args)..., box);
        return;
    }
    const unsigned ux = (unsigned)bx, uy = (unsigned)(threads / bx);
    launch_step_kernel(kernel, early, dim3((box.per_row.d + ux - 1) / ux, (box.rows.d + uy - 1) / uy, (unsigned)box.nz),
                       dim3(ux, uy), stream, 0, std::forward<A>(args)..., box);
}

// ... over a lattice with walls, whose interior rows (no link crosses a y or z wall)
// run the periodic code, or with walls on x the code that has the x-wall selects
// only, and whose rows at y and z walls run the walled one.  All of them compute a
// cell with the same operations, so the results are bitwise the same.  Running the
// walled code on the wall rows only took the walled channel 512x256x256 from 84.3 to
// 89.1 GLUPS (FP16 A/B) and from 80.0 to 86.9 (BF16), and a cavity (walls on x, y and
// z) 512x256x256 from 0.76 to 0.95 of the copy bandwidth.
// One launch for all of them waits once for the step before; with the wall rows in a
// launch of their own beside the other, closed boxes took 3.7 us a step at 32^3 (FP16
// A/B; now 2.9) and 102 at 256x192x160 (BF16; now 97).
template <typename... P, typename... A>
static void launch_step_walls(void (*kernel)(P...), bool early, WalledBox box, int threads, cudaStream_t stream,
                              A &&...args)
{
    box.inner.waits = early;
    launch_step_kernel(kernel, early, box.blocks(threads), threads, stream, 0, std::forward<A>(args)..., box);
}

// The one-cell A/B step stays one launch over all rows: its walled kernel
// already runs at the periodic kernel's speed (walled channel 512x256x256,
// FP32: 45.2 GLUPS as one launch, 44.8 split).
template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_ab1(const Planes<T> &S, const Planes<T> &D, const Geo &g, const Relax<typename Storage<T>::R> &p,
                       int threads, cudaStream_t stream)
{
    const Box box(g.nx, 0, g.ny, 0, g.nz);
    launch_step_box(k_ab1<T, RHO0, WALLS, MRT>, true, box, 0, threads, stream, S, D, g, p);
}

// FP64 in-place steps, bound by arithmetic, are not launched early: blocks that
// are placed while the launch before still holds slots end up unevenly spread
// over the SMs (32^3: 11.8 -> 19.4 us a step; the A/B step gains, 11.8 -> 10.8).
template <typename T> constexpr bool aa1_early = sizeof(T) < 8;

// The one-cell AA odd step, with the wall rows apart like the four-cell one
// (walled channel 512x256x256, FP32: odd step 0.72 of the copy bandwidth with the
// walled code on every row).
template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_aa_odd1(const Planes<T> &P, const Geo &g, const Relax<typename Storage<T>::R> &p, int threads,
                           cudaStream_t stream)
{
    if constexpr (WALLS)
        launch_step_walls(g.wall_x ? k_aa_odd1_walls<T, RHO0, MRT, true> : k_aa_odd1_walls<T, RHO0, MRT, false>, aa1_early<T>,
                          WalledBox(g.nx, g.nx, g, threads, false), threads, stream, P, g, p);
    else
        launch_step_box(k_aa_odd1<T, RHO0, MRT>, aa1_early<T>, Box(g.nx, 0, g.ny, 0, g.nz), 0, threads, stream, P, g, p);
}

constexpr int QUAD_THREADS = 128;  // threads per block of the four-cell kernels

template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_ab4(const Planes<T> &S, const Planes<T> &D, const Geo &g, const Relax<float> &p, cudaStream_t stream)
{
    if constexpr (WALLS)
        launch_step_walls(g.wall_x ? k_ab4_walls<T, RHO0, MRT, true> : k_ab4_walls<T, RHO0, MRT, false>, true,
                          WalledBox(g.nx / 4, g.nx / 4, g, QUAD_THREADS, false), QUAD_THREADS, stream, S, D, g, p);
    else
        launch_step_box(k_ab4<T, RHO0, MRT>, true, Box(g.nx / 4, 0, g.ny, 0, g.nz), 0, QUAD_THREADS, stream, S, D, g, p);
}

// The four-cell AA odd step, with the wall rows apart: four cells a thread with the
// selects of all walls spill, and ran the walled channel 512x256x256's odd step at
// 0.55 of the copy bandwidth (FP16 and BF16).  Each location is read and written by one cell's
// thread only, so the blocks may run in any order.
template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_aa_odd4(const Planes<T> &P, const Geo &g, const Relax<float> &p, cudaStream_t stream)
{
    if constexpr (WALLS) {
        const WalledBox box(g.nx / 4, g.nx, g, QUAD_THREADS, true);
        launch_step_walls(box.bx_log2 < 0 ? k_aa_odd4<T, RHO0, true, MRT> : k_aa_odd4<T, RHO0, true, MRT, ROWS_OF_BLOCKS>, false,
                          box, QUAD_THREADS, stream, P, g, p);
    } else {
        const Box box(g.nx / 4, 0, g.ny, 0, g.nz);
        // the form for grids that stay in L2 (129 MB, with the next step's share)
        // serves periodic lattices only (128^3 with walls: 33.4 us, 29.1 in blocks)
        const bool cached = g.ncell * Q * (long long)sizeof(T) < (100LL << 20);
        const int bx = cached ? 0 : box.block_x(QUAD_THREADS);
        // BF16 takes that form for every sequence (192^3: 101 against 103 us)
        constexpr OddForm seq = std::is_same_v<T, __nv_bfloat16> ? SEQUENCE_CACHED : SEQUENCE;
        auto k = cached ? k_aa_odd4<T, RHO0, false, MRT, SEQUENCE_CACHED>
                        : (bx ? k_aa_odd4<T, RHO0, false, MRT, ROWS_OF_BLOCKS> : k_aa_odd4<T, RHO0, false, MRT, seq>);
        launch_step_box(k, false, box, bx, QUAD_THREADS, stream, P, g, p);
    }
}

// One-cell step of either pattern.
template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_step1(int kind, void *src, const Planes<T> &D, const Geo &g,
                         const Relax<typename Storage<T>::R> &p, int threads, cudaStream_t stream)
{
    if (kind == 0)
        launch_ab1<T, RHO0, WALLS, MRT>(planes_of<T>(src, g.ncell), D, g, p, threads, stream);
    else if (kind == 1)
        launch_step_kernel(k_aa_even1<T, RHO0, MRT>, aa1_early<T>, blocks_for(g.ncell, threads), threads, stream, 0, D, D, g, p,
                           Box());
    else
        launch_aa_odd1<T, RHO0, WALLS, MRT>(D, g, p, threads, stream);
}

// Four-cell step of either pattern (16-bit storage, nx a multiple of 4).
template <typename T, bool RHO0, bool WALLS, bool MRT>
static void launch_step4(int kind, void *src, const Planes<T> &D, const Geo &g, const Relax<float> &p,
                         cudaStream_t stream)
{
    if (kind == 0)
        launch_ab4<T, RHO0, WALLS, MRT>(planes_of<T>(src, g.ncell), D, g, p, stream);
    else if (kind == 1)
        launch_step_kernel(k_aa_even4<T, RHO0, MRT>, true, blocks_for(g.ncell / 4, QUAD_THREADS), QUAD_THREADS, stream, 0,
                           D, D, g, p, Box());
    else
        launch_aa_odd4<T, RHO0, WALLS, MRT>(D, g, p, stream);
}

template <typename T, bool RHO0, bool WALLS>
static cudaError_t step_t(int kind, void *src, void *dst, const Geo &g, const CollBoth &cb, LaunchShape ls,
                          cudaStream_t stream)
{
    using R = typename Storage<T>::R;
    const Relax<R> p = to_relax<R>(cb);
    const Planes<T> D = planes_of<T>(dst, g.ncell);
    const int threads = ls.threads;
    if constexpr (sizeof(T) == 2) {
        if (ls.cells_x == 4 && g.nx % 4 == 0) {
            if (cb.mrt)
                launch_step4<T, RHO0, WALLS, true>(kind, src, D, g, p, stream);
            else
                launch_step4<T, RHO0, WALLS, false>(kind, src, D, g, p, stream);
            return cudaGetLastError();
        }
    }
    if (!cb.mrt && ls.cells_x >= 2 && (g.nx % 2) == 0 && (ls.bx % 32) == 0) {
        const Box box(g.nx / 2, 0, g.ny, 0, g.nz);
        if (kind == 0) {
            if constexpr (sizeof(T) == 2)
                launch_step_box(k_ab2w<T, RHO0, WALLS>, true, box, 0, QUAD_THREADS, stream, planes_of<T>(src, g.ncell), D,
                                g, p);
            else
                launch_step_box(k_ab2<T, RHO0, WALLS>, true, box, 0, threads, stream, planes_of<T>(src, g.ncell), D, g, p);
        }
        else if (kind == 1)
            launch_step_box(k_aa_even2<T, RHO0>, true, box, 0, threads, stream, D, g, p);
        else {
            if constexpr (WALLS)
                launch_step_walls(g.wall_x ? k_aa_odd2_walls<T, RHO0, true> : k_aa_odd2_walls<T, RHO0, false>, true,
                                  WalledBox(g.nx / 2, g.nx / 2, g, threads, false), threads, stream, D, g, p);
            else
                launch_step_box(k_aa_odd2<T, RHO0>, true, box, 0, threads, stream, D, g, p);
        }
        return cudaGetLastError();
    }
    if (cb.mrt)
        launch_step1<T, RHO0, WALLS, true>(kind, src, D, g, p, threads, stream);
    else
        launch_step1<T, RHO0, WALLS, false>(kind, src, D, g, p, threads, stream);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t step_any(int kind, void *src, void *dst, const Geo &g, const CollBoth &cb, LaunchShape s,
                            cudaStream_t stream)
{
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
    if (cb.rho0_is_rho)
        return walls ? step_t<T, true, true>(kind, src, dst, g, cb, s, stream)
                     : step_t<T, true, false>(kind, src, dst, g, cb, s, stream);
    return walls ? step_t<T, false, true>(kind, src, dst, g, cb, s, stream)
                 : step_t<T, false, false>(kind, src, dst, g, cb, s, stream);
}

}  // namespace lbm
