// Kernels around the time step: initialisation f = feq(rho, u), macroscopic
// moments (Eq. 16, Eq. 17), canonical copies of the state, and the FP64
// global reductions (mass, kinetic energy, momentum, max |u|, non-finite count).

#include "lbm_device.cuh"
#include "lbm_launch.h"
#include "lbm_step.cuh"  // Planes, Site, gather1

namespace lbm {

constexpr int CELL_THREADS = 256;
static Box cell_box(const Geo &g) { return Box(g.nx, 0, g.ny, 0, g.nz); }
static unsigned cell_blocks(const Geo &g) { return (unsigned)((g.ncell + CELL_THREADS - 1) / CELL_THREADS); }

#define LBM_CELL_PROLOGUE                                          \
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;      \
    if (i >= box.count) return;                                    \
    int x, y, z;                                                   \
    box.at(i, x, y, z);                                            \
    Cell c(x, y, z, g);                                            \
    const long long cell = i;

// The populations f_q - w_q of one cell in layout L, with the step kernels'
// addressing (plane pointers from the parameters, 32-bit offsets, no wall logic
// on periodic lattices).
template <int L, bool WALLS, typename T, typename R>
__device__ __forceinline__ void gather_state(const Planes<T> &P, const Site<WALLS> &s, R f[Q])
{
    if constexpr (L == AA_EVEN) {
#pragma unroll
        for (int q = 0; q < Q; ++q) f[q] = Storage<T>::load(P.p[q] + s.own + s.x);
    } else {
        gather1<L == AA_ODD>(P, s, f);
    }
}

// Calls f(layout, walls) with both as compile-time constants (an AA even state
// needs no neighbours, so no walls either).
template <typename F>
static cudaError_t by_layout(int layout, const Geo &g, F &&f)
{
    using LAB = std::integral_constant<int, AB>;
    using LEven = std::integral_constant<int, AA_EVEN>;
    using LOdd = std::integral_constant<int, AA_ODD>;
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
    if (layout == AA_EVEN) f(LEven{}, std::false_type{});
    else if (layout == AB && walls) f(LAB{}, std::true_type{});
    else if (layout == AB) f(LAB{}, std::false_type{});
    else if (walls) f(LOdd{}, std::true_type{});
    else f(LOdd{}, std::false_type{});
    return cudaGetLastError();
}

// ---------------------------------------------------------------- init

template <typename T, typename In, int D>
__global__ void k_init(T *grid, const In *rho, const In *u, Geo g, Coll<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    LBM_CELL_PROLOGUE
    R r = rho ? R(rho[cell]) : R(1);
    R uv[3] = {R(u[cell]), R(u[g.ncell + cell]), R(u[2 * g.ncell + cell])};
    R f[Q];
    equilibrium_all(r, uv, p, f);
    scatter<D>(grid, c, g.ncell, f);
}

template <typename T, typename In>
static cudaError_t init_t(int layout, void *grid, const void *rho, const void *u, const Geo &g, const CollBoth &cb,
                          cudaStream_t s)
{
    using R = typename Storage<T>::R;
    Coll<R> p = to_coll<R>(cb);
    if (layout == AB)
        k_init<T, In, D_AB_CANON><<<cell_blocks(g), CELL_THREADS, 0, s>>>((T *)grid, (const In *)rho, (const In *)u, g, p,
                                                                       cell_box(g));
    else
        k_init<T, In, D_AB_NEXT><<<cell_blocks(g), CELL_THREADS, 0, s>>>((T *)grid, (const In *)rho, (const In *)u, g, p,
                                                                        cell_box(g));  // natural order = AA even layout
    return cudaGetLastError();
}

// ---------------------------------------------------------------- moments

template <typename T, typename Out, int L, bool WALLS>
__global__ void __launch_bounds__(CELL_THREADS) k_moments(Planes<T> P, Out *rho, Out *u, Geo g,
                                                          Coll<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= box.count) return;
    int x, y, z;
    box.at(i, x, y, z);
    R f[Q];
    gather_state<L>(P, Site<WALLS>(x, y, z, 1, g), f);
    R drho, rho0, uv[3];
    macro(f, p, drho, rho0, uv);
    const long long cell = i;
    if (rho) rho[cell] = Out(R(1) + drho);
    if (u) {
        u[cell] = Out(uv[0]);
        u[g.ncell + cell] = Out(uv[1]);
        u[2 * g.ncell + cell] = Out(uv[2]);
    }
}

// ---------------------------------------------------------------- canonical copies

template <typename T, int L>
__global__ void k_get(const T *__restrict__ grid, T *__restrict__ dst, Geo g, Box box)
{
    LBM_CELL_PROLOGUE
    const int self = (int)cell;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long off;
        if (L == AA_EVEN) {
            off = (long long)q * g.ncell + self;
        } else {
            bool wall;
            int src = c.template along<-1>(q, wall);
            if (L == AB)
                off = wall ? (long long)OPP(q) * g.ncell + self : (long long)q * g.ncell + src;
            else
                off = wall ? (long long)q * g.ncell + self : (long long)OPP(q) * g.ncell + src;
        }
        dst[(long long)q * g.ncell + self] = grid[off];
    }
}

// CANON_AB = 1: write so that the AB gather returns src; 0: natural order
// (the AA even layout).
template <typename T, int CANON_AB>
__global__ void k_set(T *grid, const T *__restrict__ src, Geo g, Box box)
{
    LBM_CELL_PROLOGUE
    const int self = (int)cell;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        long long off;
        if (!CANON_AB) {
            off = (long long)q * g.ncell + self;
        } else {
            bool wall;
            int dst = c.template along<-1>(q, wall);
            off = wall ? (long long)OPP(q) * g.ncell + self : (long long)q * g.ncell + dst;
        }
        grid[off] = src[(long long)q * g.ncell + self];
    }
}

// ---------------------------------------------------------------- reductions

constexpr int RED_THREADS = 256;
// All resident at once.  Three blocks per SM, whose 85 registers a thread the sums need:
// lbm_reduce of 192^3 FP16 (whole call) 151 us, four blocks 160 (spills), five 169.
constexpr int RED_SMS = 152, RED_PER_SM = 3, RED_BLOCKS = RED_SMS * RED_PER_SM;
int reduce_blocks() { return RED_BLOCKS; }

// A running sum.  This GPU adds about 64 FP32 numbers in the time of one FP64
// number, so cells of FP32 arithmetic are summed exactly in FP32: as an unevaluated
// sum hi + lo + rest, whose two leading parts take every rounding error (TwoSum;
// exact products by fma) and whose last one, of the order of 2^-48 of the sum, is
// rounded.  That keeps about 70 bits of a few cells, whose sum is then added to an
// FP64 total: fewer FP64 roundings than adding every cell to it.  (hi + lo alone, 48
// bits, fell short of FP64 sums.)
template <typename R> struct Sum;
template <> struct Sum<float> {
    float hi = 0.f, lo = 0.f, rest = 0.f;
    __device__ __forceinline__ void add_low(float v) { two_sum_acc(lo, rest, v); }
    __device__ __forceinline__ void add(float v)
    {
        float e = 0.f;
        two_sum_acc(hi, e, v);
        add_low(e);
    }
    __device__ __forceinline__ void add_product(float a, float b)
    {
        const float p = __fmul_rn(a, b);
        add(p);
        add_low(fmaf(a, b, -p));
    }
    // adds the sum less `minus` to the total
    __device__ __forceinline__ void flush(double &total, double minus = 0.0)
    {
        total += ((double)hi - minus) + ((double)lo + (double)rest);
        hi = lo = rest = 0.f;
    }
};
template <> struct Sum<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add_product(double a, double b) { v = fma(a, b, v); }
    __device__ __forceinline__ void flush(double &total, double minus = 0.0)
    {
        total += v - minus;
        v = 0.0;
    }
};
constexpr int SUM_CELLS = 64;  // cells between two flushes (with 16, lbm_reduce takes 6 % longer)

// Whether products of FP32 numbers whose largest square is about v can be split
// into value and rounding error in FP32: not where they come near its range's
// ends (nor for NaN); those few cells are summed in FP64 at once.
__device__ __forceinline__ bool fits_products(float v) { return v > 1e-20f && v < 1e30f; }
__device__ __forceinline__ bool fits_products(double v) { return isfinite(v); }
// ... and whether a group's sum of such values v stays far from overflow
__device__ __forceinline__ bool fits_sum(float v) { return fabsf(v) < 1e15f; }
__device__ __forceinline__ bool fits_sum(double v) { return isfinite(v); }
// ... and whether one product's rounding error is a normal number (or zero)
__device__ __forceinline__ bool exact_product(float a, float b)
{
    const float p = fabsf(a * b);
    return p > 1e-30f || a == 0.f || b == 0.f;
}
__device__ __forceinline__ bool exact_product(double, double) { return true; }

// A bound below v, the largest |u|^2 so far, so far off that the squares of a cell below
// it cannot be larger in exact arithmetic; where squares of R lose bits near the end of its
// range, none.
__device__ __forceinline__ float near_square(float v) { return fits_products(v) ? v * 0.999999f : -1.f; }
__device__ __forceinline__ double near_square(double v) { return v > 1e-280 ? v * 0.999999 : -1.0; }

__device__ __forceinline__ double warp_sum_or_max(double v, bool largest)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_down_sync(0xffffffffu, v, o);
        v = largest ? fmax(v, w) : v + w;
    }
    return v;
}

// Mass, energy, momentum, max |u| and non-finite cells: one partial row per
// block of a fixed grid, in a fixed order (deterministic for a lattice size).
// The kernel was bound by FP64 work, about 45 operations a cell (a square root
// among them) and a 64-bit division; with the sums above, the root taken of the
// thread's largest |u|^2 only and the row found by a multiplication a call takes 151
// instead of 397 us at 192^3 FP16, whose bytes take 40 at the copy bandwidth.
template <typename T, int L, bool WALLS>
__global__ void __launch_bounds__(RED_THREADS, RED_PER_SM)
    k_reduce(Planes<T> P, double *partial, Geo g, Coll<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    __shared__ double sh[7][RED_THREADS];
    double acc[5] = {0, 0, 0, 0, 0}, uumax = 0.0;  // drho, |u|^2, rho0 u; largest |u|^2
    Sum<R> sum[5];
    R near_max = R(-1);  // |u|^2 below this cannot be the largest
    int bad = 0, n = 0, summed = 0;  // summed: cells in sum[] since the last flush
    auto flush = [&] {
        sum[0].flush(acc[0]);
        sum[1].flush(acc[1]);
#pragma unroll
        for (int i = 0; i < 3; ++i) sum[2 + i].flush(acc[2 + i], summed * (double)p.half_a[i]);  // rho0 u = j + a/2
        summed = 0;
    };
    for (long long cell = (long long)blockIdx.x * blockDim.x + threadIdx.x; cell < g.ncell;
         cell += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        box.at((unsigned)cell, x, y, z);
        R f[Q];
        gather_state<L>(P, Site<WALLS>(x, y, z, 1, g), f);
        R drho, rho0, u[3];
        macro(f, p, drho, rho0, u);
        bool finite = isfinite(drho);  // a sum with an infinity or a NaN in it is not finite
        if (!finite) {
            finite = true;
#pragma unroll
            for (int q = 0; q < Q; ++q) finite &= isfinite(f[q]);
        }
        const R uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        bad += !finite;
        bool fits = finite && fits_products(uu) && fits_sum(drho);
        if (p.rho0_is_rho) {
#pragma unroll
            for (int i = 0; i < 3; ++i) fits &= exact_product(rho0, u[i]);
        }
        if (fits) {
            ++summed;
            sum[0].add(drho);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                sum[1].add_product(u[i], u[i]);
                if (p.rho0_is_rho)
                    sum[2 + i].add_product(rho0, u[i]);
                else
                    sum[2 + i].add(u[i]);
            }
        } else {
            acc[0] += (double)drho;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                acc[1] += (double)u[i] * (double)u[i];
                acc[2 + i] += (double)rho0 * (double)u[i] - (double)p.half_a[i];
            }
        }
        if (!(uu < near_max)) {
            const double v[3] = {(double)u[0], (double)u[1], (double)u[2]};
            uumax = fmax(uumax, v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
            near_max = near_square(R(uumax));
        }
        if (++n % SUM_CELLS == 0) flush();
    }
    flush();
    acc[1] *= 0.5;
    // one warp per result sums the block's threads (a shuffle tree of every warp
    // for every result would cost four times the FP64 additions)
    const double slot[7] = {acc[0], acc[1], acc[2], acc[3], acc[4], sqrt(uumax), (double)bad};
#pragma unroll
    for (int k = 0; k < 7; ++k) sh[k][threadIdx.x] = slot[k];
    __syncthreads();
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k < 7) {
        double v = sh[k][lane];
#pragma unroll
        for (int i = 32; i < RED_THREADS; i += 32) v = (k == 5) ? fmax(v, sh[k][lane + i]) : v + sh[k][lane + i];
        v = warp_sum_or_max(v, k == 5);
        if (lane == 0) partial[blockIdx.x * 8 + k] = v;
    }
}

// One warp per result, so that all rows' loads are in flight together.
__global__ void __launch_bounds__(RED_THREADS) k_reduce_final(const double *partial, int nblocks, double *result,
                                                              double ncell)
{
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = 0.0;
    if (k < 7) {
        constexpr int U = 20;  // loads in flight
        for (int b = lane; b < nblocks; b += 32 * U) {
            double row[U];
#pragma unroll
            for (int i = 0; i < U; ++i) row[i] = b + 32 * i < nblocks ? partial[(b + 32 * i) * 8 + k] : 0.0;
#pragma unroll
            for (int i = 0; i < U; ++i) v = (k == 5) ? fmax(v, row[i]) : v + row[i];
        }
        v = warp_sum_or_max(v, k == 5);
    }
    if (lane == 0) result[k] = (k == 0) ? ncell + v : v;  // slot 7 is 0
}

// Enstrophy 1/2 <|curl u|^2> of the state, with second-order central
// differences of u (Eq. 17) between the axis neighbours.  Periodic axes wrap;
// across a half-way bounce-back wall the ghost velocity is -u of the own cell
// (the wall at rest halfway between them).  A block owns a tile of
// columns (EnsTiles) with a halo of one and marches along z: every thread forms the
// velocity of its column's cell once per plane, keeps those of three planes in
// registers and shares the middle one through shared memory.  (Gathering all
// six neighbours' populations instead took 133 loads a cell and FP64
// differences: 192^3 FP16 1.2 ms.)  Differences of FP32 velocities are taken
// and squared to about 70 bits (Sum): a call at 192^3 takes 238 us (657 before the tiles;
// 190 with 48-bit terms, which fall short of FP64); FP64 storage uses FP64.  Deterministic: fixed grid,
// fixed tiles, fixed per-thread order, fixed trees.
constexpr int ENS_THREADS = 512, ENS_PER_SM = 2;  // resident blocks
// Tile shape: 2^lanes_log2 columns along x (the halo included) and as many rows as a
// block has threads for them: 32 columns, or another power of two where fewer tiles
// cover the lattice (a call on 8x302x356 with 32 and now: FP32 87 and 71 us, FP64 640
// and 319; six gathers a cell took 95 and 580).
struct EnsTiles {
    int lanes_log2, planes;  // planes of a tile
    int x, y;                // columns and rows a tile owns
};

static EnsTiles enstrophy_tiles(const Geo &g)
{
    EnsTiles t{};
    long long columns = -1;
    for (const int l : {5, 4, 6, 3, 7, 2}) {
        const int x = (1 << l) - 2, y = (ENS_THREADS >> l) - 2;
        const long long c = (long long)((g.nx - 1) / x + 1) * ((g.ny - 1) / y + 1);
        if (columns < 0 || c < columns) {
            columns = c;
            t.lanes_log2 = l;
            t.x = x;
            t.y = y;
        }
    }
    // planes per tile: the resident blocks take the tiles in turns, and each tile costs
    // two more planes than it has
    long long best = -1;
    t.planes = g.nz;
    for (int len = 1; len <= g.nz; len += 1 + len / 16) {
        const long long tiles = columns * ((g.nz + len - 1) / len);
        const long long cost = (tiles + RED_SMS * ENS_PER_SM - 1) / (RED_SMS * ENS_PER_SM) * (len + 2);
        if (best < 0 || cost < best) {
            best = cost;
            t.planes = len;
        }
    }
    return t;
}

// a - b, exact as a double-float
__device__ __forceinline__ DF exact_diff(float a, float b)
{
    DF r{a, 0.f};
    two_sum_acc(r.hi, r.lo, -b);
    return r;
}
// (a1 - a0) - (b1 - b0), twice a component of the curl, squared and added to s or total
__device__ __forceinline__ void add_square_of_curl(Sum<float> &s, double &total, float a1, float a0, float b1, float b0)
{
    const DF a = exact_diff(a1, a0), b = exact_diff(b0, b1);
    // w = hi + lo + rest, the leading parts exact
    float hi = a.hi, e = 0.f, lo = a.lo, rest = 0.f;
    two_sum_acc(hi, e, b.hi);
    two_sum_acc(lo, rest, b.lo);
    two_sum_acc(lo, rest, e);
    // (hi is a multiple of half the last bit of a.hi or b.hi, and so of lo's last bit:
    // then hi + lo without TwoSum's second half is exact also where |lo| > |hi|)
    const float w = hi + lo;
    lo -= w - hi;
    if (fits_products(w * w)) {
        // w^2 + 2 w lo + (2 w rest + lo^2), by size of the parts
        const float twice = 2.f * w, p = __fmul_rn(twice, lo);
        s.add_product(w, w);
        s.add_low(p);
        s.rest += fmaf(twice, rest, fmaf(lo, lo, fmaf(twice, lo, -p)));
    } else if (w != 0.f) {
        const double v = ((double)a1 - (double)a0) - ((double)b1 - (double)b0);
        total += v * v;
    }
}
__device__ __forceinline__ void add_square_of_curl(Sum<double> &s, double &, double a1, double a0, double b1, double b0)
{
    const double w = (a1 - a0) - (b1 - b0);
    s.add_product(w, w);
}

template <typename T, int L, bool WALLS>
__global__ void __launch_bounds__(ENS_THREADS, ENS_PER_SM)
    k_enstrophy(Planes<T> P, double *partial, Geo g, Coll<typename Storage<T>::R> p, EnsTiles tile)
{
    using R = typename Storage<T>::R;
    __shared__ R su[2][3][ENS_THREADS];
    __shared__ double sh[32];
    const int lanes = 1 << tile.lanes_log2;
    const int tid = threadIdx.x, lane = tid & (lanes - 1), row = tid >> tile.lanes_log2;
    const int ntx = (g.nx - 1) / tile.x + 1, nty = (g.ny - 1) / tile.y + 1;
    const int ntz = (g.nz + tile.planes - 1) / tile.planes;
    const long long tiles = (long long)ntx * nty * ntz;
    double acc = 0.0;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int tx = (int)(t % ntx), ty = (int)(t / ntx % nty), tz = (int)(t / ntx / nty);
        // one more than the thread's column and row (an edge, and the halo past it, may pass 2^31 - 1)
        const unsigned xr = (unsigned)tx * tile.x + lane, yr = (unsigned)ty * tile.y + row;
        const int z0 = tz * tile.planes, z1 = min(z0 + tile.planes, g.nz);
        // this thread's column, wrapped; beyond the halo it repeats some column of the lattice
        const int x = (int)(((xr == 0 ? (unsigned)g.nx : xr) - 1u) % (unsigned)g.nx);
        const int y = (int)(((yr == 0 ? (unsigned)g.ny : yr) - 1u) % (unsigned)g.ny);
        const bool own = lane >= 1 && lane <= tile.x && row >= 1 && row <= tile.y && xr <= (unsigned)g.nx &&
                         yr <= (unsigned)g.ny;
        auto velocity = [&](int z, R u[3]) {
            R f[Q];
            gather_state<L>(P, Site<WALLS>(x, y, z < 0 ? z + g.nz : (z >= g.nz ? z - g.nz : z), 1, g), f);
            R drho, rho0;
            macro(f, p, drho, rho0, u);
        };
        R um[3], uc[3], up[3];
        velocity(z0 - 1, um);
        velocity(z0, uc);
        Sum<R> s;
        for (int z = z0; z < z1; ++z) {
            const int b = z & 1;  // the other buffer may still be read for the plane before
#pragma unroll
            for (int i = 0; i < 3; ++i) su[b][i][tid] = uc[i];
            velocity(z + 1, up);
            __syncthreads();
            if (own) {
                // neighbours' velocities; a walled axis' ghost is -u of the own cell
                auto nb = [&](int i, int at, bool wall) { return wall ? -uc[i] : su[b][i][at]; };
                const bool wxm = g.wall_x && x == 0, wxp = g.wall_x && x == g.nx - 1;
                const bool wym = g.wall_y && y == 0, wyp = g.wall_y && y == g.ny - 1;
                const bool wzm = g.wall_z && z == 0, wzp = g.wall_z && z == g.nz - 1;
                const R zm0 = wzm ? -uc[0] : um[0], zm1 = wzm ? -uc[1] : um[1];
                const R zp0 = wzp ? -uc[0] : up[0], zp1 = wzp ? -uc[1] : up[1];
                // 2 (d_y u_z - d_z u_y), 2 (d_z u_x - d_x u_z), 2 (d_x u_y - d_y u_x)
                add_square_of_curl(s, acc, nb(2, tid + lanes, wyp), nb(2, tid - lanes, wym), zp1, zm1);
                add_square_of_curl(s, acc, zp0, zm0, nb(2, tid + 1, wxp), nb(2, tid - 1, wxm));
                add_square_of_curl(s, acc, nb(1, tid + 1, wxp), nb(1, tid - 1, wxm), nb(0, tid + lanes, wyp),
                                   nb(0, tid - lanes, wym));
            }
            if ((z - z0) % SUM_CELLS == SUM_CELLS - 1) s.flush(acc);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                um[i] = uc[i];
                uc[i] = up[i];
            }
        }
        s.flush(acc);
        __syncthreads();
    }
    const double v = block_sum(acc, sh);
    if (tid == 0) partial[blockIdx.x * 8] = v;
}

__global__ void __launch_bounds__(RED_THREADS) k_enstrophy_final(const double *partial, int nblocks,
                                                                 double *result, double ncell)
{
    __shared__ double sh[32];
    double v = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v += partial[b * 8];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) result[0] = 0.125 * v / ncell;  // (twice the curl)^2, and 1/2
}

// ---------------------------------------------------------------- dispatch

template <typename F>
static cudaError_t by_prec(int prec, F &&f)
{
    switch (prec) {
    case P_F64: return f(double());
    case P_F32: return f(float());
    case P_F16: return f(__half());
    case P_BF16: return f(__nv_bfloat16());
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_init(int prec, int layout, void *grid, const void *rho, const void *u, int dtype, const Geo &g,
                        const CollBoth &c, cudaStream_t s)
{
    return by_prec(prec, [&](auto t) {
        using T = decltype(t);
        return dtype == 0 ? init_t<T, double>(layout, grid, rho, u, g, c, s)
                          : init_t<T, float>(layout, grid, rho, u, g, c, s);
    });
}

cudaError_t launch_moments(int prec, int layout, const void *grid, void *rho, void *u, int dtype, const Geo &g,
                           const CollBoth &cb, cudaStream_t s)
{
    return by_prec(prec, [&](auto t) {
        using T = decltype(t);
        const auto p = to_coll<typename Storage<T>::R>(cb);
        const Planes<T> P = planes_of<T>(const_cast<void *>(grid), g.ncell);
        const Box box = cell_box(g);
        return by_layout(layout, g, [&](auto l, auto w) {
            constexpr int L = decltype(l)::value;
            constexpr bool W = decltype(w)::value;
            if (dtype == 0)
                k_moments<T, double, L, W><<<cell_blocks(g), CELL_THREADS, 0, s>>>(P, (double *)rho, (double *)u, g, p, box);
            else
                k_moments<T, float, L, W><<<cell_blocks(g), CELL_THREADS, 0, s>>>(P, (float *)rho, (float *)u, g, p, box);
        });
    });
}

cudaError_t launch_get_pdfs(int prec, int layout, const void *grid, void *dst, const Geo &g, cudaStream_t s)
{
    return by_prec(prec, [&](auto t) {
        using T = decltype(t);
        const T *gr = (const T *)grid;
        T *d = (T *)dst;
        if (layout == AB) k_get<T, AB><<<cell_blocks(g), CELL_THREADS, 0, s>>>(gr, d, g, cell_box(g));
        else if (layout == AA_EVEN) k_get<T, AA_EVEN><<<cell_blocks(g), CELL_THREADS, 0, s>>>(gr, d, g, cell_box(g));
        else k_get<T, AA_ODD><<<cell_blocks(g), CELL_THREADS, 0, s>>>(gr, d, g, cell_box(g));
        return cudaGetLastError();
    });
}

cudaError_t launch_set_pdfs(int prec, int layout, void *grid, const void *src, const Geo &g, cudaStream_t s)
{
    return by_prec(prec, [&](auto t) {
        using T = decltype(t);
        T *gr = (T *)grid;
        const T *sr = (const T *)src;
        if (layout == AB) k_set<T, 1><<<cell_blocks(g), CELL_THREADS, 0, s>>>(gr, sr, g, cell_box(g));
        else k_set<T, 0><<<cell_blocks(g), CELL_THREADS, 0, s>>>(gr, sr, g, cell_box(g));
        return cudaGetLastError();
    });
}

cudaError_t launch_reduce(int prec, int layout, const void *grid, double *scratch, double *result, const Geo &g,
                          const CollBoth &cb, cudaStream_t s)
{
    cudaError_t e = by_prec(prec, [&](auto t) {
        using T = decltype(t);
        const auto p = to_coll<typename Storage<T>::R>(cb);
        const Planes<T> P = planes_of<T>(const_cast<void *>(grid), g.ncell);
        const Box box = cell_box(g);
        return by_layout(layout, g, [&](auto l, auto w) {
            k_reduce<T, decltype(l)::value, decltype(w)::value><<<RED_BLOCKS, RED_THREADS, 0, s>>>(P, scratch, g, p, box);
        });
    });
    if (e != cudaSuccess) return e;
    k_reduce_final<<<1, RED_THREADS, 0, s>>>(scratch, RED_BLOCKS, result, (double)g.ncell);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- reduction without caller scratch
//
// lbm_reduce_noalloc serves callers that cannot allocate device memory (for
// example code running inside an allocator-less host, or a caller whose
// memory budget is fixed up front): its FP64 block partials and results live
// in this file-scope array instead of the scratch buffer lent to lbm_bind.
// Every GPU that loads the library holds the array until the process exits.
// In host code `g_reduce_scratch` only names a host-side stand-in; the device
// address is looked up with cudaGetSymbolAddress on every call, with the
// calling thread's current device, which must be the device of the bound
// stream (checked).  Looking it up each time keeps it right after the
// primary context has been destroyed and created again (cudaDeviceReset); the
// first lookup on a device may load the library's module, so the first call
// on a device should come before any stream capture.  All calls share the
// array and each call overwrites all of it that it reads (every block writes
// its partial row, the final kernel writes the results), so nothing needs
// clearing between calls; calls that overlap on the GPU (several streams or
// handles at once) race on it.
constexpr int NOALLOC_MAX_BLOCKS = 1024;                 // partial rows the array holds
constexpr int NOALLOC_DOUBLES = NOALLOC_MAX_BLOCKS * 8 + 8;  // 64 KiB + results
static __device__ __align__(256) double g_reduce_scratch[NOALLOC_DOUBLES];

int reduce_noalloc_capacity_doubles() { return NOALLOC_DOUBLES; }

cudaError_t launch_enstrophy(int prec, int layout, const void *grid, double *scratch, double *result, const Geo &g,
                             const CollBoth &c, cudaStream_t s)
{
    constexpr int blocks = RED_SMS * ENS_PER_SM;
    cudaError_t e = by_prec(prec, [&](auto tag) {
        using T = decltype(tag);
        const auto p = to_coll<typename Storage<T>::R>(c);
        const Planes<T> P = planes_of<T>(const_cast<void *>(grid), g.ncell);
        const EnsTiles tiles = enstrophy_tiles(g);
        return by_layout(layout, g, [&](auto l, auto w) {
            k_enstrophy<T, decltype(l)::value, decltype(w)::value><<<blocks, ENS_THREADS, 0, s>>>(P, scratch, g, p, tiles);
        });
    });
    if (e != cudaSuccess) return e;
    k_enstrophy_final<<<1, RED_THREADS, 0, s>>>(scratch, blocks, result, (double)g.ncell);
    return cudaGetLastError();
}

cudaError_t launch_reduce_noalloc(int prec, int layout, const void *grid, const Geo &g, const CollBoth &c,
                                  cudaStream_t s, double **result)
{
    if ((long long)RED_BLOCKS * 8 + 8 > NOALLOC_DOUBLES) return cudaErrorInvalidValue;
    int dev = -1, sdev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaStreamGetDevice(s, &sdev);
    if (e != cudaSuccess) return e;
    if (sdev != dev) return cudaErrorInvalidDevice;
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_reduce_scratch);
    if (e != cudaSuccess) return e;
    double *base = static_cast<double *>(p);
    *result = base + (size_t)RED_BLOCKS * 8;
    return launch_reduce(prec, layout, grid, base, *result, g, c, s);
}

}  // namespace lbm
