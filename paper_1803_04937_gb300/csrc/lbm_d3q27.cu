// D3Q27 stream + collide (Sec. 2.3 lattice; on D3Q27 the moment-matching
// construction of Sec. 3.1 gives the standard equilibrium of Eq. 14, so both
// equilibrium choices run Eq. 14), for the paper's D3Q19 / D3Q27 comparison:
// the same A/B pull scheme, force, TRT, boundaries and storage precisions as
// the D3Q19 path, with 27 loads + 27 stores per cell.  One cell per thread,
// or four for 16-bit storage.
//
// Also: initialisation f = feq(rho, u), moments and canonical copies for
// D3Q27 lattices.  (Reductions, AA and the adjoint are D3Q19 only.)
#include <cmath>

#include "lbm_pair.cuh"
#include "lbm_step.cuh"

namespace lbm {
namespace q27 {

constexpr int Q27 = 27;

// This library's D3Q27 order: rest, then 13 pairs (q, q + 1) with
// c_{q+1} = -c_q: 3 faces, 6 edges, 4 corners.
__host__ __device__ constexpr int CX(int q)
{
    constexpr int t[Q27] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1};
    return t[q];
}
__host__ __device__ constexpr int CY(int q)
{
    constexpr int t[Q27] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, -1, 1, -1, 1};
    return t[q];
}
__host__ __device__ constexpr int CZ(int q)
{
    constexpr int t[Q27] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[q];
}
__host__ __device__ constexpr int OPP(int q) { return q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1); }
__host__ __device__ constexpr int NORM2(int q) { return CX(q) * CX(q) + CY(q) * CY(q) + CZ(q) * CZ(q); }
__host__ __device__ constexpr double WQ(int q)
{
    return NORM2(q) == 0 ? 8.0 / 27.0 : (NORM2(q) == 1 ? 2.0 / 27.0 : (NORM2(q) == 2 ? 1.0 / 54.0 : 1.0 / 216.0));
}

// Per-launch constants.  The antisymmetric equilibrium of a pair is
// (A_k / 2) c.u with A = 6 w; per axis the first moment is A_face + 4 A_edge +
// 4 A_corner = 1, and the constants are chosen so that this holds exactly in
// the working precision (no systematic momentum drift).
template <typename R>
struct Relax27 {
    R hp, hm, wp;
    R w[4];    // rest, face, edge, corner
    R K[4];    // 9/2 w
    R A[4];    // 6 w (A[0] unused)
    R half_a[3];
    R force[13];
};

template <typename R>
static inline Relax27<R> to_relax27(const CollBoth &c)
{
    Relax27<R> r;
    r.hp = R(0.5 * c.omega_p);
    r.hm = R(0.5 * c.omega_m);
    r.wp = R(c.omega_p);
    const double w[4] = {8.0 / 27.0, 2.0 / 27.0, 1.0 / 54.0, 1.0 / 216.0};
    for (int i = 0; i < 4; ++i) {
        r.w[i] = R(w[i]);
        r.K[i] = R(4.5 * w[i]);
    }
    // A_edge = R(1/9); A_corner rounded to a multiple of ulp(A_edge) / 4 so
    // that 1 - 4 A_edge - 4 A_corner is exactly representable in R.
    // (In FP32: ulp(1/9) = 2^-27, and 1 - 4 A_edge - 4 A_corner is a multiple
    // of 2^-25 in [1/4, 1/2), exact in FP32 and computed exactly in double.
    // In FP64 the residual is at the 1e-16 level.)
    double ae = 1.0 / 9.0, ac = 1.0 / 36.0;
    if (sizeof(R) == 4) {
        ae = (double)(float)(1.0 / 9.0);
        ac = std::round((1.0 / 36.0) * 134217728.0) / 134217728.0;  // multiple of 2^-27
    }
    r.A[0] = R(0);
    r.A[2] = R(ae);
    r.A[3] = R(ac);
    r.A[1] = R(1.0 - 4.0 * ae - 4.0 * ac);
    for (int i = 0; i < 3; ++i) r.half_a[i] = R(c.half_a[i]);
    const double wm = c.omega_m;
    for (int k = 0; k < 13; ++k) {
        const int q = 2 * k + 1;
        const double ca = CX(q) * 2.0 * c.half_a[0] + CY(q) * 2.0 * c.half_a[1] + CZ(q) * 2.0 * c.half_a[2];
        r.force[k] = R((1.0 - 0.5 * wm) * 3.0 * WQ(q) * ca);
    }
    return r;
}

// ONE_ROUNDING adds each population's change to g in one rounding, as the
// D3Q19 collision (relax_pair) does for FP32 and FP64 storage.
template <typename R, bool RHO0, bool ONE_ROUNDING>
__device__ __forceinline__ void collide27(R g[Q27], const Relax27<R> &p)
{
    R s[13], d[13];
#pragma unroll
    for (int k = 0; k < 13; ++k) {
        s[k] = g[2 * k + 1] + g[2 * k + 2];
        d[k] = g[2 * k + 1] - g[2 * k + 2];
    }
    R drho = g[0];
#pragma unroll
    for (int k = 0; k < 13; ++k) drho += s[k];
    R P = R(1), u[3], du[3] = {R(0), R(0), R(0)};
    constexpr bool COMP = compensated_v<R, ONE_ROUNDING> && !RHO0;
    // momentum; pair k < 3 is the face pair of axis k (c = +e_k) and starts the sum
    R j[3] = {d[0], d[1], d[2]};
    if (COMP) {
        // compensated momentum, as CellEq does for D3Q19 (FP32 storage): u is
        // rounded, du = (j + a/2) - u exactly, and the face pair of each axis
        // takes du out of its antisymmetric non-equilibrium, so the momentum
        // balance stays exact
        R lo[3] = {R(0), R(0), R(0)};
#pragma unroll
        for (int k = 3; k < 13; ++k) {
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
        for (int k = 3; k < 13; ++k) {
            const int q = 2 * k + 1;
            if (CX(q)) j[0] = CX(q) > 0 ? j[0] + d[k] : j[0] - d[k];
            if (CY(q)) j[1] = CY(q) > 0 ? j[1] + d[k] : j[1] - d[k];
            if (CZ(q)) j[2] = CZ(q) > 0 ? j[2] + d[k] : j[2] - d[k];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) u[i] = j[i] + p.half_a[i];
        if (RHO0) {
            P = R(1) + drho;
            const R inv = R(1) / P;
#pragma unroll
            for (int i = 0; i < 3; ++i) u[i] = mul(u[i], inv);
        }
    }
    const R uu = mad(u[2], u[2], mad(u[1], u[1], mul(u[0], u[0])));
    const R base = mad(RHO0 ? mul(R(-1.5f), P) : R(-1.5f), uu, drho);
    g[0] = mad(-p.wp, mad(-p.w[0], base, g[0]), g[0]);
    R K[4], A[4], wb[4];
#pragma unroll
    for (int c = 1; c < 4; ++c) {
        K[c] = RHO0 ? mul(P, p.K[c]) : p.K[c];
        A[c] = RHO0 ? mul(P, p.A[c]) : p.A[c];
        wb[c] = mul(p.w[c], base);
    }
#pragma unroll
    for (int k = 0; k < 13; ++k) {
        const int q = 2 * k + 1;
        const int cls = NORM2(q);
        const R cu = along(CX(q), CY(q), CZ(q), u);
        const R sym = mad(K[cls], mul(cu, cu), wb[cls]);
        const R nsym = mad(R(-2), sym, s[k]);
        R nasym = mad(-A[cls], cu, d[k]);
        if (COMP && k < 3) nasym -= du[k];
        const R b = mad(p.hm, nasym, -p.force[k]);
        if (ONE_ROUNDING) {
            g[q] = g[q] - mad(p.hp, nsym, b);
            g[q + 1] = g[q + 1] - mad(p.hp, nsym, -b);
        } else {
            g[q] = mad(-p.hp, nsym, g[q]) - b;
            g[q + 1] = mad(-p.hp, nsym, g[q + 1]) + b;
        }
    }
}

// A/B pull step, one cell per thread.  FLAT: the cells as one sequence, or in
// blocks that are rectangles of rows, which is faster with walls where rows are
// multiples of 128 cells (256^3 FP32: 549 -> 536 us) and slower elsewhere (513x100x100:
// 170 -> 205).  Four blocks per SM, also with rho0 = rho (left alone, 73 registers and
// three blocks: 259x307x95 with walls 325 us, 260 now).
template <typename T, bool RHO0, bool WALLS, bool FLAT = true>
__global__ void __launch_bounds__(256, sizeof(typename Storage<T>::R) == 4 ? 4 : 1) k27_ab1(const T *src, T *dst, Geo g,
                                               Relax27<typename Storage<T>::R> p, Box box)
{
    using R = typename Storage<T>::R;
    int x, y, z;
    if constexpr (FLAT) {
        const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= box.count) return;
        box.at(i, x, y, z);
    } else if (!box.at_block(x, y, z)) {
        return;
    }
    const Site<WALLS> s(x, y, z, 1, g);
    step_begin(box);
    R f[Q27];
#pragma unroll
    for (int q = 0; q < Q27; ++q) {
        const int cx = CX(q), cy = CY(q), cz = CZ(q);
        const int xs = cx == 0 ? x : (cx > 0 ? s.xm : s.xp);
        bool w = false;
        if (WALLS) {
            if (cx > 0) w |= s.bxm;
            if (cx < 0) w |= s.bxp;
            if (cy > 0) w |= s.bym;
            if (cy < 0) w |= s.byp;
            if (cz > 0) w |= s.bzm;
            if (cz < 0) w |= s.bzp;
        }
        const long long a = w ? (long long)OPP(q) * g.ncell + s.own + x
                              : (long long)q * g.ncell + s.row[1 - cy][1 - cz] + xs;
        f[q] = Storage<T>::load(src + a);
    }
    collide27<R, RHO0, one_rounding_v<T>>(f, p);
#pragma unroll
    for (int q = 0; q < Q27; ++q) Storage<T>::store(dst + (long long)q * g.ncell + s.own + x, f[q]);
}

// A/B pull step for 16-bit storage, four cells per thread (nx % 4 == 0): the
// same windowed quads as the D3Q19 four-cell step (each +-x shifted window
// formed by funnel shifts from the aligned quad and its aligned neighbour),
// 27 populations.  Bitwise the same results as k27_ab1.
template <typename T, bool RHO0, bool WALLS>
__device__ __forceinline__ void ab4_body27(const T *src, T *dst, const Site<WALLS> &s, const Geo &g,
                                           const Relax27<float> &p)
{
    const int x0 = s.x;
    const int xprev = x0 == 0 ? g.nx - 4 : x0 - 4;
    const int xnext = x0 + 4 >= g.nx ? 0 : x0 + 4;
    const unsigned short *base = reinterpret_cast<const unsigned short *>(src);
    uint2 win[Q27], nb[Q27];
#pragma unroll
    for (int q = 0; q < Q27; ++q) {
        const int cx = CX(q), cy = CY(q), cz = CZ(q);
        bool w = false;
        if (WALLS) {
            if (cy > 0) w |= s.bym;
            if (cy < 0) w |= s.byp;
            if (cz > 0) w |= s.bzm;
            if (cz < 0) w |= s.bzp;
        }
        const unsigned short *plane = base + (long long)q * g.ncell + s.row[1 - cy][1 - cz];
        const unsigned short *bnc = base + (long long)OPP(q) * g.ncell + s.own;
        const uint2 *pq = reinterpret_cast<const uint2 *>(w ? bnc + x0 : plane + x0);
        const uint2 *pn = reinterpret_cast<const uint2 *>(plane + (cx > 0 ? xprev : xnext));
        const bool xwall = WALLS && ((cx > 0 && s.bxm) || (cx < 0 && s.bxp));
        if (xwall && !w) pn = reinterpret_cast<const uint2 *>(bnc + x0);
        win[q] = __ldg(pq);  // so not launched early (launch_step_kernel)
        if (cx != 0) nb[q] = w ? make_uint2(0u, 0u) : __ldg(pn);
    }
#pragma unroll
    for (int q = 0; q < Q27; ++q) {
        const int cx = CX(q), cy = CY(q), cz = CZ(q);
        bool w = false;
        if (WALLS) {
            if (cy > 0) w |= s.bym;
            if (cy < 0) w |= s.byp;
            if (cz > 0) w |= s.bzm;
            if (cz < 0) w |= s.bzp;
        }
        if (cx == 0 || w) continue;
        const uint2 c = win[q];
        uint2 n = nb[q];
        if (cx > 0) {
            if (WALLS && s.bxm) n.y = n.x << 16;
            win[q].x = __funnelshift_l(n.y, c.x, 16);
            win[q].y = __funnelshift_l(c.x, c.y, 16);
        } else {
            if (WALLS && s.bxp) n.x = n.y >> 16;
            win[q].x = __funnelshift_r(c.x, c.y, 16);
            win[q].y = __funnelshift_r(c.y, n.x, 16);
        }
    }
#define LBM_AB27_CELL(c)                                                                     \
    {                                                                                        \
        float f[Q27];                                                                        \
        _Pragma("unroll") for (int q = 0; q < Q27; ++q) f[q] = Bits16<T>::to_float(quad_get<c>(win[q]));   \
        collide27<float, RHO0, false>(f, p);                                                 \
        _Pragma("unroll") for (int q = 0; q < Q27; ++q) quad_set<c>(win[q], Bits16<T>::from_float(f[q]));  \
    }
    LBM_AB27_CELL(0) LBM_AB27_CELL(1) LBM_AB27_CELL(2) LBM_AB27_CELL(3)
#undef LBM_AB27_CELL
    unsigned short *out = reinterpret_cast<unsigned short *>(dst);
#pragma unroll
    for (int q = 0; q < Q27; ++q)
        *reinterpret_cast<uint2 *>(out + (long long)q * g.ncell + s.own + x0) = win[q];
}

// FLAT as in k27_ab1 (256^3 FP16: 280 -> 268 us in rectangles).
template <typename T, bool RHO0, bool FLAT>
__global__ void __launch_bounds__(128, 4) k27_ab4(const T *src, T *dst, Geo g, Relax27<float> p, Box box)
{
    int xq, y, z;
    if constexpr (FLAT) {
        const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= box.count) return;
        box.at(i, xq, y, z);
    } else if (!box.at_block(xq, y, z)) {
        return;
    }
    ab4_body27<T, RHO0>(src, dst, Site<false>(4 * xq, y, z, 4, g), g, p);
}

// With walls (WalledBox), the cells as one sequence (BF16 256^3 with walls on all axes: 287
// us, 335 in rectangles; FP16 with rho0 = rho 286 against 333).  XWALLS: walls on x too.
template <typename T, bool RHO0, bool XWALLS>
__global__ void __launch_bounds__(128, 4) k27_ab4_walls(const T *src, T *dst, Geo g, Relax27<float> p, WalledBox box)
{
    int xq, y, z;
    if (box.at_walls()) {
        const unsigned i = box.wall_item();
        if (i >= box.walls.count) return;
        box.walls.at_wall(i, xq, y, z);
        ab4_body27<T, RHO0>(src, dst, Site<true>(4 * xq, y, z, 4, g), g, p);
    } else {
        const unsigned i = box.inner_item();
        if (i >= box.inner.count) return;
        box.inner.at(i, xq, y, z);
        Site<XWALLS> s(4 * xq, y, z, 4, g);
        drop_yz(s);
        ab4_body27<T, RHO0>(src, dst, s, g, p);
    }
}

// The lattice for two FP32 steps per pass (k_pair).  16 rows leave 128 registers a
// thread for the 27 populations in hand and the 27 on their way; with 20 rows they
// spill (256^3: 454 against 564 us a step, one-step kernel 520; walled channel
// 512x256x256 954 against 1567, one-step 1067).
struct Lat27 {
    static constexpr int NQ = Q27;
    using Consts = Relax27<float>;
    template <bool WALLS> static constexpr int warps = 16;
    static __host__ __device__ constexpr int cx(int q) { return CX(q); }
    static __host__ __device__ constexpr int cy(int q) { return CY(q); }
    static __host__ __device__ constexpr int cz(int q) { return CZ(q); }
    template <bool RHO0, bool WALLS, bool MRT>
    static __device__ __forceinline__ void collide(float g[Q27], const Relax27<float> &p)
    {
        collide27<float, RHO0, true>(g, p);
    }
};

// Writes the canonical populations fc (f_q(x) - w_q) of cell x into an A/B
// grid so that the pull gather returns them: plane q at x - c_q, or through a
// wall plane qbar of x.
template <typename T, bool WALLS>
__device__ __forceinline__ void put_canonical(T *grid, const Site<WALLS> &s, int x, const Geo &g,
                                              const typename Storage<T>::R fc[Q27])
{
#pragma unroll
    for (int q = 0; q < Q27; ++q) {
        const int cx = CX(q), cy = CY(q), cz = CZ(q);
        const int xs = cx == 0 ? x : (cx > 0 ? s.xm : s.xp);
        bool w = false;
        if (WALLS) {
            if (cx > 0) w |= s.bxm;
            if (cx < 0) w |= s.bxp;
            if (cy > 0) w |= s.bym;
            if (cy < 0) w |= s.byp;
            if (cz > 0) w |= s.bzm;
            if (cz < 0) w |= s.bzp;
        }
        const long long a = w ? (long long)OPP(q) * g.ncell + s.own + x
                              : (long long)q * g.ncell + s.row[1 - cy][1 - cz] + xs;
        Storage<T>::store(grid + a, fc[q]);
    }
}

template <typename T, bool WALLS>
__device__ __forceinline__ void get_canonical(const T *grid, const Site<WALLS> &s, int x, const Geo &g,
                                              typename Storage<T>::R fc[Q27])
{
#pragma unroll
    for (int q = 0; q < Q27; ++q) {
        const int cx = CX(q), cy = CY(q), cz = CZ(q);
        const int xs = cx == 0 ? x : (cx > 0 ? s.xm : s.xp);
        bool w = false;
        if (WALLS) {
            if (cx > 0) w |= s.bxm;
            if (cx < 0) w |= s.bxp;
            if (cy > 0) w |= s.bym;
            if (cy < 0) w |= s.byp;
            if (cz > 0) w |= s.bzm;
            if (cz < 0) w |= s.bzp;
        }
        const long long a = w ? (long long)OPP(q) * g.ncell + s.own + x
                              : (long long)q * g.ncell + s.row[1 - cy][1 - cz] + xs;
        fc[q] = Storage<T>::load(grid + a);
    }
}

// FLAT as in k27_ab1.
#define LBM_Q27_PROLOGUE                                             \
    int x, y, z;                                                     \
    if (FLAT) {                                                      \
        const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;    \
        if (i >= box.count) return;                                  \
        box.at(i, x, y, z);                                          \
    } else if (!box.at_block(x, y, z)) {                             \
        return;                                                      \
    }                                                                \
    const Site<true> s(x, y, z, 1, g);                               \
    const long long cell = s.own + x;

// f = feq(rho, u) (Eq. 14, shifted), written in the A/B layout.
template <typename T, typename In>
__global__ void k27_init(T *grid, const In *rho, const In *u, Geo g, Relax27<typename Storage<T>::R> p, int rho0_mode,
                         Box box)
{
    using R = typename Storage<T>::R;
    constexpr bool FLAT = true;
    LBM_Q27_PROLOGUE
    const R r = rho ? R(rho[cell]) : R(1);
    const R uv[3] = {R(u[cell]), R(u[g.ncell + cell]), R(u[2 * g.ncell + cell])};
    const R P = rho0_mode ? r : R(1);
    const R drho = r - R(1);
    const R uu = uv[0] * uv[0] + uv[1] * uv[1] + uv[2] * uv[2];
    const R base = drho - R(1.5) * P * uu;
    R fc[Q27];
    fc[0] = p.w[0] * base;
#pragma unroll
    for (int k = 0; k < 13; ++k) {
        const int q = 2 * k + 1, cls = NORM2(q);
        const R cu = R(CX(q)) * uv[0] + R(CY(q)) * uv[1] + R(CZ(q)) * uv[2];
        const R sym = p.w[cls] * base + P * p.K[cls] * cu * cu;
        const R asym = R(0.5) * P * p.A[cls] * cu;
        fc[q] = sym + asym;
        fc[q + 1] = sym - asym;
    }
    put_canonical<T, true>(grid, s, x, g, fc);
}

template <typename T, typename Out, bool FLAT>
__global__ void k27_moments(const T *__restrict__ grid, Out *rho, Out *u, Geo g, Relax27<typename Storage<T>::R> p,
                            int rho0_mode, Box box)
{
    using R = typename Storage<T>::R;
    LBM_Q27_PROLOGUE
    R fc[Q27];
    get_canonical<T, true>(grid, s, x, g, fc);
    R drho = fc[0], j[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int q = 1; q < Q27; ++q) {
        drho += fc[q];
        j[0] += R(CX(q)) * fc[q];
        j[1] += R(CY(q)) * fc[q];
        j[2] += R(CZ(q)) * fc[q];
    }
    const R inv = rho0_mode ? R(1) / (R(1) + drho) : R(1);
    if (rho) rho[cell] = Out(R(1) + drho);
    if (u)
        for (int i = 0; i < 3; ++i) u[i * g.ncell + cell] = Out((j[i] + p.half_a[i]) * inv);
}

template <typename T, bool FLAT>
__global__ void k27_get(const T *__restrict__ grid, T *__restrict__ dst, Geo g, Box box)
{
    LBM_Q27_PROLOGUE
    typename Storage<T>::R fc[Q27];
    get_canonical<T, true>(grid, s, x, g, fc);
#pragma unroll
    for (int q = 0; q < Q27; ++q) Storage<T>::store(dst + (long long)q * g.ncell + cell, fc[q]);
}

template <typename T, bool FLAT>
__global__ void k27_set(T *grid, const T *__restrict__ src, Geo g, Box box)
{
    LBM_Q27_PROLOGUE
    typename Storage<T>::R fc[Q27];
#pragma unroll
    for (int q = 0; q < Q27; ++q) fc[q] = Storage<T>::load(src + (long long)q * g.ncell + cell);
    put_canonical<T, true>(grid, s, x, g, fc);
}

}  // namespace q27

// ---------------------------------------------------------------- dispatch

template <typename F>
static cudaError_t q27_by_prec(int prec, F &&f)
{
    switch (prec) {
    case P_F64: return f(double());
    case P_F32: return f(float());
    case P_F16: return f(__half());
    case P_BF16: return f(__nv_bfloat16());
    }
    return cudaErrorInvalidValue;
}

constexpr int Q27_THREADS = 256;
static Box q27_box(const Geo &g) { return Box(g.nx, 0, g.ny, 0, g.nz); }
// Threads along x of blocks that are rectangles of rows, 128 where `rows` says that they
// pay and the grid can have the rows; 0: the cells as one sequence.
static int q27_block(const Geo &g, int threads, bool rows)
{
    return rows && threads % 128 == 0 && (g.ny + threads / 128 - 1) / (threads / 128) <= 65535 ? 128 : 0;
}

template <typename... P, typename... A>
static cudaError_t launch27(void (*flat)(P...), void (*rectangles)(P...), const Geo &g, bool rows, cudaStream_t stream,
                            A &&...args)
{
    const int bx = q27_block(g, Q27_THREADS, rows);
    launch_step_box(bx ? rectangles : flat, false, q27_box(g), bx, Q27_THREADS, stream, std::forward<A>(args)...);
    return cudaGetLastError();
}

cudaError_t launch_step27(int prec, const void *src, void *dst, const Geo &g, const CollBoth &c, LaunchShape s,
                          cudaStream_t stream)
{
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
    return q27_by_prec(prec, [&](auto t) {
        using T = decltype(t);
        using R = typename Storage<T>::R;
        const q27::Relax27<R> p = q27::to_relax27<R>(c);
        const T *a = (const T *)src;
        T *b = (T *)dst;
        if constexpr (sizeof(T) == 2) {
            if (s.cells_x == 4 && g.nx % 4 == 0) {
                // four cells per thread; with walls, the interior rows run the periodic
                // code (or with walls on x the x-walls-only one) and the wall rows the
                // walled one: walled channel 512x256x256, FP16, 0.68 -> 1.0 of the copy
                // bandwidth
                auto run = [&](auto rho0, auto walled) {
                    constexpr bool RH = decltype(rho0)::value, W = decltype(walled)::value;
                    if constexpr (W) {
                        launch_step_walls(g.wall_x ? q27::k27_ab4_walls<T, RH, true> : q27::k27_ab4_walls<T, RH, false>, false,
                                          WalledBox(g.nx / 4, g.nx / 4, g, QUAD_THREADS, false), QUAD_THREADS, stream, a, b, g,
                                          p);
                    } else {
                        const Box box(g.nx / 4, 0, g.ny, 0, g.nz);
                        const int bx = box.block_x(QUAD_THREADS);
                        launch_step_box(bx ? q27::k27_ab4<T, RH, false> : q27::k27_ab4<T, RH, true>, false, box, bx, QUAD_THREADS,
                                        stream, a, b, g, p);
                    }
                };
                if (c.rho0_is_rho && walls) run(std::true_type{}, std::true_type{});
                else if (c.rho0_is_rho) run(std::true_type{}, std::false_type{});
                else if (walls) run(std::false_type{}, std::true_type{});
                else run(std::false_type{}, std::false_type{});
                return cudaGetLastError();
            }
        }
        const Box box = q27_box(g);
        const int bx = q27_block(g, s.threads, walls && g.nx % 128 == 0);
        auto k = c.rho0_is_rho ? (bx      ? q27::k27_ab1<T, true, true, false>
                                  : walls ? q27::k27_ab1<T, true, true>
                                          : q27::k27_ab1<T, true, false>)
                               : (bx      ? q27::k27_ab1<T, false, true, false>
                                  : walls ? q27::k27_ab1<T, false, true>
                                          : q27::k27_ab1<T, false, false>);
        launch_step_box(k, true, box, bx, s.threads, stream, a, b, g, p);
        return cudaGetLastError();
    });
}

bool pair_runs27_f32(const Geo &g, bool always) { return pair_runs<q27::Lat27>(g, always, {3.05, 3.0, 1.3, 32.0}); }

cudaError_t launch_pair27_f32(const void *src, void *dst, const Geo &g, const CollBoth &c, cudaStream_t s)
{
    using L = q27::Lat27;
    const q27::Relax27<float> p = q27::to_relax27<float>(c);
    const PairPlanes<L> S = pair_planes<L>(src, g.ncell), D = pair_planes<L>(dst, g.ncell);
    const bool walls = g.wall_x || g.wall_y || g.wall_z;
    if (c.rho0_is_rho)
        return walls ? launch_pair_k<L, true, true, false>(S, D, g, p, s) : launch_pair_k<L, true, false, false>(S, D, g, p, s);
    return walls ? launch_pair_k<L, false, true, false>(S, D, g, p, s) : launch_pair_k<L, false, false, false>(S, D, g, p, s);
}

cudaError_t launch_init27(int prec, void *grid, const void *rho, const void *u, int dtype, const Geo &g,
                          const CollBoth &c, cudaStream_t stream)
{
    return q27_by_prec(prec, [&](auto t) {
        using T = decltype(t);
        using R = typename Storage<T>::R;
        const q27::Relax27<R> p = q27::to_relax27<R>(c);
        if (dtype == 0)
            return launch27(q27::k27_init<T, double>, q27::k27_init<T, double>, g, false, stream, (T *)grid,
                            (const double *)rho, (const double *)u, g, p, c.rho0_is_rho);
        return launch27(q27::k27_init<T, float>, q27::k27_init<T, float>, g, false, stream, (T *)grid, (const float *)rho,
                        (const float *)u, g, p, c.rho0_is_rho);
    });
}

cudaError_t launch_moments27(int prec, const void *grid, void *rho, void *u, int dtype, const Geo &g,
                             const CollBoth &c, cudaStream_t stream)
{
    return q27_by_prec(prec, [&](auto t) {
        using T = decltype(t);
        using R = typename Storage<T>::R;
        const q27::Relax27<R> p = q27::to_relax27<R>(c);
        if (dtype == 0)
            return launch27(q27::k27_moments<T, double, true>, q27::k27_moments<T, double, false>, g, g.nx % 128 == 0, stream,
                            (const T *)grid, (double *)rho, (double *)u, g, p, c.rho0_is_rho);
        return launch27(q27::k27_moments<T, float, true>, q27::k27_moments<T, float, false>, g, g.nx % 128 == 0, stream, (const T *)grid,
                        (float *)rho, (float *)u, g, p, c.rho0_is_rho);
    });
}

cudaError_t launch_get27(int prec, const void *grid, void *dst, const Geo &g, cudaStream_t stream)
{
    return q27_by_prec(prec, [&](auto t) {
        using T = decltype(t);
        return launch27(q27::k27_get<T, true>, q27::k27_get<T, false>, g, g.nx % 128 == 0, stream, (const T *)grid, (T *)dst, g);
    });
}

cudaError_t launch_set27(int prec, void *grid, const void *src, const Geo &g, cudaStream_t stream)
{
    return q27_by_prec(prec, [&](auto t) {
        using T = decltype(t);
        // its scattered stores run faster in rectangles although those leave lanes idle
        // (FP32: 259x307x95 327 against 274 us, 70x200x200 128 against 112; FP16 33x300x300
        // 100 against 128)
        return launch27(q27::k27_set<T, true>, q27::k27_set<T, false>, g, g.nx > 64, stream, (T *)grid, (const T *)src, g);
    });
}

int velocity_set27(int *c, double *w, int *opp)
{
    for (int q = 0; q < q27::Q27; ++q) {
        if (c) {
            c[3 * q + 0] = q27::CX(q);
            c[3 * q + 1] = q27::CY(q);
            c[3 * q + 2] = q27::CZ(q);
        }
        if (w) w[q] = q27::WQ(q);
        if (opp) opp[q] = q27::OPP(q);
    }
    return q27::Q27;
}

}  // namespace lbm
