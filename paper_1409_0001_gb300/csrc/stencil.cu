// stencil.cu -- diffusion smoothing on a uniform hex mesh (Section 2.6 step 2,
// Section 3.2 Eq. (diffusion), zero-flux walls of Section 3.2.2).
//
// Finite-volume 7-point Laplacian per unit cell volume: (L u)_k = sum over the
// existing face neighbours l of (u_l - u_k) / dx^2.  A wall face carries no flux, so
// a missing neighbour drops out of both the sum and the diagonal.  One pseudo-step of
// implicit Euler solves A u^{n+1} = u^n with A = I - c L (c = dtau/dx^2, L unscaled);
// Crank-Nicolson (the paper's scheme, Section 5.1) solves (I - c/2 L) u^{n+1} =
// (I + c/2 L) u^n; explicit Euler is u += c L u.
//
// Two solvers:
//  * FP64: conjugate gradients in two fused passes per iteration (pass 1 forms the new
//    search direction p = r + beta p on the fly at a cell and its neighbours, and
//    accumulates p.Ap; pass 2 recomputes Ap, updates x and r, and accumulates r.r).
//    Scalars stay on the device; the last block of each pass finishes the reduction
//    in a fixed order, so results are run-to-run deterministic.
//  * Mixed: FP64 iterative refinement.  A fused FP64 pass applies the previous
//    correction (x += d), forms the true residual r = b - A x in FP64 and stores it in
//    FP32 (or BF16); the correction A d = r is then solved in FP32 by Chebyshev
//    iteration, whose spectrum bounds are known in closed form on this mesh:
//    lambda(A) lies in [1, 1 + 4 c sum_axes sin^2(pi (n-1) / (2n))] (DCT-II
//    eigenvalues).  Chebyshev needs no inner products, only stencil sweeps.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <type_traits>
#include <mutex>
#include <vector>

#include "grid_stride.cuh"
#include "internal.cuh"
#include "reduce.cuh"

namespace cgk {

namespace {

constexpr int TX = 32, TY = 8;     // xy tile of the 2.5D sweeps (one thread per column)

struct Geo {
    int nx, ny, nz;
    int nxy;
    int n;
    int per = 0;   // periodic axes: bit 0 x, bit 1 y, bit 2 z (scalar engines only)
};

// Launch geometry of a 2.5D sweep: blocks of TX x TY columns, each marching over zlen
// planes; blockIdx.z = f * nzc + z-chunk.
struct Sweep {
    dim3 grid;
    int zlen, nzc, nb;   // planes per chunk, chunks, blocks per field
};

// Geometry for a given z-chunk length (planes per block).
Sweep make_sweep_z(const Geo &g, int nf, int zlen) {
    Sweep s;
    int gx = (g.nx + TX - 1) / TX, gy = (g.ny + TY - 1) / TY;
    zlen = zlen < 1 ? 1 : (zlen > g.nz ? g.nz : zlen);
    int nzc = (g.nz + zlen - 1) / zlen;
    s.grid = dim3(gx, gy, nzc * nf);
    s.zlen = zlen;
    s.nzc = nzc;
    s.nb = gx * gy * nzc;
    return s;
}

// Whether a launch of zlen planes a block has a valid grid (blockIdx.z: chunks x fields).
inline bool grid_z_fits(const Geo &g, int nf, int zlen) {
    return (long long)((g.nz + zlen - 1) / zlen) * nf <= 65535;
}

Sweep make_sweep(const Geo &g, int nf) {
    Sweep s;
    int gx = (g.nx + TX - 1) / TX, gy = (g.ny + TY - 1) / TY;
    long long cols = (long long)gx * gy * nf;
    long long target = (long long)num_sms() * 16;   // ~2 waves of 8 resident blocks per SM
    int nzc = (int)((target + cols - 1) / cols);
    int zlen = (g.nz + nzc - 1) / nzc;
    if (zlen < 4) zlen = g.nz < 4 ? g.nz : 4;
    nzc = (g.nz + zlen - 1) / zlen;
    s.grid = dim3(gx, gy, nzc * nf);
    s.zlen = zlen;
    s.nzc = nzc;
    s.nb = gx * gy * nzc;
    return s;
}

struct BlockPos {
    int f, z0, z1, bid, nb;
};

__device__ __forceinline__ BlockPos block_pos(const Geo &g, int zlen, int nzc) {
    BlockPos p;
    p.f = blockIdx.z / nzc;
    int zc = blockIdx.z - p.f * nzc;
    p.z0 = zc * zlen;
    p.z1 = min(g.nz, p.z0 + zlen);
    p.bid = (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    p.nb = gridDim.x * gridDim.y * nzc;
    return p;
}

// The 2.5D engine.  Each thread owns one (x, y) column of the tile and marches over the
// planes [z0, z1): the value of the stencil field at a cell is produced once
// (produce(k)), kept in a 3-deep register queue for the z neighbours and published in a
// shared (TY+2) x (TX+2) plane for the x and y neighbours; pre(k) loads the values the
// update needs at the cell itself.  Every load for plane z+1 (its values, the
// cell-local operands and the tile's halo) is issued while plane z is being computed,
// so the memory latency of a plane hides behind the work of the previous one.  For
// every cell of the column, consume(k, v, s, nn, pt) receives its value v, the sum s of
// its face neighbours (order x-, x+, y-, y+, z-, z+), their number nn and pre's result
// pt.  A wall face has no neighbour: its shared-memory slot and queue entry stay zero,
// so it adds nothing to s, and it is not counted in nn (zero flux).
struct NoPre {};

// load(k) returns a cell's raw operands and finish(raw) its stencil value; the next
// plane's operands are loaded before the current plane is computed and finished after it
// (a double-float sum of iterate and correction does not wait on its loads in front of
// the plane's work).  sweep25_at below is the form with values that need no finishing.
template <class T, class Load, class Finish, class Pre, class Consume>
__device__ __forceinline__ void sweep25_lf(const Geo &g, int bx, int by, int z0, int z1, Load load,
                                           Finish finish, Pre pre, Consume consume) {
    __shared__ T pl[TY + 2][TX + 2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = bx * TX + tx, y = by * TY + ty;
    const bool own = (x < g.nx) && (y < g.ny);
    const int kxy = y * g.nx + x;
    const bool px = g.per & 1, py = (g.per >> 1) & 1, pz = (g.per >> 2) & 1;
    // halo roles: which neighbour column (if any) this thread also loads -- the first
    // and the last column / row of the tile inside the mesh; across a periodic axis the
    // neighbour of the mesh's first (last) cell is its last (first)
    const int xe = min(bx * TX + TX, g.nx) - 1, ye = min(by * TY + TY, g.ny) - 1;
    const bool hxl = (tx == 0) && (x > 0 || px) && (y < g.ny) && (x < g.nx);
    const bool hxh = (x == xe) && (x + 1 < g.nx || px) && (y < g.ny);
    const bool hyl = (ty == 0) && (y > 0 || py) && (x < g.nx) && (y < g.ny);
    const bool hyh = (y == ye) && (y + 1 < g.ny || py) && (x < g.nx);
    const int dxl = x > 0 ? -1 : g.nx - 1, dxh = x + 1 < g.nx ? 1 : 1 - g.nx;
    const int dyl = y > 0 ? -g.nx : (g.ny - 1) * g.nx, dyh = y + 1 < g.ny ? g.nx : (1 - g.ny) * g.nx;
    const int nnxy = (px ? 2 : (x > 0) + (x + 1 < g.nx)) + (py ? 2 : (y > 0) + (y + 1 < g.ny));
    // plane offsets of the z neighbours (periodic z wraps)
    auto zdn = [&](int z) { return z > 0 ? -g.nxy : (g.nz - 1) * g.nxy; };
    auto zup = [&](int z) { return z + 1 < g.nz ? g.nxy : (1 - g.nz) * g.nxy; };
    // zero the plane once: wall slots and the slots of columns outside the mesh are
    // never written again
    for (int i = ty * TX + tx; i < (TY + 2) * (TX + 2); i += TX * TY) (&pl[0][0])[i] = T();
    __syncthreads();

    using P = decltype(pre(0));
    using RAW = decltype(load(0));
    auto produce = [&](int k) { return finish(load(k)); };
    T vdn = T(), vc = T(), vup = T();               // v(z-1), v(z), v(z+1) of the column
    T hxa = T(), hxb = T(), hya = T(), hyb = T();   // halo values of plane z
    P pt{};                                         // cell-local operands of plane z
    if (z0 < z1) {
        const int k0 = kxy + z0 * g.nxy;
        if (own) {
            if (z0 > 0 || pz) vdn = produce(k0 + zdn(z0));
            vc = produce(k0);
            if (z0 + 1 < g.nz || pz) vup = produce(k0 + zup(z0));
            pt = pre(k0);
        }
        if (hxl) hxa = produce(k0 + dxl);
        if (hxh) hxb = produce(k0 + dxh);
        if (hyl) hya = produce(k0 + dyl);
        if (hyh) hyb = produce(k0 + dyh);
    }
    for (int z = z0; z < z1; ++z) {
        const int kz = kxy + z * g.nxy;
        // loads for the next plane of this block (raw operands, finished below)
        RAW nup{}, nxa{}, nxb{}, nya{}, nyb{};
        P npt{};
        if (z + 1 < z1) {
            const int kn = kz + g.nxy;
            if (own) {
                if (z + 2 < g.nz || pz) nup = load(kn + zup(z + 1));
                npt = pre(kn);
            }
            if (hxl) nxa = load(kn + dxl);
            if (hxh) nxb = load(kn + dxh);
            if (hyl) nya = load(kn + dyl);
            if (hyh) nyb = load(kn + dyh);
        }
        // publish plane z and update its cells
        if (own) pl[ty + 1][tx + 1] = vc;
        if (hxl) pl[ty + 1][0] = hxa;
        if (hxh) pl[ty + 1][tx + 2] = hxb;
        if (hyl) pl[0][tx + 1] = hya;
        if (hyh) pl[ty + 2][tx + 1] = hyb;
        __syncthreads();
        if (own) {
            T s = pl[ty + 1][tx];
            s += pl[ty + 1][tx + 2];
            s += pl[ty][tx + 1];
            s += pl[ty + 2][tx + 1];
            s += vdn;
            s += vup;
            const int nn = nnxy + (pz ? 2 : (z > 0) + (z + 1 < g.nz));
            consume(kz, vc, s, nn, pt);
        }
        __syncthreads();
        vdn = vc;
        vc = vup;
        vup = finish(nup);   // a zero operand set finishes to a zero value
        pt = npt;
        hxa = finish(nxa);
        hxb = finish(nxb);
        hya = finish(nya);
        hyb = finish(nyb);
    }
}

template <class T, class Produce, class Pre, class Consume>
__device__ __forceinline__ void sweep25_at(const Geo &g, int bx, int by, int z0, int z1,
                                           Produce produce, Pre pre, Consume consume) {
    sweep25_lf<T>(g, bx, by, z0, z1, produce, [](T v) { return v; }, pre, consume);
}

// A flat-plane variant of the engine for meshes of short rows (nx <= kFlatMaxNx,
// walls only), whose cost does not depend on nx: the block covers CPT kThreads
// consecutive cells [q0, q0 + CPT kThreads) of the flattened xy plane (q = y nx + x;
// thread t holds the cells q0 + t + kThreads j, j < CPT, so every load is coalesced
// whatever nx is) and
// marches over the planes [z0, z1).  Plane z is published in a shared segment with nx
// cells of halo either side, which holds every x and y neighbour; z neighbours come from
// register queues; loads for plane z+1 are issued while plane z is computed.  consume()
// receives exactly what sweep25_at gives it -- the same neighbour sum in the same order
// (x-, x+, y-, y+, z-, z+, a wall adding a zero) -- so results are bit-identical.
constexpr int kFlatMaxNx = 512;
constexpr int kFlatCpt = 4;     // cells per thread of the FP32 / BF16 sweeps
constexpr int kFlatCptDF = 2;   // ... of the double-float refinement passes

//
// load(k) returns a cell's raw operands and finish(raw) its stencil value: the loads for
// plane z+1 are issued before plane z is computed, and finish() runs after it, so the
// arithmetic that turns them into values (a double-float sum of the iterate and its
// correction) does not wait on the loads in front of the plane's work.
template <class T, int CPT, class Load, class Finish, class Pre, class Consume>
__device__ __forceinline__ void sweep_flat_at(const Geo &g, int pts, int chunk, int z0, int z1,
                                              Load load, Finish finish, Pre pre, Consume consume) {
    constexpr int kFlatCells = CPT * kThreads;
    __shared__ T sp[kFlatCells + 2 * kFlatMaxNx];
    const int t = threadIdx.y * TX + threadIdx.x;
    const int nx = g.nx, nxy = g.nxy;
    const int q0 = chunk * kFlatCells;
    // the block's cells and their x/y neighbours (bits: x-, x+, y-, y+)
    int nnxy[CPT];
    unsigned nb[CPT];
    bool own[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        const int q = q0 + t + kThreads * j;
        own[j] = q < nxy;
        const int iy = q / nx, ix = q - iy * nx;
        nb[j] = (ix > 0 ? 1u : 0u) | (ix + 1 < nx ? 2u : 0u) | (iy > 0 ? 4u : 0u) |
                (iy + 1 < g.ny ? 8u : 0u);
        nnxy[j] = __popc(nb[j]);
    }
    // halo cells of the segment: [q0 - nx, q0) and [q0 + kFlatCells, q0 + kFlatCells + nx)
    // inside the plane; thread t loads cells t and t + kThreads of each side
    const int lo0 = max(q0 - nx, 0);
    const int hi0 = q0 + kFlatCells, hi1 = min(q0 + kFlatCells + nx, nxy);
    bool hl[2], hh[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        hl[j] = lo0 + t + kThreads * j < q0;
        hh[j] = hi0 + t + kThreads * j < hi1;
    }
    using P = decltype(pre(0));
    using RAW = decltype(load(0, 0));
    // a cell's index k in the dense field and kt in the inner vectors (planes pts apart)
    auto produce = [&](int k, int kt) { return finish(load(k, kt)); };
    T vdn[CPT], vc[CPT], vup[CPT], ha[2], hb[2];
    P pt[CPT];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
        vdn[j] = T();
        vc[j] = T();
        vup[j] = T();
        pt[j] = P{};
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        ha[j] = T();
        hb[j] = T();
    }
    if (z0 < z1) {
        const int kz = z0 * nxy, kzt = z0 * pts;
#pragma unroll
        for (int j = 0; j < CPT; ++j)
            if (own[j]) {
                const int k = kz + q0 + t + kThreads * j, kt = kzt + q0 + t + kThreads * j;
                if (z0 > 0) vdn[j] = produce(k - nxy, kt - pts);
                vc[j] = produce(k, kt);
                if (z0 + 1 < g.nz) vup[j] = produce(k + nxy, kt + pts);
                pt[j] = pre(k);
            }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (hl[j]) ha[j] = produce(kz + lo0 + t + kThreads * j, kzt + lo0 + t + kThreads * j);
            if (hh[j]) hb[j] = produce(kz + hi0 + t + kThreads * j, kzt + hi0 + t + kThreads * j);
        }
    }
    // segment slot of cell q: q - q0 + nx
    for (int z = z0; z < z1; ++z) {
        const int kz = z * nxy, kzt = z * pts;
        RAW nup[CPT], na[2], nbv[2];   // raw operands of plane z+1's (z+2's) values
        P npt[CPT];
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            nup[j] = RAW{};
            npt[j] = P{};
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            na[j] = RAW{};
            nbv[j] = RAW{};
        }
        if (z + 1 < z1) {
            const int kn = kz + nxy, knt = kzt + pts;
#pragma unroll
            for (int j = 0; j < CPT; ++j)
                if (own[j]) {
                    const int k = kn + q0 + t + kThreads * j, kt = knt + q0 + t + kThreads * j;
                    if (z + 2 < g.nz) nup[j] = load(k + nxy, kt + pts);
                    npt[j] = pre(k);
                }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (hl[j]) na[j] = load(kn + lo0 + t + kThreads * j, knt + lo0 + t + kThreads * j);
                if (hh[j]) nbv[j] = load(kn + hi0 + t + kThreads * j, knt + hi0 + t + kThreads * j);
            }
        }
#pragma unroll
        for (int j = 0; j < CPT; ++j)
            if (own[j]) sp[t + kThreads * j + nx] = vc[j];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (hl[j]) sp[lo0 + t + kThreads * j - q0 + nx] = ha[j];
            if (hh[j]) sp[hi0 + t + kThreads * j - q0 + nx] = hb[j];
        }
        __syncthreads();
        const int nnz = (z > 0) + (z + 1 < g.nz);
#pragma unroll
        for (int j = 0; j < CPT; ++j)
            if (own[j]) {
                const int i = t + kThreads * j + nx;
                T s = (nb[j] & 1u) ? sp[i - 1] : T();
                s += (nb[j] & 2u) ? sp[i + 1] : T();
                s += (nb[j] & 4u) ? sp[i - nx] : T();
                s += (nb[j] & 8u) ? sp[i + nx] : T();
                s += vdn[j];
                s += vup[j];
                consume(kz + q0 + t + kThreads * j, kzt + q0 + t + kThreads * j, vc[j], s, nnxy[j] + nnz,
                        pt[j]);
            }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            vdn[j] = vc[j];
            vc[j] = vup[j];
            vup[j] = finish(nup[j]);   // a zero operand set finishes to a zero value
            pt[j] = npt[j];
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            ha[j] = finish(na[j]);
            hb[j] = finish(nbv[j]);
        }
    }
}

// Without cell-local prefetch: consume(k, v, s, nn).
template <class T, class Produce, class Consume>
__device__ __forceinline__ void sweep25_at(const Geo &g, int bx, int by, int z0, int z1,
                                           Produce produce, Consume consume) {
    sweep25_at<T>(
        g, bx, by, z0, z1, produce, [](int) { return NoPre{}; },
        [&](int k, T v, T s, int nn, NoPre) { consume(k, v, s, nn); });
}

template <class T, class Produce, class Pre, class Consume>
__device__ __forceinline__ void sweep25p(const Geo &g, int z0, int z1, Produce produce, Pre pre,
                                         Consume consume) {
    sweep25_at<T>(g, blockIdx.x, blockIdx.y, z0, z1, produce, pre, consume);
}

template <class T, class Produce, class Consume>
__device__ __forceinline__ void sweep25(const Geo &g, int z0, int z1, Produce produce,
                                        Consume consume) {
    sweep25_at<T>(g, blockIdx.x, blockIdx.y, z0, z1, produce, consume);
}

// A register-blocked variant of the engine for short sweeps: the block covers ZB planes
// [z0, z0+ZB) of its tile and every thread issues all of its loads for them at once (the
// column's ZB+2 values, the cell-local operands of the ZB planes and its halo values),
// publishes the ZB planes in shared memory, passes one barrier and updates its ZB cells.
// Many independent loads per thread and a single barrier per block keep the memory
// pipes busy.  consume() receives the same arguments as with sweep25_at.
template <int ZB, class T, class Produce, class Pre, class Consume>
__device__ __forceinline__ void sweepzb(const Geo &g, int bx, int by, int z0, Produce produce,
                                        Pre pre, Consume consume) {
    __shared__ T pl[ZB][TY + 2][TX + 2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = bx * TX + tx, y = by * TY + ty;
    const bool own = (x < g.nx) && (y < g.ny);
    const int kxy = y * g.nx + x;
    const bool hxl = (tx == 0) && (x > 0) && (y < g.ny);
    const bool hxh = (tx == TX - 1) && (x + 1 < g.nx) && (y < g.ny);
    const bool hyl = (ty == 0) && (y > 0) && (x < g.nx);
    const bool hyh = (ty == TY - 1) && (y + 1 < g.ny) && (x < g.nx);
    const int nnxy = (x > 0) + (x + 1 < g.nx) + (y > 0) + (y + 1 < g.ny);
    using P = decltype(pre(0));
    T v[ZB + 2];
    P pt[ZB];
#pragma unroll
    for (int i = 0; i < ZB + 2; ++i) {
        const int z = z0 - 1 + i;
        v[i] = (own && z >= 0 && z < g.nz) ? produce(kxy + z * g.nxy) : T();
    }
#pragma unroll
    for (int i = 0; i < ZB; ++i) {
        const int z = z0 + i;
        pt[i] = (own && z < g.nz) ? pre(kxy + z * g.nxy) : P{};
    }
    T hal[ZB];
    const bool halo = hxl || hxh || hyl || hyh;
    const int hoff = hxl ? -1 : (hxh ? 1 : (hyl ? -g.nx : g.nx));
#pragma unroll
    for (int i = 0; i < ZB; ++i) {
        const int z = z0 + i;
        hal[i] = (halo && z < g.nz) ? produce(kxy + z * g.nxy + hoff) : T();
    }
    // a corner thread of the tile holds two halo roles: its second one (y) is loaded here
    const bool halo2 = (hxl || hxh) && (hyl || hyh);
    const int hoff2 = hyl ? -g.nx : g.nx;
    T hal2[ZB];
#pragma unroll
    for (int i = 0; i < ZB; ++i) {
        const int z = z0 + i;
        hal2[i] = (halo2 && z < g.nz) ? produce(kxy + z * g.nxy + hoff2) : T();
    }
    // publish: zero everything first (walls and columns outside the mesh stay zero)
    for (int i = ty * TX + tx; i < ZB * (TY + 2) * (TX + 2); i += TX * TY) (&pl[0][0][0])[i] = T();
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ZB; ++i) {
        if (own) pl[i][ty + 1][tx + 1] = v[i + 1];
        if (hxl) pl[i][ty + 1][0] = hal[i];
        else if (hxh) pl[i][ty + 1][TX + 1] = hal[i];
        else if (hyl) pl[i][0][tx + 1] = hal[i];
        else if (hyh) pl[i][TY + 1][tx + 1] = hal[i];
        if (halo2) {
            if (hyl) pl[i][0][tx + 1] = hal2[i];
            else pl[i][TY + 1][tx + 1] = hal2[i];
        }
    }
    __syncthreads();
    if (own) {
#pragma unroll
        for (int i = 0; i < ZB; ++i) {
            const int z = z0 + i;
            if (z < g.nz) {
                T s = pl[i][ty + 1][tx];
                s += pl[i][ty + 1][tx + 2];
                s += pl[i][ty][tx + 1];
                s += pl[i][ty + 2][tx + 1];
                s += v[i];
                s += v[i + 2];
                const int nn = nnxy + (z > 0) + (z + 1 < g.nz);
                consume(kxy + z * g.nxy, v[i + 1], s, nn, pt[i]);
            }
        }
    }
}

struct Scal {
    double rr, bb, alpha, beta;
    int done, iters;
    unsigned int ticket;
    int breakdown;
};

// Diagonal of A = I - ce L per neighbour count: dg[nn] = 1 + ce * nn.
struct Coef64 {
    double ce;
    double dg[7];
};
struct Coef32 {
    float ce;
    float dg[7];
};

// ================================================================ FP64 conjugate gradients
// r = b - A x = c L x for both schemes (x = u^n), p = r; b = u^n (implicit Euler) or
// u^n + c/2 L u^n (Crank-Nicolson).  rr and bb are reduced.
__global__ void __launch_bounds__(kThreads) k_cg_init(Geo g, int zlen, int nzc, double c,
                                                      int scheme, const double *__restrict__ xall,
                                                      double *__restrict__ rall,
                                                      double *__restrict__ pall,
                                                      double *__restrict__ partials_all,
                                                      Scal *__restrict__ sc, double tol2) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const double *x = xall + off;
    double *r = rall + off;
    double *p = pall + off;
    double rr = 0.0, bb = 0.0;
    sweep25<double>(
        g, bp.z0, bp.z1, [&](int k) { return x[k]; },
        [&](int k, double v, double s, int nn) {
            double lx = s - nn * v;
            double rk = c * lx;
            double bk = scheme == 1 ? v + 0.5 * c * lx : v;
            r[k] = rk;
            p[k] = rk;
            rr += rk * rk;
            bb += bk * bk;
        });
    double vals[2] = {block_sum(rr), block_sum(bb)};
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, 2, vals, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double RR = finish_sum(partials, 0, bp.nb);
        double BB = finish_sum(partials, 1, bp.nb);
        if (is_thread0()) {
            Scal &S = sc[bp.f];
            S.rr = RR;
            S.bb = BB;
            S.beta = 0.0;
            S.iters = 0;
            S.breakdown = 0;
            S.done = (RR <= tol2 * BB) ? 1 : 0;
            S.ticket = 0;
        }
    }
}

// pass 1: p = r + beta p (produced once per cell), accumulate p.Ap; A p is kept in q
// (q_all != nullptr) for k_cg_update, which then needs no stencil of its own
__global__ void __launch_bounds__(kThreads) k_cg_pass1(Geo g, int zlen, int nzc, Coef64 cf,
                                                       const double *__restrict__ rall,
                                                       const double *__restrict__ pin_all,
                                                       double *__restrict__ pout_all,
                                                       double *__restrict__ q_all,
                                                       double *__restrict__ partials_all,
                                                       Scal *__restrict__ sc) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    if (sc[bp.f].done) return;
    const double beta = sc[bp.f].beta;
    const size_t off = (size_t)bp.f * g.n;
    const double *r = rall + off;
    const double *pin = pin_all + off;
    double *pout = pout_all + off;
    double *qv = q_all ? q_all + off : nullptr;
    double pap = 0.0;
    __shared__ double sdg[8];
    stage_table(sdg, cf.dg);
    sweep25<double>(
        g, bp.z0, bp.z1, [&](int k) { return fma(beta, pin[k], r[k]); },
        [&](int k, double v, double s, int nn) {
            double ap = fma(sdg[nn], v, -cf.ce * s);
            pout[k] = v;
            if (qv) qv[k] = ap;
            pap = fma(v, ap, pap);
        });
    double val = block_sum(pap);
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, 1, &val, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double PAP = finish_sum(partials, 0, bp.nb);
        if (is_thread0()) {
            Scal &S = sc[bp.f];
            if (PAP > 0.0) {
                S.alpha = S.rr / PAP;
            } else {
                S.alpha = 0.0;
                S.breakdown = 1;
                S.done = 1;
            }
            S.ticket = 0;
        }
    }
}

// pass 2: recompute Ap, x += alpha p, r -= alpha Ap, accumulate r.r
__global__ void __launch_bounds__(kThreads) k_cg_pass2(Geo g, int zlen, int nzc, Coef64 cf,
                                                       const double *__restrict__ pall,
                                                       double *__restrict__ xall,
                                                       double *__restrict__ rall,
                                                       double *__restrict__ partials_all,
                                                       Scal *__restrict__ sc, double tol2) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    if (sc[bp.f].done) return;
    const double alpha = sc[bp.f].alpha;
    const size_t off = (size_t)bp.f * g.n;
    const double *p = pall + off;
    double *x = xall + off;
    double *r = rall + off;
    double rr = 0.0;
    __shared__ double sdg[8];
    stage_table(sdg, cf.dg);
    sweep25p<double>(
        g, bp.z0, bp.z1, [&](int k) { return p[k]; },
        [&](int k) { return double2{x[k], r[k]}; },
        [&](int k, double v, double s, int nn, double2 xr) {
            double ap = fma(sdg[nn], v, -cf.ce * s);
            x[k] = fma(alpha, v, xr.x);
            double rk = fma(-alpha, ap, xr.y);
            r[k] = rk;
            rr = fma(rk, rk, rr);
        });
    double val = block_sum(rr);
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, 1, &val, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double RR = finish_sum(partials, 0, bp.nb);
        if (is_thread0()) {
            Scal &S = sc[bp.f];
            S.beta = RR / S.rr;
            S.rr = RR;
            S.iters += 1;
            S.done = (RR <= tol2 * S.bb) ? 1 : 0;
            S.ticket = 0;
        }
    }
}

// pass 2 with A p at hand: x += alpha p, r -= alpha q, accumulate r.r.  Pointwise, four
// cells in flight per thread: 3 FP64 instructions per cell instead of the 10 of k_cg_pass2
// (the FP64 pipe is what bounds both), for 8 more bytes written and 8 more read.  Per
// iteration (both passes) 100^3 91.5 -> 70.2 us, 128^3 124.8 -> 96.8 us.
__global__ void __launch_bounds__(kThreads) k_cg_update(int n, int nb, const double *__restrict__ pall,
                                                        const double *__restrict__ qall,
                                                        double *__restrict__ xall,
                                                        double *__restrict__ rall,
                                                        double *__restrict__ partials_all,
                                                        Scal *__restrict__ sc, double tol2) {
    const int f = blockIdx.y;
    if (sc[f].done) return;
    const double alpha = sc[f].alpha;
    const size_t off = (size_t)f * n;
    const double *p = pall + off, *q = qall + off;
    double *x = xall + off, *r = rall + off;
    double rr = 0.0;
    grid_stride<4>(
        n, blockIdx.x * kThreads + threadIdx.x, gridDim.x * kThreads,
        [&](uint32_t k, uint32_t step) {   // four cells in flight
            double pv[4], qv[4], xv[4], rv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                pv[j] = p[k + j * step];
                qv[j] = q[k + j * step];
                xv[j] = x[k + j * step];
                rv[j] = r[k + j * step];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                x[k + j * step] = fma(alpha, pv[j], xv[j]);
                const double rk = fma(-alpha, qv[j], rv[j]);
                r[k + j * step] = rk;
                rr = fma(rk, rk, rr);
            }
        },
        [&](uint32_t k) {
            x[k] = fma(alpha, p[k], x[k]);
            const double rk = fma(-alpha, q[k], r[k]);
            r[k] = rk;
            rr = fma(rk, rk, rr);
        });
    double val = block_sum(rr);
    double *partials = partials_all + (size_t)f * 2 * nb;
    if (arrive(partials, 1, &val, blockIdx.x, gridDim.x, &sc[f].ticket)) {
        double RR = finish_sum(partials, 0, gridDim.x);
        if (is_thread0()) {
            Scal &S = sc[f];
            S.beta = RR / S.rr;
            S.rr = RR;
            S.iters += 1;
            S.done = (RR <= tol2 * S.bb) ? 1 : 0;
            S.ticket = 0;
        }
    }
}

// ---------------------------------------------------------------- FP64 CG on the chip
// The whole FP64 solve of a call (every step, every field, every iteration) as one
// cooperative launch for meshes whose x, r and p fit in the SMs' registers: a block owns
// a run of consecutive cells, a thread up to C of them (x, r and p as 6 C registers), and
// only p (for the neighbours' stencils) and one partial sum per block go through global
// memory.  Per iteration three grid barriers: p published, p.Ap reduced, r.r reduced.
// Bound: the FP64 pipe (two lanes per clock and SM: 12 FP64 instructions per cell and
// iteration against 19 in the two-launch form that forms A p twice) plus the barriers;
// the two-launch form spends 12-13 us per launch on meshes this small, most of it launch
// latency, the last block's sum of the partials and too few resident warps.  Measured per
// iteration (b = 3 dx, one field): 32^3 27.0 -> 9.6 us, 48^3 27.1 -> 11.5, 64^3 33.0 ->
// 15.3, 96^3 65.1 -> 30.1.  Each block adds all blocks' partials itself, in block order,
// so the sums are the same bits in every block and every run.  (Partials tagged with the
// sum's number and polled by every block, which needs no arrival counter, took 2 us more
// at 32^3: 152 blocks polling 152 slots.)
// Fields are independent, so several run at a time on meshes whose blocks have 128 threads: the
// launch's blocks form groups of `blocks`, up to four blocks to an SM, each with its own barrier and partial sums; group q solves fields q, q + groups,
// .. and the groups meet once per step.  A field's block layout, and with it its bits, do not
// depend on how many there are.  (One field after the other, 8^3 x 8 fields took 12.7 ms a
// call and 32^3 x 5 fields 10.9, against 5.7 and 7.4 in the two-launch form, which runs all
// fields in one launch; in groups 1.8 and 4.9.)
struct __align__(128) CoopBar {   // a group's; the last one is the whole launch's
    unsigned int count;
    int err;
    int failed[2];   // a field of an even / odd step did not converge (the last one's)
};
constexpr int kCoopMaxC = 12;    // cells per thread: 6 C registers of state within 128
// Blocks that an SM's registers hold: 72 and 80 registers a thread for one and two cells, else
// 128.  Small solves of several streams share the SMs the better the more of them fit (six
// calls of 32^3 at a time 5.4 ms, 7.6 with four blocks of 104 registers).
constexpr int coop_blocks_per_sm(int NT, int C) { return NT == 128 && C <= 2 ? 8 - C : 512 / NT; }

// One group's place in the launch.
struct CoopGroup {
    int id, count, block, blocks;   // the group, of how many; this block's number in it, of how many
    CoopBar *bars;                  // every group's, then the whole launch's
};

// Arrival of every block that counts on bar b, `target` in all; bounded like grid_sync.  A wait
// that gives up raises every bar's err, so that no other block waits on.
__device__ __forceinline__ bool coop_sync(const CoopGroup &cg, int b, unsigned target, long long budget) {
    CoopBar *gb = cg.bars + b;
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->count) : "memory");
        const long long t0 = clock64();
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&gb->count) : "memory");
            if ((int)(v - target) >= 0) break;
            if (*(volatile int *)&gb->err) { ok = 0; break; }
            if (clock64() - t0 > budget) {
                for (int q = 0; q <= cg.count; ++q) atomicExch(&cg.bars[q].err, 1);
                ok = 0;
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// The scalars of a field's iteration, kept by thread 0 of every block: one thread divides
// and compares (on every thread these few FP64 operations would cost more pipe time than
// a small mesh's stencils).
struct CoopScal {
    double rr, bb, stop, alpha, beta;
    int done, breakdown;
};

// Group-wide sums of a value (TWO: two values) per thread, the same bits in every block;
// fin(a, b) runs on thread 0 with the totals, and its writes to shared memory are visible
// to the block on return.  The block sum goes through shared memory in full-warp
// additions (36 FP64 warp instructions for 512 threads; a shuffle tree in every warp
// would take 85).  NT: the block's threads (a multiple of 128).
template <int NT, bool TWO, class Fin>
__device__ __forceinline__ bool coop_sum(double a, double b, double2 *part, const CoopGroup &cg, unsigned target,
                                         long long budget, Fin fin) {
    __shared__ double2 sv[NT];
    const int t = threadIdx.x;
    sv[t] = make_double2(a, b);
    __syncthreads();
    if (t < 128) {
        double2 v = sv[t];
#pragma unroll
        for (int q = 1; q < NT / 128; ++q) {
            const double2 o = sv[t + 128 * q];
            v.x += o.x;
            if (TWO) v.y += o.y;
        }
        sv[t] = v;
    }
    __syncthreads();
    if (t < 32) {
        double2 v = sv[t];
#pragma unroll
        for (int q = 1; q < 4; ++q) {
            const double2 o = sv[t + 32 * q];
            v.x += o.x;
            if (TWO) v.y += o.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            if (TWO) v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if (t == 0) __stcg(&part[cg.block], v);
    }
    if (!coop_sync(cg, cg.id, target, budget)) return false;
    if (t < 32) {
        double2 v = make_double2(0.0, 0.0);
        for (int i = t; i < cg.blocks; i += 32) {
            const double2 o = __ldcg(&part[i]);
            v.x += o.x;
            if (TWO) v.y += o.y;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
            if (TWO) v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
        }
        if (t == 0) fin(v.x, v.y);
    }
    __syncthreads();
    return true;
}

// cells (read only) -> X (the solution); V: per group (vstride apart) the vector published
// for the neighbours; part: 2 x gridDim.x partials (alternating); hist[s * nf + f].  A
// field's iteration stops as in the two-launch form: converged, breakdown, or max_it.  After
// a step in which a field did not converge nothing more runs.
template <int NT, int C>
__global__ void __launch_bounds__(NT, coop_blocks_per_sm(NT, C)) k_cg_coop(
    Geo g, int blocks, int per_block, double c, Coef64 cf, int scheme, int nf, int nsteps, int max_it, double tol2,
    const double *__restrict__ cells, double *X, double *V, size_t vstride, double2 *part,
    Scal *__restrict__ hist, CoopBar *bars, long long budget) {
    __shared__ double sdg[8];
    __shared__ unsigned short face[C][NT];
    __shared__ CoopScal S;
    stage_table(sdg, cf.dg);
    __syncthreads();
    const int n = g.n, nx = g.nx, nxy = g.nxy;
    const int gid = (int)blockIdx.x / blocks;
    const CoopGroup cg{gid, (int)gridDim.x / blocks, (int)blockIdx.x - gid * blocks, blocks, bars};
    V += gid * vstride;
    part += 2 * gid * blocks;
    const int k0 = cg.block * per_block + threadIdx.x;
    const int kend = min(n, (cg.block + 1) * per_block);
    // per cell: which neighbours lie across a wall (no neighbour) or a periodic face, two
    // bits per face (0: the adjacent cell, 1: none, 2: the other end of the axis)
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int k = k0 + j * NT;
        if (k < kend) {
            const int z = k / nxy, q = k - z * nxy, y = q / nx, x = q - y * nx;
            const unsigned wx = (g.per & 1) ? 2u : 1u, wy = (g.per & 2) ? 2u : 1u, wz = (g.per & 4) ? 2u : 1u;
            face[j][threadIdx.x] = (unsigned short)(
                (x == 0 ? wx : 0u) | (x + 1 == nx ? wx : 0u) << 2 | (y == 0 ? wy : 0u) << 4 |
                (y + 1 == g.ny ? wy : 0u) << 6 | (z == 0 ? wz : 0u) << 8 | (z + 1 == g.nz ? wz : 0u) << 10);
        }
    }
    unsigned target = 0, target_all = 0;
    int par = 0;
    auto nb = [&](const double *v, int k, unsigned w, int step, int wrap) -> double {
        return w == 1u ? 0.0 : __ldcg(v + k + (w == 0u ? step : wrap));
    };
    // sum of the neighbours of cell k (x-, x+, y-, y+, z-, z+) and their number
    auto stencil = [&](const double *v, int k, unsigned f, int &nn) -> double {
        const double a0 = nb(v, k, f & 3u, -1, nx - 1), a1 = nb(v, k, f >> 2 & 3u, 1, 1 - nx);
        const double a2 = nb(v, k, f >> 4 & 3u, -nx, nxy - nx), a3 = nb(v, k, f >> 6 & 3u, nx, nx - nxy);
        const double a4 = nb(v, k, f >> 8 & 3u, -nxy, n - nxy), a5 = nb(v, k, f >> 10 & 3u, nxy, nxy - n);
        nn = 6 - __popc(f & 0x555u);
        return ((((a0 + a1) + a2) + a3) + a4) + a5;
    };
    bool failed = false;
    for (int s = 0; s < nsteps && !failed; ++s) {
        for (int f = cg.id; f < nf; f += cg.count) {
            double *Xf = X + (size_t)f * n;
            const double *xin = s == 0 ? cells + (size_t)f * n : Xf;
            double x[C], r[C], p[C];
            double rr = 0.0, bb = 0.0;
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int k = k0 + j * NT;
                x[j] = r[j] = p[j] = 0.0;
                if (k < kend) {
                    int nn;
                    const double v = __ldcg(xin + k), sm = stencil(xin, k, face[j][threadIdx.x], nn);
                    const double lx = sm - nn * v;
                    const double rk = c * lx, bk = scheme == 1 ? v + 0.5 * c * lx : v;
                    x[j] = v;
                    r[j] = rk;
                    rr += rk * rk;
                    bb += bk * bk;
                }
            }
            target += blocks;
            if (!coop_sum<NT, true>(rr, bb, part + par * blocks, cg, target, budget, [&](double RR, double BB) {
                    S.rr = RR;
                    S.bb = BB;
                    S.stop = tol2 * BB;
                    S.beta = 0.0;
                    S.done = RR <= S.stop;
                    S.breakdown = 0;
                }))
                return;
            par ^= 1;
            int it = 0;
            while (!S.done && it < max_it) {
                const double beta = S.beta;
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const int k = k0 + j * NT;
                    if (k < kend) {
                        p[j] = fma(beta, p[j], r[j]);
                        __stcg(V + k, p[j]);
                    }
                }
                target += blocks;
                if (!coop_sync(cg, cg.id, target, budget)) return;
                double ap[C];
                double pap = 0.0;
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    const int k = k0 + j * NT;
                    ap[j] = 0.0;
                    if (k < kend) {
                        int nn;
                        const double sm = stencil(V, k, face[j][threadIdx.x], nn);
                        ap[j] = fma(sdg[nn], p[j], -cf.ce * sm);
                        pap = fma(p[j], ap[j], pap);
                    }
                }
                target += blocks;
                if (!coop_sum<NT, false>(pap, 0.0, part + par * blocks, cg, target, budget, [&](double PAP, double) {
                        S.breakdown = !(PAP > 0.0);
                        S.alpha = S.rr / PAP;
                    }))
                    return;
                par ^= 1;
                if (S.breakdown) break;
                const double alpha = S.alpha;
                double rn = 0.0;
#pragma unroll
                for (int j = 0; j < C; ++j) {
                    x[j] = fma(alpha, p[j], x[j]);
                    r[j] = fma(-alpha, ap[j], r[j]);
                    rn = fma(r[j], r[j], rn);
                }
                target += blocks;
                if (!coop_sum<NT, false>(rn, 0.0, part + par * blocks, cg, target, budget, [&](double RR, double) {
                        S.beta = RR / S.rr;
                        S.rr = RR;
                        S.done = RR <= S.stop;
                    }))
                    return;
                par ^= 1;
                ++it;
            }
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const int k = k0 + j * NT;
                if (k < kend) __stcg(Xf + k, x[j]);
            }
            if (cg.block == 0 && threadIdx.x == 0) {
                Scal &H = hist[(size_t)s * nf + f];
                H.rr = S.rr;
                H.bb = S.bb;
                H.iters = it;
                H.breakdown = S.breakdown;
                H.done = S.done;
            }
            if (S.breakdown ? S.rr > S.stop : !S.done) failed = true;
            // X is read by other blocks in the next step's first pass (and V rewritten)
            target += blocks;
            if (!coop_sync(cg, cg.id, target, budget)) return;
        }
        if (cg.count > 1) {   // every group has finished the step; one that failed stops all
            int *flag = &bars[cg.count].failed[s & 1];   // (alternating: read before it is set again)
            if (failed && cg.block == 0 && threadIdx.x == 0) atomicExch(flag, 1);
            target_all += gridDim.x;
            if (!coop_sync(cg, cg.count, target_all, budget)) return;
            failed = *(volatile int *)flag != 0;
        }
    }
}

// The solution of k_cg_coop into the caller's array, unless a wait gave up (the caller's
// field is then as it was, and the two-launch form solves it).
__global__ void k_cg_coop_out(size_t n, const double *__restrict__ X, double *__restrict__ cells,
                              const CoopBar *bars) {
    if (bars->err) return;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        cells[i] = X[i];
}

// explicit Euler: x_out = x + c L x (FP64)
__global__ void __launch_bounds__(kThreads) k_explicit(Geo g, int zlen, int nzc, double c,
                                                       const double *__restrict__ xin_all,
                                                       double *__restrict__ xout_all) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const double *x = xin_all + off;
    double *y = xout_all + off;
    sweep25<double>(
        g, bp.z0, bp.z1, [&](int k) { return x[k]; },
        [&](int k, double v, double s, int nn) { y[k] = v + c * (s - nn * v); });
}

// ---------------------------------------------------------------- explicit Euler, temporally blocked
// K explicit Euler steps per launch in FP32 storage and arithmetic (3.5D blocking).  A
// block holds a tile of kEW x kEH columns (32 lanes x two x-cells, 16 warps x two rows)
// and marches in z.  At iteration p it loads plane p of the input (level 0) and computes
// level t at plane p - t for t = 1..K, so a level's z neighbours are the last three
// planes of the level below, kept per thread in registers, and its x and y neighbours
// are the level below at the same plane: lane shuffles in x, the thread's own second row
// or a shared plane per level in y.  That shared plane was written one iteration earlier
// into the other of two buffers, so one barrier per iteration orders every exchange.
// The valid region shrinks by one column and row per level on each side; the block
// writes level K on its inner (kEW - 2K) x (kEH - 2K) columns.  Cells outside the mesh
// (and planes outside it) hold zero and are not counted as neighbours (zero-flux walls);
// on a periodic axis coordinates wrap and every cell has both neighbours.  Every cell
// update is the same expression in the same order whatever K, so the result does not
// depend on K.
constexpr int kEW = 64, kEH = 32;
constexpr dim3 kEBlock(32, 16);
constexpr int kEStages = 4;   // input planes staged ahead by cp.async (three in flight)

__host__ __device__ constexpr size_t explicit_tb_smem(int K) {
    return (size_t)(kEStages + 2 * K) * kEH * kEW * sizeof(float);
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Asynchronous global -> shared copies of 16, 8 or 4 bytes (both addresses aligned to
// the size); they land in the group the next cp_async_commit closes.
__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ int wrap_coord(int i, int n) {
    i %= n;
    return i < 0 ? i + n : i;
}

__global__ void k_to_f32(size_t n, const double *__restrict__ u, float *__restrict__ v) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        v[i] = __double2float_rn(u[i]);
}

__global__ void k_from_f32(size_t n, const float *__restrict__ v, double *__restrict__ u) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        u[i] = (double)v[i];
}

// The same K-step explicit march with four consecutive x-cells per thread (nx % 4 == 0):
// a block of 32 lanes x 32 rows holds a tile of 128 columns x 32 rows.  x neighbours
// inside a thread's four cells are in registers, across lanes they come by shuffle; y
// neighbours come from the per-level shared plane as 128-bit loads; each thread stages
// its own four input cells of a plane with one 16-byte cp.async.  Between tiles there is a
// fixed halo of four columns (so every tile starts 16-byte aligned, whatever K) and of K
// rows; a tile at a wall starts or ends there without one, so that a tile writes 120, 124
// or 128 columns and 32 - 2K, 32 - K or 32 rows: 128 columns take one tile, not two.
// Beyond a tile's edge the x and y neighbours read zero (a zero row precedes every shared
// plane), which is the wall's value, and in a halo never reaches a written cell.  Every cell
// update is k_explicit_tb's expression in the same order, so the two kernels agree bit
// for bit.
// Issue-bound, so the instructions per cell and step decide: sums and updates run on cell
// pairs (16 arithmetic instructions per four cells against 36 as scalars), the march is
// unrolled by the ring's four slots (slots, parities and shared addresses are constants,
// and the two queue planes of a level change roles by name), the plane to stage is
// carried along instead of wrapped anew, and the z walls' face counts are off the common
// path: 41 -> 26 instructions per cell and step, 143 -> 110 us per launch of three steps on
// 512 x 256 x 256; what bounds it now is the shared planes' traffic (70 % of the LSU data
// pipe) beside issue (62 %).  40 steps, three per launch: 256 x 128 x 128 with two fields
// 0.88 -> 0.71 ms, 512 x 256 x 256 2.33 -> 1.87, 128^3 0.44 -> 0.36 and, with one tile over
// the 128 columns, 0.31.
constexpr int kE4W = 128, kE4H = 32, kE4OX = kE4W - 8;
constexpr int kE4P = kE4H + 1;   // rows of a level's shared plane: a zero row, then the tile's
constexpr dim3 kE4Block(32, kE4H);

__host__ __device__ constexpr size_t explicit_tb4_smem(int K) {
    return ((size_t)kEStages * kE4H + (size_t)2 * K * kE4P + 1) * kE4W * sizeof(float);
}

template <int K>
__global__ void __launch_bounds__(1024, 1) k_explicit_tb4(Geo g, int zlen, int nzc, float c,
                                                          const float *__restrict__ uin_all,
                                                          float *__restrict__ uout_all) {
    extern __shared__ float4 tb4_smem[];
    // stage[slot][row][128]; buf[level][parity][1 + row][128], levels 0..K-1, row 0 zero (and
    // a last zero row after the last plane)
    float(*stage)[kE4H][kE4W] = reinterpret_cast<float(*)[kE4H][kE4W]>(tb4_smem);
    float(*buf)[2][kE4P][kE4W] = reinterpret_cast<float(*)[2][kE4P][kE4W]>(&stage[kEStages][0][0]);
    constexpr int OY = kE4H - 2 * K;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int f = blockIdx.z / nzc, zc = blockIdx.z - f * nzc;
    const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
    const bool px = g.per & 1, py = (g.per >> 1) & 1, pz = (g.per >> 2) & 1;
    const float *uin = uin_all + (size_t)f * g.n;
    float *uout = uout_all + (size_t)f * g.n;

    // this thread's four cells: columns 4 lane .. 4 lane + 3 of row w
    const int xa = (int)blockIdx.x * kE4OX - (px ? 4 : 0) + 4 * lane;   // first column (a multiple of 4)
    const int y = (int)blockIdx.y * OY - (py ? K : 0) + w;
    const bool ey = py || (y >= 0 && y < g.ny);
    const bool ex = px || (xa >= 0 && xa < g.nx);        // the four cells share it (nx % 4 == 0)
    const int gx = px ? wrap_coord(xa, g.nx) : min(max(xa, 0), g.nx - 4);
    const int rowoff = (py ? wrap_coord(y, g.ny) : min(max(y, 0), g.ny - 1)) * g.nx + gx;
    const float cy = py ? 2.f : (float)((y > 0) + (y < g.ny - 1));
    float nxy[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        nxy[i] = (px ? 2.f : (float)((xa + i > 0) + (xa + i < g.nx - 1))) + cy;
    // a cell outside the mesh holds zero at every level: its step factor is zero
    const float2 cm = (ex && ey) ? make_float2(c, c) : make_float2(0.f, 0.f);
    const float2 nm01 = make_float2(-(nxy[0] + 2.f), -(nxy[1] + 2.f));   // - faces, away from the z walls
    const float2 nm23 = make_float2(-(nxy[2] + 2.f), -(nxy[3] + 2.f));
    // written: the mesh's cells that no other tile writes.  At a wall the first tile writes
    // from its first column and row, the last one to the mesh's end.
    const bool wx = xa >= 0 && xa < g.nx && (lane >= 1 || (!px && blockIdx.x == 0)) &&
                    (lane <= 30 || (!px && blockIdx.x == gridDim.x - 1));
    const bool wy = y >= 0 && y < g.ny && (w >= K || (!py && blockIdx.y == 0)) &&
                    (w < kE4H - K || (!py && blockIdx.y == gridDim.y - 1));
    const bool wr = wx && wy;
    // the level buffers start at zero, so every value a cell ever reads is finite
    for (int k = threadIdx.y * 32 + threadIdx.x; k < (K * 2 * kE4P + 1) * kE4W; k += 1024)
        (&buf[0][0][0][0])[k] = 0.f;
    __syncthreads();
    float4 Q[K][2];   // planes q-1 and q of the level below K; the planes of the march alternate
#pragma unroll
    for (int t = 0; t < K; ++t) Q[t][0] = Q[t][1] = make_float4(0.f, 0.f, 0.f, 0.f);

    const int p_begin = pz ? z0 - K : max(z0 - K, 0);
    const int p_end = pz ? z1 + K : min(z1 + K, g.nz + K);
    // level t's planes in this chunk: [lo(t), hi(t)), inside the mesh unless z is periodic
    auto lo = [&](int t) { return pz ? z0 - (K - t) : max(z0 - (K - t), 0); };
    auto hi = [&](int t) { return pz ? z1 + (K - t) : min(z1 + (K - t), g.nz); };
    // the next plane to stage: its number and, wrapped or clamped, its plane of the mesh
    int sp = p_begin, si = pz ? wrap_coord(p_begin, g.nz) : p_begin;
    const int sp_end = min(p_end, pz ? p_end : g.nz);
    const float *src = uin + rowoff;
    const unsigned stage0 = (unsigned)__cvta_generic_to_shared(&stage[0][w][4 * lane]);
    auto stage_plane = [&](int slot) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(stage0 + (unsigned)(slot * kE4H * kE4W * 4)),
                     "l"(src + (size_t)si * g.nxy), "r"((sp < sp_end && ex && ey) ? 16 : 0)
                     : "memory");
        cp_async_commit();
        ++sp;
        if (++si >= g.nz) si = pz ? 0 : g.nz - 1;
    };
    float *out = uout + (ptrdiff_t)(p_begin - K) * g.nxy + rowoff;   // level K's plane at p
    float(*const own)[2][kE4P][kE4W] = reinterpret_cast<float(*)[2][kE4P][kE4W]>(&buf[0][0][1 + w][4 * lane]);
#pragma unroll
    for (int d = 0; d < kEStages - 1; ++d) stage_plane(d);
    for (int p0 = p_begin; p0 < p_end; p0 += kEStages) {
#pragma unroll
        for (int i = 0; i < kEStages; ++i) {
            const int p = p0 + i, par = i & 1;
            if (p >= p_end) break;   // uniform
            stage_plane((i + kEStages - 1) & (kEStages - 1));   // past the end: an empty (zero-filled) group
            cp_async_wait<kEStages - 1>();                      // plane p has landed
            float4 nw = *reinterpret_cast<const float4 *>(&stage[i][w][4 * lane]);
            *reinterpret_cast<float4 *>(&own[0][par][0][0]) = nw;
#pragma unroll
            for (int t = 1; t <= K; ++t) {
                const int q = p - t;
                const bool in = q >= lo(t) && q < hi(t);   // uniform
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (in) {
                    float2 n01 = nm01, n23 = nm23;
                    if (!pz && (q == 0 || q == g.nz - 1)) {   // uniform: a z wall, or both
                        const float a = (float)((q == 0) + (q == g.nz - 1));
                        n01 = __fadd2_rn(n01, make_float2(a, a));
                        n23 = __fadd2_rn(n23, make_float2(a, a));
                    }
                    const float4 b = Q[t - 1][par ^ 1], za = Q[t - 1][par];
                    const float4 up = *reinterpret_cast<const float4 *>(&own[t - 1][par ^ 1][0][0] - kE4W);
                    const float4 dn = *reinterpret_cast<const float4 *>(&own[t - 1][par ^ 1][0][0] + kE4W);
                    float xl = __shfl_up_sync(0xffffffffu, b.w, 1);
                    float xr = __shfl_down_sync(0xffffffffu, b.x, 1);
                    if (lane == 0) xl = 0.f;
                    if (lane == 31) xr = 0.f;
                    const float2 b01 = make_float2(b.x, b.y), b23 = make_float2(b.z, b.w);
                    float2 s01 = make_float2(__fadd_rn(xl, b.y), __fadd_rn(b.x, b.z));
                    float2 s23 = make_float2(__fadd_rn(b.y, b.w), __fadd_rn(b.z, xr));
                    s01 = __fadd2_rn(s01, __fadd2_rn(make_float2(up.x, up.y), make_float2(dn.x, dn.y)));
                    s23 = __fadd2_rn(s23, __fadd2_rn(make_float2(up.z, up.w), make_float2(dn.z, dn.w)));
                    s01 = __fadd2_rn(s01, __fadd2_rn(make_float2(za.x, za.y), make_float2(nw.x, nw.y)));
                    s23 = __fadd2_rn(s23, __fadd2_rn(make_float2(za.z, za.w), make_float2(nw.z, nw.w)));
                    const float2 v01 = __ffma2_rn(cm, __ffma2_rn(n01, b01, s01), b01);
                    const float2 v23 = __ffma2_rn(cm, __ffma2_rn(n23, b23, s23), b23);
                    v = make_float4(v01.x, v01.y, v23.x, v23.y);
                }
                if (t < K)
                    *reinterpret_cast<float4 *>(&own[t][par][0][0]) = v;
                else if (in && wr)
                    *reinterpret_cast<float4 *>(out) = v;
                Q[t - 1][par] = nw;
                nw = v;
            }
            out += g.nxy;
            __syncthreads();
        }
    }
}

template <int K>
__global__ void __launch_bounds__(512, 2) k_explicit_tb(Geo g, int zlen, int nzc, float c,
                                                        const float *__restrict__ uin_all,
                                                        float *__restrict__ uout_all) {
    extern __shared__ float4 tb_smem[];
    // stage[slot][row][column]: input planes in flight; buf[level][parity][row][column],
    // levels 0..K-1
    float(*stage)[kEH][kEW] = reinterpret_cast<float(*)[kEH][kEW]>(tb_smem);
    float(*buf)[2][kEH][kEW] = reinterpret_cast<float(*)[2][kEH][kEW]>(&stage[kEStages][0][0]);
    constexpr int OX = kEW - 2 * K, OY = kEH - 2 * K;
    const int lane = threadIdx.x, w = threadIdx.y;
    const int f = blockIdx.z / nzc, zc = blockIdx.z - f * nzc;
    const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
    const bool px = g.per & 1, py = (g.per >> 1) & 1, pz = (g.per >> 2) & 1;
    const float *uin = uin_all + (size_t)f * g.n;
    float *uout = uout_all + (size_t)f * g.n;

    // per cell (row h, column i of the thread's 2 x 2): its offset in a plane, whether it
    // is in the mesh (as a 0/1 factor and as a copy size), its x-y face count, and
    // whether the block writes it
    int off[2][2], csz[2][2];
    float msk[2][2], nxy[2][2];
    bool wr[2][2];
    {
        int gx[2], gy[2];
        bool ex[2], ey[2], wx[2], wy[2];
        float cx[2], cy[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int j = 2 * lane + i, x = blockIdx.x * OX - K + j;
            ex[i] = px || (x >= 0 && x < g.nx);
            gx[i] = px ? wrap_coord(x, g.nx) : min(max(x, 0), g.nx - 1);
            cx[i] = px ? 2.f : (float)((x > 0) + (x < g.nx - 1));
            wx[i] = j >= K && j < kEW - K && x >= 0 && x < g.nx;
            const int r = 2 * w + i, y = blockIdx.y * OY - K + r;
            ey[i] = py || (y >= 0 && y < g.ny);
            gy[i] = py ? wrap_coord(y, g.ny) : min(max(y, 0), g.ny - 1);
            cy[i] = py ? 2.f : (float)((y > 0) + (y < g.ny - 1));
            wy[i] = r >= K && r < kEH - K && y >= 0 && y < g.ny;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                off[h][i] = gy[h] * g.nx + gx[i];
                csz[h][i] = (ex[i] && ey[h]) ? 4 : 0;
                msk[h][i] = (ex[i] && ey[h]) ? 1.f : 0.f;
                nxy[h][i] = cx[i] + cy[h];
                wr[h][i] = wx[i] && wy[h];
            }
    }
    // the level buffers start at zero, so every value a cell ever reads is finite
    for (int k = threadIdx.y * 32 + threadIdx.x; k < K * 2 * kEH * kEW; k += 512) (&buf[0][0][0][0])[k] = 0.f;
    __syncthreads();
    // queue of each level below K: planes q-1 (qa) and q (qb) of this thread's 2 x 2 cells
    float qa[K][2][2], qb[K][2][2];
#pragma unroll
    for (int t = 0; t < K; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i) qa[t][h][i] = qb[t][h][i] = 0.f;

    const int p_begin = pz ? z0 - K : max(z0 - K, 0);
    const int p_end = pz ? z1 + K : min(z1 + K, g.nz + K);
    // each thread stages its own four cells of a plane (zero outside the mesh), so
    // reading them back needs only its own wait, no barrier
    const unsigned stage0 = (unsigned)__cvta_generic_to_shared(&stage[0][2 * w][2 * lane]);
    auto stage_plane = [&](int p) {
        const bool zok = p < p_end && (pz || (p >= 0 && p < g.nz));
        const float *src = uin + (size_t)(pz ? wrap_coord(p, g.nz) : min(max(p, 0), g.nz - 1)) * g.nxy;
        const unsigned dst = stage0 + (unsigned)(((p - p_begin) & (kEStages - 1)) * kEH * kEW * 4);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int i = 0; i < 2; ++i)
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + (h * kEW + i) * 4),
                             "l"(src + off[h][i]), "r"(zok ? csz[h][i] : 0)
                             : "memory");
        cp_async_commit();
    };
#pragma unroll
    for (int d = 0; d < kEStages - 1; ++d) stage_plane(p_begin + d);
    for (int p = p_begin; p < p_end; ++p) {
        stage_plane(p + kEStages - 1);   // past the end: an empty (zero-filled) group
        cp_async_wait<kEStages - 1>();     // plane p has landed
        float nw[2][2];   // the newest plane of the level below: level 0 at plane p
        {
            const float(*src)[kEW] = stage[(p - p_begin) & (kEStages - 1)];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 v = *reinterpret_cast<const float2 *>(&src[2 * w + h][2 * lane]);
                nw[h][0] = v.x;
                nw[h][1] = v.y;
            }
        }
        const int par = p & 1;
#pragma unroll
        for (int h = 0; h < 2; ++h)
            *reinterpret_cast<float2 *>(&buf[0][par][2 * w + h][2 * lane]) = make_float2(nw[h][0], nw[h][1]);
#pragma unroll
        for (int t = 1; t <= K; ++t) {
            const int q = p - t;
            float v[2][2];
            if (q >= z0 - (K - t) && q < z1 + (K - t) && (pz || (q >= 0 && q < g.nz))) {   // uniform
                const float cz = pz ? 2.f : (float)((q > 0) + (q < g.nz - 1));
                // y neighbours outside the thread's two rows (row 2w-1 above, 2w+2 below)
                const float2 up = *reinterpret_cast<const float2 *>(&buf[t - 1][par ^ 1][max(2 * w - 1, 0)][2 * lane]);
                const float2 dn = *reinterpret_cast<const float2 *>(&buf[t - 1][par ^ 1][min(2 * w + 2, kEH - 1)][2 * lane]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float b0 = qb[t - 1][h][0], b1 = qb[t - 1][h][1];
                    const float xl = __shfl_up_sync(0xffffffffu, b1, 1);
                    const float xr = __shfl_down_sync(0xffffffffu, b0, 1);
                    const float yu0 = h ? qb[t - 1][0][0] : up.x, yu1 = h ? qb[t - 1][0][1] : up.y;
                    const float yd0 = h ? dn.x : qb[t - 1][1][0], yd1 = h ? dn.y : qb[t - 1][1][1];
                    const float s0 = ((xl + b1) + (yu0 + yd0)) + (qa[t - 1][h][0] + nw[h][0]);
                    const float s1 = ((b0 + xr) + (yu1 + yd1)) + (qa[t - 1][h][1] + nw[h][1]);
                    v[h][0] = msk[h][0] * fmaf(c, fmaf(-(nxy[h][0] + cz), b0, s0), b0);
                    v[h][1] = msk[h][1] * fmaf(c, fmaf(-(nxy[h][1] + cz), b1, s1), b1);
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) v[h][0] = v[h][1] = 0.f;
            }
            if (t < K) {
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<float2 *>(&buf[t][par][2 * w + h][2 * lane]) = make_float2(v[h][0], v[h][1]);
            } else if (q >= z0 && q < z1) {   // uniform
                float *dst = uout + (size_t)q * g.nxy;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        if (wr[h][i]) dst[off[h][i]] = v[h][i];
            }
            // shift the queue of level t-1; level t's new plane feeds level t+1
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    qa[t - 1][h][i] = qb[t - 1][h][i];
                    qb[t - 1][h][i] = nw[h][i];
                    nw[h][i] = v[h][i];
                }
        }
        __syncthreads();
    }
}

// ================================================================ mixed precision
template <class TS> __device__ __forceinline__ float ld(const TS *p, int i);
template <> __device__ __forceinline__ float ld<float>(const float *p, int i) { return p[i]; }
template <> __device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16 *p, int i) {
    return __bfloat162float(p[i]);
}
// L2-coherent loads (bypass L1) for data that other blocks of the same launch write.
template <class TS> __device__ __forceinline__ float ldcg(const TS *p, int i);
template <> __device__ __forceinline__ float ldcg<float>(const float *p, int i) {
    return __ldcg(p + i);
}
template <> __device__ __forceinline__ float ldcg<__nv_bfloat16>(const __nv_bfloat16 *p, int i) {
    unsigned short u = __ldcg(reinterpret_cast<const unsigned short *>(p) + i);
    return __bfloat162float(__ushort_as_bfloat16(u));
}
template <class TS> __device__ __forceinline__ void st(TS *p, int i, float v);
template <> __device__ __forceinline__ void st<float>(float *p, int i, float v) { p[i] = v; }
template <> __device__ __forceinline__ void st<__nv_bfloat16>(__nv_bfloat16 *p, int i, float v) {
    p[i] = __float2bfloat16_rn(v);
}

struct RefScal {
    double rr, bb;
    unsigned int ticket;
    int pad;
};

// One FP64 refinement pass.  kFirst: x = x_in (no correction), r = c L x_in, and
// b = x_in (implicit Euler) or x_in + c/2 L x_in written to b_out (Crank-Nicolson).
// Otherwise x = x_in + d (produced once per cell), x_out = x, r = b - A x.  Stores r and
// the first Chebyshev iterate y1 = gamma r in the storage type; reduces ||r||^2 (and
// ||b||^2 on the first pass) in FP64.
template <class TS, bool kFirst>
__global__ void __launch_bounds__(kThreads) k_refine(Geo g, int zlen, int nzc, double c,
                                                     Coef64 cf, int scheme,
                                                     const double *__restrict__ xin_all,
                                                     const TS *__restrict__ d_all,
                                                     const double *__restrict__ b_all,
                                                     double *__restrict__ xout_all,
                                                     double *__restrict__ bout_all,
                                                     TS *__restrict__ r_all, TS *__restrict__ y1_all,
                                                     float gamma, double *__restrict__ partials_all,
                                                     RefScal *__restrict__ sc) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const double *xin = xin_all + off;
    TS *r = r_all + off;
    TS *y1 = y1_all + off;
    double rr = 0.0, bb = 0.0;
    if (kFirst) {
        sweep25<double>(
            g, bp.z0, bp.z1, [&](int k) { return xin[k]; },
            [&](int k, double v, double s, int nn) {
                double lx = s - nn * v;
                double rk = c * lx;
                double bk = v;
                if (scheme == 1) {
                    bk = fma(0.5 * c, lx, v);
                    bout_all[off + k] = bk;
                }
                bb = fma(bk, bk, bb);
                float rf = (float)rk;
                st(r, k, rf);
                st(y1, k, gamma * rf);
                rr = fma(rk, rk, rr);
            });
    } else {
        const TS *d = d_all + off;
        const double *b = b_all + off;
        double *xout = xout_all + off;
        __shared__ double sdg[8];
        stage_table(sdg, cf.dg);
        sweep25p<double>(
            g, bp.z0, bp.z1, [&](int k) { return xin[k] + (double)ld(d, k); },
            [&](int k) { return b[k]; },
            [&](int k, double v, double s, int nn, double bk) {
                xout[k] = v;
                double rk = fma(cf.ce, s, fma(-sdg[nn], v, bk));   // b - (dg v - ce s)
                float rf = (float)rk;
                st(r, k, rf);
                st(y1, k, gamma * rf);
                rr = fma(rk, rk, rr);
            });
    }
    double vals[2] = {block_sum(rr), kFirst ? block_sum(bb) : 0.0};
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, kFirst ? 2 : 1, vals, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double RR = finish_sum(partials, 0, bp.nb);
        double BB = kFirst ? finish_sum(partials, 1, bp.nb) : 0.0;
        if (is_thread0()) {
            sc[bp.f].rr = RR;
            if (kFirst) sc[bp.f].bb = BB;
            sc[bp.f].ticket = 0;
        }
    }
}

// One Chebyshev iteration (see k_cheb_loop for the recurrence) as its own launch:
// y_next = omega (y - y_prev + gamma (r - A y)) + y_prev; y_prev == nullptr means 0.
// y_next may alias y_prev (both are accessed only at the cell itself).
template <class TS>
__global__ void __launch_bounds__(kThreads) k_cheb(Geo g, int zlen, int nzc, Coef32 cf,
                                                   float gamma, float omega,
                                                   const TS *__restrict__ y_all,
                                                   const TS *yprev_all,
                                                   const TS *__restrict__ r_all, TS *ynext_all) {
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const TS *y = y_all + off;
    const TS *r = r_all + off;
    const TS *yp = yprev_all ? yprev_all + off : nullptr;
    TS *yn = ynext_all + off;
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    sweep25p<float>(
        g, bp.z0, bp.z1, [&](int k) { return ld(y, k); },
        [&](int k) { return float2{yp ? ld(yp, k) : 0.0f, ld(r, k)}; },
        [&](int k, float v, float s, int nn, float2 pt) {
            float ay = fmaf(sdg[nn], v, -cf.ce * s);
            st(yn, k, fmaf(omega, v - pt.x + gamma * (pt.y - ay), pt.x));
        });
}

// ---------------------------------------------------------------- double-float refinement
// An FP64-class residual without FP64 arithmetic (GB300 runs FP64 at a small fraction
// of its FP32 rate).  A value is the unevaluated sum hi + lo of two FP32 numbers
// (about 48 significant bits), combined with the error-free transformations of
// Knuth (TwoSum: s + e = a + b exactly) and Dekker (Fast2Sum for |a| >= |b|; the
// rounding error of a product recovered with a fused multiply-add).  The sum below is
// the "sloppy" variant: its error is bounded relative to |a| + |b| rather than to the
// result, which is what a residual b - A x needs (accurate relative to |b|).
struct DF {
    float hi, lo;
};

__device__ __forceinline__ DF df_two_sum(float a, float b) {
    float s = a + b;
    float bb = s - a;
    float e = (a - (s - bb)) + (b - bb);
    return DF{s, e};
}
__device__ __forceinline__ DF df_fast2sum(float a, float b) {
    float s = a + b;
    float e = b - (s - a);
    return DF{s, e};
}
__device__ __forceinline__ DF operator+(DF a, DF b) {
    DF s = df_two_sum(a.hi, b.hi);
    s.lo += a.lo + b.lo;
    return df_fast2sum(s.hi, s.lo);
}
// Accumulation of a neighbour sum (every `s += x` on double-float values is one): the
// hi parts by a TwoSum cascade, the cascade's errors and the lo parts added in FP32,
// with no renormalisation per term (Ogita, Rump and Oishi's Sum2 applied to the hi
// parts).  The result is an unevaluated, unnormalised pair; its error is of the order
// u^2 times the sum of the terms' magnitudes (u = 2^-24), the same order as a chain of
// normalised additions, at 8 instead of 11 operations per term.
__device__ __forceinline__ DF &operator+=(DF &a, DF b) {
    const DF t = df_two_sum(a.hi, b.hi);
    a.hi = t.hi;
    a.lo = a.lo + (t.lo + b.lo);
    return a;
}
__device__ __forceinline__ DF df_add_f(DF a, float b) {
    DF s = df_two_sum(a.hi, b);
    s.lo += a.lo;
    return df_fast2sum(s.hi, s.lo);
}
// (Products are rounded explicitly: fused into the sum that follows, as the compiler may in
// one instantiation and not in another, they would change its bits.)
__device__ __forceinline__ DF df_mul(DF a, DF b) {
    float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return df_fast2sum(p, e);
}
__device__ __forceinline__ float df_f(DF a) { return a.hi + a.lo; }

// c * a without the final renormalisation: the exact product of the hi parts (FMA) plus
// the cross terms, as an unevaluated pair (for a value that is rounded to FP32 or added
// into another pair next).
__device__ __forceinline__ DF df_mul_un(DF c, DF a) {
    const float p = __fmul_rn(c.hi, a.hi);
    float e = fmaf(c.hi, a.hi, -p);
    e = fmaf(c.hi, a.lo, e);
    e = fmaf(c.lo, a.hi, e);
    return DF{p, e};
}

// L = s - nn v: the Laplacian numerator of a cell from its neighbour sum s (as the
// engines accumulate it) and its own value v; one TwoSum where the two meet.
__device__ __forceinline__ DF df_lap(DF s, DF v, float nn) {
    const float p = __fmul_rn(nn, v.hi);
    const float ep = fmaf(nn, v.hi, -p);
    const DF t = df_two_sum(s.hi, -p);
    return DF{t.hi, ((s.lo - fmaf(nn, v.lo, ep)) + t.lo)};
}

// The residual of an implicit step at a cell, r = b - A v with A v = v - ce L
// (ce = theta dtau / dx^2, L = df_lap): r = (b - v) + ce L, one TwoSum for b - v and one
// where it meets ce L; returned unnormalised (df_f gives its FP32 value).
__device__ __forceinline__ DF df_res(DF b, DF v, DF ce, DF L) {
    const DF t = df_two_sum(b.hi, -v.hi);
    const float tl = (b.lo - v.lo) + t.lo;
    const DF q = df_mul_un(ce, L);
    const DF u = df_two_sum(t.hi, q.hi);
    return DF{u.hi, (tl + q.lo) + u.lo};
}

struct CoefDF {
    DF c, half_c, ce;
    DF dg[7];
};

// ---- the same double-float operations on a cell pair, one packed instruction per pair
// (the f32x2 add, multiply and fused multiply-add of sm_100 and later).  A DF2 holds the
// hi parts of two cells in one float2 and their lo parts in another; every operation
// below is, cell by cell, the IEEE operation of its scalar counterpart above, in the same
// order, so the two cells' results are bit-identical to two scalar evaluations.
// Negations that the scalar forms get for free as operand modifiers are folded instead:
// a constant's negative is kept beside it, and an exact product error is carried negated
// (p - c a is exact, so it equals -(c a - p) without rounding).
struct DF2 {
    float2 hi, lo;
};
struct DFd {    // a double-float iterate and its FP32 correction, not yet added
    DF x;
    float d;
};
struct DF2n {   // the pair value hi - nlo (a product with its error carried negated)
    float2 hi, nlo;
};
struct DFc2 {   // a double-float constant broadcast to both cells, with its negative
    float2 hi, lo, nhi, nlo;
};
__device__ __forceinline__ DFc2 dfc2(DF c) {
    return DFc2{make_float2(c.hi, c.hi), make_float2(c.lo, c.lo), make_float2(-c.hi, -c.hi),
                make_float2(-c.lo, -c.lo)};
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b as one fused multiply-add, -1 * b + a: the exact product, then a single rounding
// of the exact difference, i.e. the IEEE difference (CUDA has no packed subtract intrinsic)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}
__device__ __forceinline__ DF2 df2_two_sum(float2 a, float2 b) {
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return DF2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ DF2 df2_fast2sum(float2 a, float2 b) {
    const float2 s = add2(a, b);
    return DF2{s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ DF2 df2_add(DF2 a, DF2 b) {   // operator+
    DF2 s = df2_two_sum(a.hi, b.hi);
    s.lo = add2(s.lo, add2(a.lo, b.lo));
    return df2_fast2sum(s.hi, s.lo);
}
__device__ __forceinline__ void df2_acc(DF2 &a, DF2 b) {  // operator+= (the cascade)
    const DF2 t = df2_two_sum(a.hi, b.hi);
    a.hi = t.hi;
    a.lo = add2(a.lo, add2(t.lo, b.lo));
}
__device__ __forceinline__ DF2 df2_add_f(DF2 a, float2 b) {
    DF2 s = df2_two_sum(a.hi, b);
    s.lo = add2(s.lo, a.lo);
    return df2_fast2sum(s.hi, s.lo);
}
__device__ __forceinline__ float2 df2_f(DF2 a) { return add2(a.hi, a.lo); }
__device__ __forceinline__ float2 df2_f(DF2n a) { return sub2(a.hi, a.nlo); }
// c * a unnormalised (df_mul_un): the error terms are accumulated negated
__device__ __forceinline__ DF2n df2_mul_un(const DFc2 &c, DF2 a) {
    const float2 p = mul2(c.hi, a.hi);
    float2 en = fma2(c.nhi, a.hi, p);
    en = fma2(c.nhi, a.lo, en);
    en = fma2(c.nlo, a.hi, en);
    return DF2n{p, en};
}
__device__ __forceinline__ DF2 df2_mul(const DFc2 &c, DF2 a) {   // df_mul(c, a)
    const DF2n q = df2_mul_un(c, a);
    const float2 s = sub2(q.hi, q.nlo);
    return DF2{s, sub2(sub2(q.hi, s), q.nlo)};
}
// df_lap: nn and its negative per cell
__device__ __forceinline__ DF2 df2_lap(DF2 s, DF2 v, float2 nn, float2 nnn) {
    const float2 np = mul2(nnn, v.hi);          // -(nn v.hi), rounded
    const float2 ep = fma2(nn, v.hi, np);        // its exact error
    const DF2 t = df2_two_sum(s.hi, np);
    return DF2{t.hi, add2(sub2(s.lo, fma2(nn, v.lo, ep)), t.lo)};
}
// df_res: r = (b - v) + ce L
__device__ __forceinline__ DF2 df2_res(DF2 b, DF2 v, const DFc2 &ce, DF2 L) {
    const float2 s = sub2(b.hi, v.hi);
    const float2 bb = sub2(s, b.hi);
    const float2 e = sub2(sub2(b.hi, sub2(s, bb)), add2(v.hi, bb));
    const float2 tl = add2(sub2(b.lo, v.lo), e);
    const DF2n q = df2_mul_un(ce, L);
    const DF2 u = df2_two_sum(s, q.hi);
    return DF2{u.hi, add2(sub2(tl, q.nlo), u.lo)};
}
// a cell pair as the two-cells-per-thread kernels store it: (hi0, hi1, lo0, lo1)
__device__ __forceinline__ DF2 df2_of(float4 v) {
    return DF2{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
__device__ __forceinline__ float4 f4_of(DF2 a) { return make_float4(a.hi.x, a.hi.y, a.lo.x, a.lo.y); }

// A double as hi = fl32(v), lo = fl32(v - hi).  (By integer arithmetic on the significand, as
// df_join: the integer to float conversion is no faster than the four FP64 instructions
// it saves, 163 against 129 us for 16.8 M values.)
__device__ __forceinline__ DF df_split(double v) {
    const float hi = __double2float_rn(v);
    return DF{hi, __double2float_rn(v - (double)hi)};
}
// fl64(hi + lo) without the FP64 pipe, which takes 16 cycles per warp instruction and bound
// the conversion (three instructions a value): where hi's exponent lies in [-70, 126], hi's
// significand with 29 more bits plus lo in units of its last one, rounded half to even; the
// FP64 definition elsewhere and where the sum falls below hi's power of two.  The same
// bits; 16.8 M values 101 -> 56 us, 512 x 256 x 256 193 -> 100 us (5.3 TB/s).
__device__ __forceinline__ double df_join(float hi, float lo) {
    const unsigned hb = __float_as_uint(hi);
    const int e = (int)((hb >> 23) & 0xffu) - 127;
    if (e >= -70 && e <= 126) {
        const float l = __fmul_rn((hb >> 31) ? -lo : lo, __uint_as_float((unsigned)(52 - e + 127) << 23));
        const float k = floorf(l), fr = __fsub_rn(l, k);
        const long long h = (long long)((hb & 0x7fffffu) | 0x800000u) << 29;
        if (fabsf(l) < 1073741824.0f) {
            const long long s0 = h + (long long)__float2int_rn(k);
            const long long s = s0 + ((fr > 0.5f || (fr == 0.5f && (s0 & 1))) ? 1 : 0);
            if (s0 >= (1ll << 52) && s <= (1ll << 53))
                return __longlong_as_double((long long)((((unsigned long long)(e + 1023)) << 52) +
                                                        (unsigned long long)(s - (1ll << 52)) +
                                                        ((unsigned long long)(hb & 0x80000000u) << 32)));
        }
    } else if (((hb | __float_as_uint(lo)) & 0x7fffffffu) == 0) {
        return __longlong_as_double((long long)((unsigned long long)(hb & __float_as_uint(lo)) << 32));
    }
    return (double)hi + (double)lo;
}

__global__ void k_to_df(size_t n, const double *__restrict__ u, DF *__restrict__ x) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        x[i] = df_split(u[i]);
}

__global__ void k_from_df(size_t n, const DF *__restrict__ x, double *__restrict__ u) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x) {
        const DF v = x[i];
        u[i] = df_join(v.hi, v.lo);
    }
}

// The same conversions in the pair layout of the two-cells-per-thread kernels: cells
// 2i and 2i + 1 as one float4 (hi0, hi1, lo0, lo1).  Same values as k_to_df / k_from_df.
// (the caller's field may start at any multiple of eight bytes)
__global__ void k_to_df_pairs(size_t npairs, const double *__restrict__ u, float4 *__restrict__ x) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npairs;
         i += (size_t)gridDim.x * blockDim.x) {
        const DF a = df_split(u[2 * i]), b = df_split(u[2 * i + 1]);
        x[i] = make_float4(a.hi, b.hi, a.lo, b.lo);
    }
}

__global__ void k_from_df_pairs(size_t npairs, const float4 *__restrict__ x, double *__restrict__ u) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npairs;
         i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = x[i];
        u[2 * i] = df_join(v.x, v.z);
        u[2 * i + 1] = df_join(v.y, v.w);
    }
}

// The refinement pass of k_refine in double-float arithmetic (same roles of the
// arguments; x, b are double-float vectors).  kMode 0: the first pass of a step; 1: a
// refinement pass; 2: a step's last refinement pass, which also starts the next step:
// with x = u^{n+1} it has A x at hand, so the next step's first residual is
// c L x = (x - A x) / theta (theta = 1 implicit Euler, 1/2 Crank-Nicolson), written to
// r and y1 (and the next Crank-Nicolson right-hand side x + c/2 L x to bout).  Its
// ||b||^2 goes to sc_next, the finished step's ||r||^2 to sc.  4: a refinement pass that
// also reduces ||b||^2 (the first pass of a step whose correction comes from the shared
// expansion); 5: a step's last refinement pass when nothing follows from its r (no r and
// y1 written).
// TD: the stored type of the correction d (FP32 for the shared expansion's increments).
template <class TS, int kMode, class TD = TS>
__global__ void __launch_bounds__(kThreads) k_refine_df(Geo g, int zlen, int nzc, CoefDF cf,
                                                        int scheme, const DF *__restrict__ xin_all,
                                                        const TD *__restrict__ d_all,
                                                        const DF *b_all, DF *__restrict__ xout_all,
                                                        DF *bout_all, TS *__restrict__ r_all,
                                                        TS *__restrict__ y1_all, float gamma,
                                                        double *__restrict__ partials_all,
                                                        RefScal *__restrict__ sc,
                                                        RefScal *__restrict__ sc_next) {
    chain_wait();
    chain_release();
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const DF *xin = xin_all + off;
    TS *r = r_all + off;
    TS *y1 = y1_all + off;
    float rr = 0.0f, bb = 0.0f;
    if (kMode == 0) {
        sweep25<DF>(
            g, bp.z0, bp.z1, [&](int k) { return xin[k]; },
            [&](int k, DF v, DF s, int nn) {
                const DF lx = df_lap(s, v, (float)nn);
                DF bk = v;
                if (scheme == 1) {
                    bk = v + df_mul(cf.half_c, lx);
                    bout_all[off + k] = bk;
                }
                float bf = df_f(bk);
                bb = fmaf(bf, bf, bb);
                float rf = df_f(df_mul_un(cf.c, lx));
                st(r, k, rf);
                st(y1, k, gamma * rf);
                rr = fmaf(rf, rf, rr);
            });
    } else {
        const TD *d = d_all + off;
        const DF *b = b_all + off;
        DF *xout = xout_all + off;
        sweep25_lf<DF>(
            g, blockIdx.x, blockIdx.y, bp.z0, bp.z1, [&](int k) { return DFd{xin[k], ld(d, k)}; },
            [](DFd v) { return df_add_f(v.x, v.d); }, [&](int k) { return b[k]; },
            [&](int k, DF v, DF s, int nn, DF bk) {
                xout[k] = v;
                const DF lx = df_lap(s, v, (float)nn);
                float rf = df_f(df_res(bk, v, cf.ce, lx));
                rr = fmaf(rf, rf, rr);
                if (kMode == 1 || kMode == 4) {
                    st(r, k, rf);
                    st(y1, k, gamma * rf);
                    if (kMode == 4) {
                        const float bf = df_f(bk);
                        bb = fmaf(bf, bf, bb);
                    }
                } else if (kMode == 2) {
                    DF cl = df_mul(cf.ce, lx);        // = theta c L v
                    DF bn = v;
                    if (scheme == 1) {
                        bn = v + cl;                  // v + c/2 L v
                        cl = cl + cl;                 // c L v
                        bout_all[off + k] = bn;
                    }
                    float bf = df_f(bn);
                    bb = fmaf(bf, bf, bb);
                    float nf_ = df_f(cl);
                    st(r, k, nf_);
                    st(y1, k, gamma * nf_);
                }
            });
    }
    constexpr bool kBB = kMode == 0 || kMode == 2 || kMode == 4;   // also reduces ||b||^2
    double vals[2] = {block_sum_f(rr), kBB ? block_sum_f(bb) : 0.0};
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, kBB ? 2 : 1, vals, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double RR = finish_sum(partials, 0, bp.nb);
        double BB = kBB ? finish_sum(partials, 1, bp.nb) : 0.0;
        if (is_thread0()) {
            sc[bp.f].rr = RR;
            if (kMode == 0 || kMode == 4) sc[bp.f].bb = BB;
            if (kMode == 2) sc_next[bp.f].bb = BB;
            sc[bp.f].ticket = 0;
        }
    }
}

// The refinement pass of k_refine_df with two x-cells per thread (nx even): a float4
// holds a cell pair's double-float values in the pair layout (hi0, hi1, lo0, lo1), and
// the pair's arithmetic is the packed DF2 form (one f32x2 instruction for both cells,
// bit-identical to the scalar form); a warp row covers 64 cells; x neighbours by shuffle
// (and the neighbouring pairs at the tile edges), y neighbours from a shared plane,
// z neighbours from a register queue.  Modes 0-2, 4 and 5 as in k_refine_df; mode 3 is one
// explicit Euler step in double-float arithmetic, xout = xin + c L xin
// (cf.c = dtau / dx^2), with no reduction.  The double-float vectors it reads and writes
// (x, b) are in the pair layout (k_to_df_pairs / k_from_df_pairs).
template <class TS> struct Pair;
template <> struct Pair<float> {
    static __device__ __forceinline__ float2 load(const float *p, int i) {
        return *reinterpret_cast<const float2 *>(p + i);
    }
    static __device__ __forceinline__ void store(float *p, size_t i, float a, float b) {
        *reinterpret_cast<float2 *>(p + i) = make_float2(a, b);
    }
};
template <> struct Pair<__nv_bfloat16> {
    static __device__ __forceinline__ float2 load(const __nv_bfloat16 *p, int i) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p + i));
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, size_t i, float a, float b) {
        *reinterpret_cast<__nv_bfloat162 *>(p + i) = __floats2bfloat162_rn(a, b);
    }
};

__device__ __forceinline__ float4 f4z() { return make_float4(0.f, 0.f, 0.f, 0.f); }
// x + d of a cell pair (pair layout in and out)
__device__ __forceinline__ float4 pair_add(float4 xv, float2 dv) { return f4_of(df2_add_f(df2_of(xv), dv)); }

// The planes ahead arrive through a per-thread cp.async ring in shared memory instead of
// registers: each thread stages its own pair's x and d two planes beyond the register
// queue, its b and its halo values beyond the next plane, and reads back only what it
// staged (no barrier).  The pass is bound by memory latency and instruction issue, not
// by its arithmetic, so deeper prefetch that costs no registers is what speeds it up.
// The march is unrolled by the ring depth: a step's ring slot is then a compile-time
// constant and the three-plane register queue rotates by renaming (the register of plane
// z-1 takes plane z+2 once the step has used it).  (One shared plane buffer per slot,
// which saves a barrier per plane, was measured slower: at 512 x 256 x 256 the larger
// shared footprint cost ~8 ms over the 80 passes of the channel case.)
constexpr int kRefRing = 3;   // ring slots: two planes in flight beyond the one consumed

template <class TS, int kMode, class TD = TS>
__global__ void __launch_bounds__(kThreads, 4) k_refine_df2(Geo g, int zlen, int nzc, CoefDF cf,
                                                         int scheme, const DF *__restrict__ xin_all,
                                                         const TD *__restrict__ d_all,
                                                         const DF *b_all, DF *__restrict__ xout_all,
                                                         DF *bout_all, TS *__restrict__ r_all,
                                                         TS *__restrict__ y1_all, float gamma,
                                                         double *__restrict__ partials_all,
                                                         RefScal *__restrict__ sc,
                                                         RefScal *__restrict__ sc_next) {
    chain_wait();
    chain_release();
    using PR = Pair<TS>;
    using PD = Pair<TD>;
    const int f = blockIdx.z / nzc;
    const int zc = blockIdx.z - f * nzc;
    const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
    const int bid = (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const int nb = gridDim.x * gridDim.y * nzc;
    const size_t off = (size_t)f * g.n;
    const float4 *X = reinterpret_cast<const float4 *>(xin_all + off);   // cell pairs
    constexpr bool kPlain = kMode == 0 || kMode == 3;   // the stencil of x itself (no d)
    const TD *D = kPlain ? nullptr : d_all + off;
    const float4 *Bp = reinterpret_cast<const float4 *>(kPlain ? nullptr : b_all + off);
    float4 *XO = reinterpret_cast<float4 *>(xout_all + off);
    float4 *BO = reinterpret_cast<float4 *>(bout_all ? bout_all + off : nullptr);
    TS *r = r_all + off;
    TS *y1 = y1_all + off;
    const DFc2 c2 = dfc2(cf.c), hc2 = dfc2(cf.half_c), ce2 = dfc2(cf.ce);
    constexpr int RS = kRefRing;
    __shared__ float4 pl[TY + 2][TX];   // the plane's tile with its y halo rows
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = blockIdx.x * (2 * TX);
    const int x = x0 + 2 * tx, y = blockIdx.y * TY + ty;
    const bool own = (x < g.nx) && (y < g.ny);
    const bool rowlo = (ty == 0) && (y > 0) && (x < g.nx);
    const bool rowhi = (ty == TY - 1) && (y + 1 < g.ny) && (x < g.nx);
    // a periodic x axis (the only periodic axis this kernel takes): the x halo cells wrap
    // and every cell has both x neighbours
    const bool px = (g.per & 1) != 0;
    const bool xl = (tx == 0) && (x > 0 || px) && (y < g.ny);
    const int xlast = min(g.nx, x0 + 2 * TX) - 2;
    const bool xr = (x == xlast) && (x + 2 < g.nx || px) && (y < g.ny);
    const int dxl = (px && x == 0) ? g.nx - 1 : -1;      // x - 1 of the pair's first cell
    const int dxr = (px && x + 2 >= g.nx) ? 2 - g.nx : 2;  // x + 1 of its second cell
    const int nyb = (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + ((x > 0 || px) ? 1 : 0) + 1, n1 = nyb + 1 + ((x + 2 < g.nx || px) ? 1 : 0);
    // the two cells' neighbour counts (and negatives) on planes with both z neighbours
    const float2 nn_mid = make_float2((float)(n0 + 2), (float)(n1 + 2));
    const float2 nnn_mid = make_float2(-nn_mid.x, -nn_mid.y);
    const int kxy = y * g.nx + x;
    // stencil value of a cell pair (pair layout) / of one cell
    auto val2 = [&](int k) -> float4 {
        const float4 xv = X[k >> 1];
        if (kPlain) return xv;
        return pair_add(xv, PD::load(D, k));
    };
    auto val1 = [&](int k) -> DF {
        const float4 pv = X[k >> 1];
        const DF xv = (k & 1) ? DF{pv.y, pv.w} : DF{pv.x, pv.z};
        if (kPlain) return xv;
        return df_add_f(xv, ld(D, k));
    };
    // d of a cell pair as stored (FP32: 8 bytes; BF16: 4 bytes); a halo column's d is
    // staged as the aligned pair that holds it (BF16 has no 2-byte asynchronous copy)
    using DPair = typename std::conditional<sizeof(TD) == 4, float2, __nv_bfloat162>::type;
    __shared__ float4 rX[RS][kThreads];    // own pair's x (plane q + 2)
    __shared__ DPair rD[RS][kThreads];     // own pair's d (plane q + 2)
    __shared__ float4 rB[RS][kThreads];    // own pair's b (plane q + 1)
    __shared__ float4 rhX[RS][2][TX];      // halo rows (plane q + 1): y - 1 (ty 0), y + 1 (ty TY-1)
    __shared__ DPair rhD[RS][2][TX];
    __shared__ float4 rcX[RS][TY][2];      // the pairs holding the halo columns (plane q + 1): x - 1, x + 2
    __shared__ typename std::conditional<sizeof(TD) == 4, float, __nv_bfloat162>::type rcD[RS][TY][2];
    auto cp_dpair = [&](void *dst, const TD *src) {
        if constexpr (sizeof(TD) == 4) cp_async8(dst, src);
        else cp_async4(dst, src);
    };
    auto dpair = [&](const DPair &v) -> float2 {
        if constexpr (sizeof(TD) == 4) return v;
        else return __bfloat1622float2(v);
    };
    const int tid = ty * TX + tx, hrow = ty == 0 ? 0 : 1;
    // the data step q reads back for step q + 1 (own x, d of plane q + 2; b and the halo of
    // plane q + 1), into ring slot sl
    auto stage = [&](int q, int sl) {
        if (q + 1 < z1) {
            const int kn = kxy + (q + 1) * g.nxy;
            if (own) {
                if (q + 2 < g.nz) {
                    cp_async16(&rX[sl][tid], X + ((kn + g.nxy) >> 1));
                    if (!kPlain) cp_dpair(&rD[sl][tid], D + kn + g.nxy);
                }
                if (!kPlain) cp_async16(&rB[sl][tid], Bp + (kn >> 1));
            }
            if (rowlo || rowhi) {
                const int kh = rowlo ? kn - g.nx : kn + g.nx;
                cp_async16(&rhX[sl][hrow][tx], X + (kh >> 1));
                if (!kPlain) cp_dpair(&rhD[sl][hrow][tx], D + kh);
            }
            // (x - 1 is the odd cell of its pair, x + 2 the even one)
            if (xl) {
                const int kl = kn + dxl;
                cp_async16(&rcX[sl][ty][0], X + (kl >> 1));
                if (!kPlain) cp_async4(&rcD[sl][ty][0], D + (sizeof(TD) == 4 ? kl : kl - 1));
            }
            if (xr) {
                const int kr = kn + dxr;
                cp_async16(&rcX[sl][ty][1], X + (kr >> 1));
                if (!kPlain) cp_async4(&rcD[sl][ty][1], D + kr);
            }
        }
        cp_async_commit();
    };
    // register state of the march: the plane queue (three registers that rotate by
    // renaming), the cell pair's b and the halo values of the current plane
    float4 qa = f4z(), qb = f4z(), qc = f4z(), bc = f4z(), hlo = f4z(), hhi = f4z();
    DF hl = DF{0.f, 0.f}, hr = DF{0.f, 0.f};
    float rr = 0.0f, bb = 0.0f;
    if (z0 < z1) {
        const int k0 = kxy + z0 * g.nxy;
        if (own) {
            if (z0 > 0) qa = val2(k0 - g.nxy);
            qb = val2(k0);
            if (z0 + 1 < g.nz) qc = val2(k0 + g.nxy);
            if (!kPlain) bc = Bp[k0 >> 1];
        }
        if (rowlo) hlo = val2(k0 - g.nx);
        if (rowhi) hhi = val2(k0 + g.nx);
        if (xl) hl = val1(k0 + dxl);
        if (xr) hr = val1(k0 + dxr);
    }
    stage(z0, 0);
    stage(z0 + 1, 1);
    // one plane: vdn, vc, vup = planes z - 1, z, z + 1; j = (z - z0) % 3 (its ring slot).
    // After the stencil vdn takes plane z + 2 from the ring.
    auto step = [&](const int z, const int j, float4 &vdn, const float4 &vc, const float4 &vup) {
        stage(z + RS - 1, (j + RS - 1) % RS);     // into the slot step z - 1 read
        const int kz = kxy + z * g.nxy;
        pl[ty + 1][tx] = vc;
        if (ty == 0) pl[0][tx] = hlo;
        if (ty == TY - 1) pl[TY + 1][tx] = hhi;
        // cell x - 1 is the second cell of the pair to the left, x + 2 the first of the
        // pair to the right
        DF left{__shfl_up_sync(0xffffffffu, vc.y, 1), __shfl_up_sync(0xffffffffu, vc.w, 1)};
        DF right{__shfl_down_sync(0xffffffffu, vc.x, 1), __shfl_down_sync(0xffffffffu, vc.z, 1)};
        if (tx == 0) left = hl;
        if (x == xlast) right = hr;
        __syncthreads();
        if (own) {
            const DF2 V = df2_of(vc);
            float2 nn = nn_mid, nnn = nnn_mid;
            if (z == 0 || z + 1 == g.nz) {   // a z wall: fewer neighbours
                const int nz_ = (z > 0) + (z + 1 < g.nz);
                nn = make_float2((float)(n0 + nz_), (float)(n1 + nz_));
                nnn = make_float2(-nn.x, -nn.y);
            }
            // each cell's neighbour sum in the order x - 1, x + 1, y - 1, y + 1, z - 1, z + 1
            DF2 S{make_float2(left.hi, vc.x), make_float2(left.lo, vc.z)};
            df2_acc(S, DF2{make_float2(vc.y, right.hi), make_float2(vc.w, right.lo)});
            df2_acc(S, df2_of(pl[ty][tx]));
            df2_acc(S, df2_of(pl[ty + 2][tx]));
            df2_acc(S, df2_of(vdn));
            df2_acc(S, df2_of(vup));
            const DF2 L = df2_lap(S, V, nn, nnn);
            if (kMode == 3) {   // one explicit Euler step: x + c L x
                XO[kz >> 1] = f4_of(df2_add(V, df2_mul(c2, L)));
            } else if (kMode == 0) {
                const float2 rf = df2_f(df2_mul_un(c2, L));
                DF2 B = V;
                if (scheme == 1) {
                    B = df2_add(V, df2_mul(hc2, L));
                    BO[kz >> 1] = f4_of(B);
                }
                const float2 fb = df2_f(B);
                bb = fmaf(fb.x, fb.x, fmaf(fb.y, fb.y, bb));
                rr = fmaf(rf.x, rf.x, fmaf(rf.y, rf.y, rr));
                PR::store(r, kz, rf.x, rf.y);
                const float2 g1 = mul2(make_float2(gamma, gamma), rf);
                PR::store(y1, kz, g1.x, g1.y);
            } else {
                XO[kz >> 1] = vc;
                const float2 rf = df2_f(df2_res(df2_of(bc), V, ce2, L));
                rr = fmaf(rf.x, rf.x, fmaf(rf.y, rf.y, rr));
                if (kMode == 1 || kMode == 4) {
                    PR::store(r, kz, rf.x, rf.y);
                    const float2 g1 = mul2(make_float2(gamma, gamma), rf);
                    PR::store(y1, kz, g1.x, g1.y);
                    if (kMode == 4) {
                        const float2 fb = df2_f(df2_of(bc));
                        bb = fmaf(fb.x, fb.x, fmaf(fb.y, fb.y, bb));
                    }
                } else if (kMode == 2) {
                    DF2 C = df2_mul(ce2, L);   // theta c L v
                    DF2 Bn = V;
                    if (scheme == 1) {
                        Bn = df2_add(V, C);      // v + c/2 L v
                        C = df2_add(C, C);       // c L v
                        BO[kz >> 1] = f4_of(Bn);
                    }
                    const float2 fb = df2_f(Bn);
                    bb = fmaf(fb.x, fb.x, fmaf(fb.y, fb.y, bb));
                    const float2 q = df2_f(C);
                    PR::store(r, kz, q.x, q.y);
                    const float2 g1 = mul2(make_float2(gamma, gamma), q);
                    PR::store(y1, kz, g1.x, g1.y);
                }
            }
        }
        __syncthreads();   // the plane buffer is rewritten by the next step
        // the next step's planes, staged two steps ago (slot j)
        cp_async_wait<RS - 1>();
        if (z + 1 < z1) {
            if (own) {
                vdn = f4z();
                if (z + 2 < g.nz) {
                    const float4 xv = rX[j][tid];
                    vdn = kPlain ? xv : pair_add(xv, dpair(rD[j][tid]));
                }
                if (!kPlain) bc = rB[j][tid];
            }
            if (rowlo || rowhi) {
                const float4 xv = rhX[j][hrow][tx];
                const float4 hv = kPlain ? xv : pair_add(xv, dpair(rhD[j][hrow][tx]));
                if (rowlo) hlo = hv;
                else hhi = hv;
            }
            if (xl) {
                const float4 pv = rcX[j][ty][0];
                const DF xv{pv.y, pv.w};
                if constexpr (sizeof(TD) == 4)
                    hl = kPlain ? xv : df_add_f(xv, rcD[j][ty][0]);
                else
                    hl = kPlain ? xv : df_add_f(xv, __high2float(rcD[j][ty][0]));
            }
            if (xr) {
                const float4 pv = rcX[j][ty][1];
                const DF xv{pv.x, pv.z};
                if constexpr (sizeof(TD) == 4)
                    hr = kPlain ? xv : df_add_f(xv, rcD[j][ty][1]);
                else
                    hr = kPlain ? xv : df_add_f(xv, __low2float(rcD[j][ty][1]));
            }
        }
    };
    static_assert(RS == 3, "the march below is unrolled for three ring slots");
    for (int z = z0; z < z1; z += RS) {
        step(z, 0, qa, qb, qc);
        if (z + 1 < z1) step(z + 1, 1, qb, qc, qa);
        if (z + 2 < z1) step(z + 2, 2, qc, qa, qb);
    }
    cp_async_wait<0>();   // no copy outlives the block
    if (kMode == 3) return;   // the explicit step reduces nothing
    constexpr bool kBB = kMode == 0 || kMode == 2 || kMode == 4;   // also reduces ||b||^2
    double vals[2] = {block_sum_f(rr), kBB ? block_sum_f(bb) : 0.0};
    double *partials = partials_all + (size_t)f * 2 * nb;
    if (arrive(partials, kBB ? 2 : 1, vals, bid, nb, &sc[f].ticket)) {
        double RR = finish_sum(partials, 0, nb);
        double BB = kBB ? finish_sum(partials, 1, nb) : 0.0;
        if (is_thread0()) {
            sc[f].rr = RR;
            if (kMode == 0 || kMode == 4) sc[f].bb = BB;
            if (kMode == 2) sc_next[f].bb = BB;
            sc[f].ticket = 0;
        }
    }
}

// ---------------------------------------------------------------- merged step pass
// With the shared expansion a step ends with x = (u_s + e_s) + d (e_s its increment, d its
// round's correction; u_{s+1} = x) and the next one starts from u_{s+1} + e_{s+1}: two
// passes that read the same cells one after the other.  Here they are one: per cell and
// neighbour the pass forms x and takes e' = e_{s+1}, and from the two neighbour sums it has
// both the finished step's residual b - A x (reduced) and the next step's first one,
//   r' = b' - A (x + e') = theta ce L x - e' + ce L e',
// b' = x (implicit Euler, theta = 1) or x + ce L x (Crank-Nicolson, theta = 2), all in
// double-float arithmetic (e' is exact in FP32).  36 B per cell instead of 60 for the two
// (x + e' is never stored), one launch instead of two; bound by instruction issue and
// latency like k_refine_df2.  Per step (one merged pass for two): 128^3 53.5 -> 32.9 us,
// 256 x 128 x 128 x 4 fields 276 -> 193 us, 512 x 256 x 256 520 -> 352 us (3.4 TB/s), and in the scalar
// form 97 x 61 x 45 x 3 fields 47 -> 37 us.  kEnd: the last step's pass, without a next step.
// the value pair of the scalar form: += is the double-float cascade on both parts
struct DFe {
    DF x, e;
};
__device__ __forceinline__ DFe &operator+=(DFe &a, DFe b) {
    a.x += b.x;
    a.e += b.e;
    return a;
}
struct DFeRaw {
    DF u;
    float e, d, en;
};

template <bool kEnd>
__global__ void __launch_bounds__(kThreads) k_refine_mid(Geo g, int zlen, int nzc, CoefDF cf, int scheme,
                                                         const DF *__restrict__ u_all,
                                                         const float *__restrict__ e_all,
                                                         const float *__restrict__ d_all,
                                                         const float *__restrict__ en_all, const DF *b_all,
                                                         DF *__restrict__ xout_all, DF *bout_all,
                                                         float *__restrict__ r_all, float *__restrict__ y1_all,
                                                         float gamma, double *__restrict__ partials_all,
                                                         RefScal *__restrict__ sc, RefScal *__restrict__ sc_next) {
    chain_wait();
    chain_release();
    const BlockPos bp = block_pos(g, zlen, nzc);
    const size_t off = (size_t)bp.f * g.n;
    const DF *u = u_all + off, *b = b_all + off;
    const float *e = e_all + off, *d = d_all + off, *en = kEnd ? nullptr : en_all + off;
    DF *xout = xout_all + off;
    float *r = r_all + off, *y1 = y1_all + off;
    float rr = 0.0f, bb = 0.0f;
    sweep25_lf<DFe>(
        g, blockIdx.x, blockIdx.y, bp.z0, bp.z1,
        [&](int k) { return DFeRaw{u[k], e[k], d[k], kEnd ? 0.0f : en[k]}; },
        [](DFeRaw v) { return DFe{df_add_f(df_add_f(v.u, v.e), v.d), DF{v.en, 0.0f}}; },
        [&](int k) { return b[k]; },
        [&](int k, DFe v, DFe s, int nn, DF bk) {
            xout[k] = v.x;
            const DF lx = df_lap(s.x, v.x, (float)nn);
            const float rf = df_f(df_res(bk, v.x, cf.ce, lx));
            rr = fmaf(rf, rf, rr);
            if constexpr (!kEnd) {
                const DF le = df_lap(s.e, v.e, (float)nn);
                DF bn = v.x, m = lx;
                if (scheme == 1) {
                    bn = v.x + df_mul(cf.ce, lx);
                    bout_all[off + k] = bn;
                    m = DF{2.0f * lx.hi, 2.0f * lx.lo};
                }
                const float bf = df_f(bn);
                bb = fmaf(bf, bf, bb);
                const DF t = df_two_sum(m.hi, le.hi);
                const DF q = df_mul_un(cf.ce, DF{t.hi, (m.lo + le.lo) + t.lo});
                const DF w = df_two_sum(-v.e.hi, q.hi);
                const float rn = w.hi + (q.lo + w.lo);
                r[k] = rn;
                y1[k] = gamma * rn;
            }
        });
    double vals[2] = {block_sum_f(rr), kEnd ? 0.0 : block_sum_f(bb)};
    double *partials = partials_all + (size_t)bp.f * 2 * bp.nb;
    if (arrive(partials, kEnd ? 1 : 2, vals, bp.bid, bp.nb, &sc[bp.f].ticket)) {
        double RR = finish_sum(partials, 0, bp.nb);
        double BB = kEnd ? 0.0 : finish_sum(partials, 1, bp.nb);
        if (is_thread0()) {
            sc[bp.f].rr = RR;
            if (!kEnd) sc_next[bp.f].bb = BB;
            sc[bp.f].ticket = 0;
        }
    }
}

// The same pass with two x-cells per thread in packed arithmetic, implicit Euler, built as
// k_refine_df2: the planes ahead come through a per-thread cp.async ring, the march is
// unrolled by its three slots.  The finished step's b is u_s, which the x of a cell is
// formed from: it stays in registers from when its plane arrives until it is the centre.
template <bool kEnd>
__global__ void __launch_bounds__(kThreads, 3) k_refine_mid2(Geo g, int zlen, int nzc, CoefDF cf,
                                                          const DF *__restrict__ u_all,
                                                          const float *__restrict__ e_all,
                                                          const float *__restrict__ d_all,
                                                          const float *__restrict__ en_all,
                                                          DF *__restrict__ xout_all, float *__restrict__ r_all,
                                                          float *__restrict__ y1_all, float gamma,
                                                          double *__restrict__ partials_all,
                                                          RefScal *__restrict__ sc, RefScal *__restrict__ sc_next) {
    chain_wait();
    chain_release();
    using PR = Pair<float>;
    constexpr int RS = kRefRing;
    const int f = blockIdx.z / nzc;
    const int zc = blockIdx.z - f * nzc;
    const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
    const int bid = (zc * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    const int nb = gridDim.x * gridDim.y * nzc;
    const size_t off = (size_t)f * g.n;
    const float4 *U = reinterpret_cast<const float4 *>(u_all + off);   // cell pairs
    const float *E = e_all + off, *D = d_all + off, *F = kEnd ? nullptr : en_all + off;
    float4 *XO = reinterpret_cast<float4 *>(xout_all + off);
    float *r = r_all + off, *y1 = y1_all + off;
    const DFc2 ce2 = dfc2(cf.ce);
    __shared__ float4 pl[TY + 2][TX];   // the plane's x with its y halo rows
    __shared__ float2 pf[kEnd ? 1 : TY + 2][TX];   // and its e'
    __shared__ float4 rU[RS][kThreads];    // own pair (plane q + 2): u, e, d, e'
    __shared__ float2 rE[RS][kThreads], rD[RS][kThreads], rF[kEnd ? 1 : RS][kEnd ? 1 : kThreads];
    __shared__ float4 rhU[RS][2][TX];      // halo rows (plane q + 1)
    __shared__ float2 rhE[RS][2][TX], rhD[RS][2][TX], rhF[kEnd ? 1 : RS][2][TX];
    __shared__ float4 rcU[RS][TY][2];      // halo columns (plane q + 1): the pairs holding x - 1, x + 2
    __shared__ float rcE[RS][TY][2], rcD[RS][TY][2], rcF[kEnd ? 1 : RS][TY][2];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = blockIdx.x * (2 * TX);
    const int x = x0 + 2 * tx, y = blockIdx.y * TY + ty;
    const bool own = (x < g.nx) && (y < g.ny);
    const bool rowlo = (ty == 0) && (y > 0) && (x < g.nx);
    const bool rowhi = (ty == TY - 1) && (y + 1 < g.ny) && (x < g.nx);
    const bool row = rowlo || rowhi;
    const bool px = (g.per & 1) != 0;   // a periodic x axis (the only one this kernel takes)
    const bool xl = (tx == 0) && (x > 0 || px) && (y < g.ny);
    const int xlast = min(g.nx, x0 + 2 * TX) - 2;
    const bool xr = (x == xlast) && (x + 2 < g.nx || px) && (y < g.ny);
    const int dxl = (px && x == 0) ? g.nx - 1 : -1;
    const int dxr = (px && x + 2 >= g.nx) ? 2 - g.nx : 2;
    const int dro = rowlo ? -g.nx : g.nx;
    const int nyb = (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + ((x > 0 || px) ? 1 : 0) + 1, n1 = nyb + 1 + ((x + 2 < g.nx || px) ? 1 : 0);
    const float2 nn_mid = make_float2((float)(n0 + 2), (float)(n1 + 2));
    const int kxy = y * g.nx + x;
    auto value = [](float4 u, float2 e, float2 d) { return pair_add(pair_add(u, e), d); };
    auto value1 = [](float4 p, bool odd, float e, float d) {   // one cell of a pair
        return df_add_f(df_add_f(odd ? DF{p.y, p.w} : DF{p.x, p.z}, e), d);
    };
    const float2 z2 = make_float2(0.f, 0.f);
    const int tid = ty * TX + tx, hrow = ty == 0 ? 0 : 1;
    auto stage = [&](int q, int sl) {
        if (q + 1 < z1) {
            const int kn = kxy + (q + 1) * g.nxy;
            if (own && q + 2 < g.nz) {
                const int k2 = kn + g.nxy;
                cp_async16(&rU[sl][tid], U + (k2 >> 1));
                cp_async8(&rE[sl][tid], E + k2);
                cp_async8(&rD[sl][tid], D + k2);
                if constexpr (!kEnd) cp_async8(&rF[sl][tid], F + k2);
            }
            if (row) {
                const int kh = kn + dro;
                cp_async16(&rhU[sl][hrow][tx], U + (kh >> 1));
                cp_async8(&rhE[sl][hrow][tx], E + kh);
                cp_async8(&rhD[sl][hrow][tx], D + kh);
                if constexpr (!kEnd) cp_async8(&rhF[sl][hrow][tx], F + kh);
            }
            if (xl) {
                const int kl = kn + dxl;
                cp_async16(&rcU[sl][ty][0], U + (kl >> 1));
                cp_async4(&rcE[sl][ty][0], E + kl);
                cp_async4(&rcD[sl][ty][0], D + kl);
                if constexpr (!kEnd) cp_async4(&rcF[sl][ty][0], F + kl);
            }
            if (xr) {
                const int kr = kn + dxr;
                cp_async16(&rcU[sl][ty][1], U + (kr >> 1));
                cp_async4(&rcE[sl][ty][1], E + kr);
                cp_async4(&rcD[sl][ty][1], D + kr);
                if constexpr (!kEnd) cp_async4(&rcF[sl][ty][1], F + kr);
            }
        }
        cp_async_commit();
    };
    // register state: the plane queues (rotating by renaming), u of planes z and z + 1, the
    // halo values of plane z
    float4 qa = f4z(), qb = f4z(), qc = f4z(), bc = f4z(), bn = f4z(), hv = f4z();
    float2 fa = z2, fb = z2, fc = z2, hf = z2;
    DF hl{0.f, 0.f}, hr{0.f, 0.f};
    float hfl = 0.f, hfr = 0.f;
    float rr = 0.0f, bb = 0.0f;
    if (z0 < z1) {
        const int k0 = kxy + z0 * g.nxy;
        auto at = [&](int k) { return value(U[k >> 1], PR::load(E, k), PR::load(D, k)); };
        auto at1 = [&](int k) { return value1(U[k >> 1], k & 1, E[k], D[k]); };
        if (own) {
            if (z0 > 0) {
                qa = at(k0 - g.nxy);
                if constexpr (!kEnd) fa = PR::load(F, k0 - g.nxy);
            }
            qb = at(k0);
            bc = U[k0 >> 1];
            if constexpr (!kEnd) fb = PR::load(F, k0);
            if (z0 + 1 < g.nz) {
                qc = at(k0 + g.nxy);
                bn = U[(k0 + g.nxy) >> 1];
                if constexpr (!kEnd) fc = PR::load(F, k0 + g.nxy);
            }
        }
        if (row) {
            hv = at(k0 + dro);
            if constexpr (!kEnd) hf = PR::load(F, k0 + dro);
        }
        if (xl) {
            hl = at1(k0 + dxl);
            if constexpr (!kEnd) hfl = F[k0 + dxl];
        }
        if (xr) {
            hr = at1(k0 + dxr);
            if constexpr (!kEnd) hfr = F[k0 + dxr];
        }
    }
    stage(z0, 0);
    stage(z0 + 1, 1);
    // one plane: planes z - 1, z, z + 1 of x (vdn, vc, vup) and e' (gdn, gc, gup);
    // j = (z - z0) % 3.  After the stencils vdn and gdn take plane z + 2.
    auto step = [&](const int z, const int j, float4 &vdn, const float4 &vc, const float4 &vup, float2 &gdn,
                    const float2 &gc, const float2 &gup) {
        stage(z + RS - 1, (j + RS - 1) % RS);
        const int kz = kxy + z * g.nxy;
        pl[ty + 1][tx] = vc;
        if constexpr (!kEnd) pf[ty + 1][tx] = gc;
        if (ty == 0 || ty == TY - 1) {   // (zero where the row lies outside the mesh)
            const int hr_ = ty == 0 ? 0 : TY + 1;
            pl[hr_][tx] = hv;
            if constexpr (!kEnd) pf[hr_][tx] = hf;
        }
        DF left{__shfl_up_sync(0xffffffffu, vc.y, 1), __shfl_up_sync(0xffffffffu, vc.w, 1)};
        DF right{__shfl_down_sync(0xffffffffu, vc.x, 1), __shfl_down_sync(0xffffffffu, vc.z, 1)};
        float fl = 0.f, fr = 0.f;
        if constexpr (!kEnd) {
            fl = __shfl_up_sync(0xffffffffu, gc.y, 1);
            fr = __shfl_down_sync(0xffffffffu, gc.x, 1);
        }
        if (tx == 0) {
            left = hl;
            fl = hfl;
        }
        if (x == xlast) {
            right = hr;
            fr = hfr;
        }
        __syncthreads();
        if (own) {
            const DF2 V = df2_of(vc);
            float2 nn = nn_mid;
            if (z == 0 || z + 1 == g.nz) {   // a z wall: fewer neighbours
                const int nz_ = (z > 0) + (z + 1 < g.nz);
                nn = make_float2((float)(n0 + nz_), (float)(n1 + nz_));
            }
            const float2 nnn = make_float2(-nn.x, -nn.y);
            DF2 S{make_float2(left.hi, vc.x), make_float2(left.lo, vc.z)};
            df2_acc(S, DF2{make_float2(vc.y, right.hi), make_float2(vc.w, right.lo)});
            df2_acc(S, df2_of(pl[ty][tx]));
            df2_acc(S, df2_of(pl[ty + 2][tx]));
            df2_acc(S, df2_of(vdn));
            df2_acc(S, df2_of(vup));
            const DF2 L = df2_lap(S, V, nn, nnn);
            XO[kz >> 1] = vc;
            const float2 rf = df2_f(df2_res(df2_of(bc), V, ce2, L));
            rr = fmaf(rf.x, rf.x, fmaf(rf.y, rf.y, rr));
            if constexpr (!kEnd) {
                // the neighbour sum of e' as a pair: the TwoSum cascade's errors
                DF2 G{make_float2(fl, gc.x), z2};
                auto acc = [&](float2 v) {
                    const DF2 t = df2_two_sum(G.hi, v);
                    G.hi = t.hi;
                    G.lo = add2(G.lo, t.lo);
                };
                acc(make_float2(gc.y, fr));
                acc(pf[ty][tx]);
                acc(pf[ty + 2][tx]);
                acc(gdn);
                acc(gup);
                const DF2 LE = df2_lap(G, DF2{gc, z2}, nn, nnn);
                const DF2 t = df2_two_sum(L.hi, LE.hi);
                const DF2n q = df2_mul_un(ce2, DF2{t.hi, add2(add2(L.lo, LE.lo), t.lo)});
                const DF2 w = df2_two_sum(q.hi, make_float2(-gc.x, -gc.y));
                const float2 rn = add2(w.hi, sub2(w.lo, q.nlo));
                const float2 fb2 = df2_f(V);
                bb = fmaf(fb2.x, fb2.x, fmaf(fb2.y, fb2.y, bb));
                PR::store(r, kz, rn.x, rn.y);
                const float2 g1 = mul2(make_float2(gamma, gamma), rn);
                PR::store(y1, kz, g1.x, g1.y);
            }
        }
        __syncthreads();   // the plane buffers are rewritten by the next step
        cp_async_wait<RS - 1>();
        if (z + 1 < z1) {
            if (own) {
                bc = bn;
                vdn = f4z();
                gdn = z2;
                if (z + 2 < g.nz) {
                    bn = rU[j][tid];
                    vdn = value(bn, rE[j][tid], rD[j][tid]);
                    if constexpr (!kEnd) gdn = rF[j][tid];
                }
            }
            if (row) {
                hv = value(rhU[j][hrow][tx], rhE[j][hrow][tx], rhD[j][hrow][tx]);
                if constexpr (!kEnd) hf = rhF[j][hrow][tx];
            }
            if (xl) {   // x - 1 is the odd cell of its pair, x + 2 the even one
                hl = value1(rcU[j][ty][0], true, rcE[j][ty][0], rcD[j][ty][0]);
                if constexpr (!kEnd) hfl = rcF[j][ty][0];
            }
            if (xr) {
                hr = value1(rcU[j][ty][1], false, rcE[j][ty][1], rcD[j][ty][1]);
                if constexpr (!kEnd) hfr = rcF[j][ty][1];
            }
        }
    };
    static_assert(RS == 3, "the march below is unrolled for three ring slots");
    for (int z = z0; z < z1; z += RS) {
        step(z, 0, qa, qb, qc, fa, fb, fc);
        if (z + 1 < z1) step(z + 1, 1, qb, qc, qa, fb, fc, fa);
        if (z + 2 < z1) step(z + 2, 2, qc, qa, qb, fc, fa, fb);
    }
    cp_async_wait<0>();   // no copy outlives the block
    double vals[2] = {block_sum_f(rr), kEnd ? 0.0 : block_sum_f(bb)};
    double *partials = partials_all + (size_t)f * 2 * nb;
    if (arrive(partials, kEnd ? 1 : 2, vals, bid, nb, &sc[f].ticket)) {
        double RR = finish_sum(partials, 0, nb);
        double BB = kEnd ? 0.0 : finish_sum(partials, 1, nb);
        if (is_thread0()) {
            sc[f].rr = RR;
            if (!kEnd) sc_next[f].bb = BB;
            sc[f].ticket = 0;
        }
    }
}

// ---------------------------------------------------------------- grid barrier
// A barrier over all blocks of a cooperative launch (all blocks co-resident).  The
// wait is bounded: a block that spins longer than `budget` clock cycles raises err and
// every block gives up at its next barrier, so the kernel always ends; the host then
// reports CG_ETIMEOUT.
struct GridBar {
    unsigned int count;
    unsigned int gen;
    int err;
    int pad;
};

__device__ __forceinline__ bool grid_sync(GridBar *gb, unsigned nblocks, long long budget) {
    __shared__ int s_ok;
    __syncthreads();
    if (is_thread0()) {
        volatile unsigned int *vgen = &gb->gen;
        volatile int *verr = &gb->err;
        const unsigned int g0 = *vgen;
        __threadfence();
        int ok = 1;
        const unsigned int arrived = atomicAdd(&gb->count, 1u);
        if (arrived == nblocks - 1) {
            gb->count = 0;
            __threadfence();
            atomicAdd(&gb->gen, 1u);
        } else {
            const long long t0 = clock64();
            while (*vgen == g0) {
                if (*verr) { ok = 0; break; }
                if (clock64() - t0 > budget) {
                    atomicExch(&gb->err, 1);
                    ok = 0;
                    break;
                }
                __nanosleep(32);
            }
        }
        __threadfence();
        if (*verr) ok = 0;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// The whole inner Chebyshev solve of one refinement round in one cooperative launch.
// Chebyshev iteration for A y = r on the spectrum [1, lmax] (theta, delta its centre
// and half-width, sigma = theta/delta, gamma = 1/theta): y_1 = gamma r, and
// y_{k+1} = omega_k (y_k - y_{k-1} + gamma (r - A y_k)) + y_{k-1} with omega_1 =
// 1/(1 - 1/(2 sigma^2)), omega_k = 1/(1 - omega_{k-1}/(4 sigma^2)); FP32 arithmetic,
// TS storage, y_{k+1} written over y_{k-1}.  Iterations k = 1 .. m-1, each a pass over every work
// item (xy tile x z-chunk x field) with a grid barrier between iterations.  y1 holds
// gamma r on entry; the result is left where the host-side rotation says.
template <class TS>
__global__ void __launch_bounds__(kThreads) k_cheb_loop(Geo g, int zlen, int nzc, int gx, int gy,
                                                        int nitems, Coef32 cf, float gamma,
                                                        double sigma, int m, TS *y1,
                                                        TS *yother, const TS *__restrict__ r_all,
                                                        GridBar *gb, long long budget) {
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    __syncthreads();
    TS *ycur = y1, *yprev = nullptr;
    double om = 1.0;
    for (int k = 1; k < m; ++k) {
        if (sigma > 0.0) {
            om = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma * sigma))
                          : 1.0 / (1.0 - om / (4.0 * sigma * sigma));
        }
        const float omega = (float)om;
        TS *ynext = yprev ? yprev : yother;
        for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
            int t = it;
            const int bx = t % gx;
            t /= gx;
            const int by = t % gy;
            t /= gy;
            const int zc = t % nzc;
            const int f = t / nzc;
            const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
            const size_t off = (size_t)f * g.n;
            const TS *y = ycur + off;
            const TS *r = r_all + off;
            const TS *yp = yprev ? yprev + off : nullptr;
            TS *yn = ynext + off;
            sweep25_at<float>(
                g, bx, by, z0, z1, [&](int q) { return ldcg(y, q); },
                [&](int q) { return float2{yp ? ldcg(yp, q) : 0.0f, ld(r, q)}; },
                [&](int q, float v, float s, int nn, float2 pt) {
                    float ay = fmaf(sdg[nn], v, -cf.ce * s);
                    st(yn, q, fmaf(omega, v - pt.x + gamma * (pt.y - ay), pt.x));
                });
        }
        yprev = ycur;
        ycur = ynext;
        if (k + 1 < m && !grid_sync(gb, gridDim.x, budget)) return;
    }
}

// The Chebyshev iteration of k_cheb on the register-blocked engine: blockIdx.z =
// f * nzb + z-block, ZB planes per block.
template <int ZB, class TS>
__global__ void __launch_bounds__(kThreads) k_cheb_zb(Geo g, int nzb, Coef32 cf, float gamma,
                                                      float omega, const TS *__restrict__ y_all,
                                                      const TS *yprev_all,
                                                      const TS *__restrict__ r_all, TS *ynext_all) {
    chain_wait();
    chain_release();
    const int f = blockIdx.z / nzb;
    const int z0 = (blockIdx.z - f * nzb) * ZB;
    const size_t off = (size_t)f * g.n;
    const TS *y = y_all + off;
    const TS *r = r_all + off;
    const TS *yp = yprev_all ? yprev_all + off : nullptr;
    TS *yn = ynext_all + off;
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    sweepzb<ZB, float>(
        g, blockIdx.x, blockIdx.y, z0, [&](int k) { return ld(y, k); },
        [&](int k) { return float2{yp ? ld(yp, k) : 0.0f, ld(r, k)}; },
        [&](int k, float v, float s, int nn, float2 pt) {
            float ay = fmaf(sdg[nn], v, -cf.ce * s);
            st(yn, k, fmaf(omega, v - pt.x + gamma * (pt.y - ay), pt.x));
        });
}

// ---------------------------------------------------------------- vectorised sweep
// The Chebyshev iteration with four consecutive x-cells per thread (nx % 4 == 0): a
// warp row covers 128 cells with 128-bit loads and stores (64-bit for BF16), the x
// neighbours inside a thread's four cells are in registers, across threads they come
// by warp shuffle and across tiles from two scalar loads; y neighbours come from a
// shared plane of the tile (rows y0-1 .. y0+8), z neighbours from a register queue.
// Loads for plane z+1 are issued while plane z is computed.  A wall contributes nothing
// and is not counted (zero flux).
template <class TS> struct Vec4;
template <> struct Vec4<float> {
    static __device__ __forceinline__ float4 load(const float *p, int i) {
        return *reinterpret_cast<const float4 *>(p + i);
    }
    static __device__ __forceinline__ void store(float *p, size_t i, float4 v) {
        *reinterpret_cast<float4 *>(p + i) = v;
    }
};
template <> struct Vec4<__nv_bfloat16> {
    static __device__ __forceinline__ float4 load(const __nv_bfloat16 *p, int i) {
        uint2 u = *reinterpret_cast<const uint2 *>(p + i);
        __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&u.x);
        __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162 *>(&u.y);
        float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
        return make_float4(fa.x, fa.y, fb.x, fb.y);
    }
    static __device__ __forceinline__ void store(__nv_bfloat16 *p, size_t i, float4 v) {
        __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
        __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
        uint2 u;
        u.x = *reinterpret_cast<unsigned *>(&a);
        u.y = *reinterpret_cast<unsigned *>(&b);
        *reinterpret_cast<uint2 *>(p + i) = u;
    }
};

__device__ __forceinline__ float4 f4zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// L2-coherent variants of the vector loads, for data written by other blocks of the
// same (persistent) launch.
template <class TS> struct Vec4cg;
template <> struct Vec4cg<float> {
    static __device__ __forceinline__ float4 load(const float *p, int i) {
        return __ldcg(reinterpret_cast<const float4 *>(p + i));
    }
};
template <> struct Vec4cg<__nv_bfloat16> {
    static __device__ __forceinline__ float4 load(const __nv_bfloat16 *p, int i) {
        uint2 u = __ldcg(reinterpret_cast<const uint2 *>(p + i));
        __nv_bfloat162 a = *reinterpret_cast<__nv_bfloat162 *>(&u.x);
        __nv_bfloat162 b = *reinterpret_cast<__nv_bfloat162 *>(&u.y);
        float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
        return make_float4(fa.x, fa.y, fb.x, fb.y);
    }
};

// One tile (128 x-cells x TY rows x planes [z0, z1)) of the vectorised Chebyshev
// iteration; L is the load policy (Vec4 or Vec4cg), sdg the diagonal table in shared
// memory.  Offsets within a field are 32-bit (a field has fewer than 2^31 cells).  Every thread of the block must call it (barriers and shuffles inside).
// ZFIX > 0: the caller guarantees at most ZFIX planes per block, so the march is
// unrolled (the register queue rotates without copies).  PER: periodic axes (g.per):
// halo rows, columns and planes wrap, every cell has both neighbours on a periodic
// axis, and the tile's rows beyond ny hold the wrapped rows (y mod ny) as neighbours.
template <class TS, template <class> class L, int ZFIX = 0, bool PER = false, bool PRED = false>
__device__ __forceinline__ void cheb_v4_tile(const Geo &g, int bx, int by, int z0, int z1,
                                             const Coef32 &cf, const float *sdg, float gamma,
                                             float omega, const TS *yv, const TS *ypv,
                                             const TS *rv, TS *ynv) {
    using V = Vec4<TS>;
    using LD = L<TS>;
    __shared__ float4 pl[TY + 2][TX];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x0 = bx * (4 * TX);
    const int x = x0 + 4 * tx, y = by * TY + ty;
    const bool px = PER && (g.per & 1), py = PER && (g.per & 2), pz = PER && (g.per & 4);
    const bool own = (x < g.nx) && (y < g.ny);
    const int yw = py ? y % g.ny : y;                                    // the row this thread holds
    const bool hold = (x < g.nx) && (yw < g.ny);                         // holds a mesh row (own or wrapped)
    const bool rowlo = (ty == 0) && (y > 0 || py) && (x < g.nx);         // loads row y-1
    const bool rowhi = (ty == TY - 1) && (y + 1 < g.ny || py) && (x < g.nx);  // loads row y+1
    const bool xl = (tx == 0) && (x > 0 || px) && (yw < g.ny);           // cell x-1
    const int xlast = min(g.nx, x0 + 4 * TX) - 4;                       // first cell of the last owned vector
    const bool xr = (x == xlast) && (x + 4 < g.nx || px) && (yw < g.ny);  // cell x+4
    // neighbour counts in x and y of the four cells (z added per plane)
    const int nyb = py ? 2 : (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + (px ? 1 : (x > 0)) + 1, n3 = nyb + 1 + (px ? 1 : (x + 4 < g.nx));
    const int n12 = nyb + 2;
    // diagonals of the four cells on planes with both z neighbours (most planes)
    const float d0i = sdg[n0 + 2], d12i = sdg[n12 + 2], d3i = sdg[n3 + 2];
    const int kxy = yw * g.nx + x;
    // neighbour offsets within a plane (wrapped across a periodic face)
    const int dlo = (PER && yw == 0) ? (g.ny - 1) * g.nx : -g.nx;
    const int dhi = (PER && yw == g.ny - 1) ? -(g.ny - 1) * g.nx : g.nx;
    const int dxl = (PER && x == 0) ? g.nx - 1 : -1;
    const int dxr = (PER && x + 4 >= g.nx) ? 4 - g.nx : 4;
    // plane index of plane q of the z march (wrapped on a periodic z axis)
    auto zp = [&](int q) -> int { return (pz ? (q + g.nz) % g.nz : q) * g.nxy; };
    float4 vdn = f4zero(), vc = f4zero(), vup = f4zero(), ypc = f4zero(), rc = f4zero();
    float4 hlo = f4zero(), hhi = f4zero();
    float hl = 0.f, hr = 0.f;
    if (z0 < z1) {
        const int k0 = kxy + zp(z0);
        if (hold) {
            if (z0 > 0 || pz) vdn = LD::load(yv, kxy + zp(z0 - 1));
            vc = LD::load(yv, k0);
            if (z0 + 1 < g.nz || pz) vup = LD::load(yv, kxy + zp(z0 + 1));
        }
        if (own) {
            if (ypv) ypc = LD::load(ypv, k0);
            if constexpr (!PRED) rc = LD::load(rv, k0);
        }
        if (rowlo) hlo = LD::load(yv, k0 + dlo);
        if (rowhi) hhi = LD::load(yv, k0 + dhi);
        if (xl) hl = ldcg(yv, k0 + dxl);
        if (xr) hr = ldcg(yv, k0 + dxr);
    }
#pragma unroll
    for (int zi = 0; zi < (ZFIX > 0 ? ZFIX : z1 - z0); ++zi) {
        const int z = z0 + zi;
        if (ZFIX > 0 && z >= z1) break;
        const int kz = kxy + (PER ? zp(z) : z * g.nxy);
        // loads for the next plane
        float4 nup = f4zero(), nyp = f4zero(), nr = f4zero(), nlo = f4zero(), nhi = f4zero();
        float nl = 0.f, nrr = 0.f;
        if (z + 1 < z1) {
            const int kn = PER ? kxy + zp(z + 1) : kz + g.nxy;
            if (hold && (z + 2 < g.nz || pz)) nup = LD::load(yv, PER ? kxy + zp(z + 2) : kn + g.nxy);
            if (own) {
                if (ypv) nyp = LD::load(ypv, kn);
                if constexpr (!PRED) nr = LD::load(rv, kn);
            }
            if (rowlo) nlo = LD::load(yv, kn + dlo);
            if (rowhi) nhi = LD::load(yv, kn + dhi);
            if (xl) nl = ldcg(yv, kn + dxl);
            if (xr) nrr = ldcg(yv, kn + dxr);
        }
        pl[ty + 1][tx] = vc;
        if (ty == 0) pl[0][tx] = hlo;
        if (ty == TY - 1) pl[TY + 1][tx] = hhi;
        // x neighbours across threads of the warp row
        float left = __shfl_up_sync(0xffffffffu, vc.w, 1);
        float right = __shfl_down_sync(0xffffffffu, vc.x, 1);
        if (tx == 0) left = hl;
        if (x == xlast) right = hr;
        __syncthreads();
        if constexpr (PRED) {   // omega the factor of the neighbour differences
            if (own) {
                // a wall's neighbour is the cell itself: its difference is zero
                float4 up = pl[ty][tx], dn = pl[ty + 2][tx], zd = vdn, zu = vup;
                if (!py && y == 0) up = vc;
                if (!py && y + 1 == g.ny) dn = vc;
                if (!pz && z == 0) zd = vc;
                if (!pz && z + 1 == g.nz) zu = vc;
                if (!px && x == 0) left = vc.x;
                if (!px && x + 4 == g.nx) right = vc.w;
                float4 d, o;
                d.x = ((left - vc.x) + (vc.y - vc.x)) + ((up.x - vc.x) + (dn.x - vc.x)) + ((zd.x - vc.x) + (zu.x - vc.x));
                d.y = ((vc.x - vc.y) + (vc.z - vc.y)) + ((up.y - vc.y) + (dn.y - vc.y)) + ((zd.y - vc.y) + (zu.y - vc.y));
                d.z = ((vc.y - vc.z) + (vc.w - vc.z)) + ((up.z - vc.z) + (dn.z - vc.z)) + ((zd.z - vc.z) + (zu.z - vc.z));
                d.w = ((vc.z - vc.w) + (right - vc.w)) + ((up.w - vc.w) + (dn.w - vc.w)) + ((zd.w - vc.w) + (zu.w - vc.w));
                if (ypv) {
                    o.x = fmaf(omega, d.x, (vc.x - ypc.x) + vc.x);
                    o.y = fmaf(omega, d.y, (vc.y - ypc.y) + vc.y);
                    o.z = fmaf(omega, d.z, (vc.z - ypc.z) + vc.z);
                    o.w = fmaf(omega, d.w, (vc.w - ypc.w) + vc.w);
                } else {
                    o.x = fmaf(omega, d.x, vc.x);
                    o.y = fmaf(omega, d.y, vc.y);
                    o.z = fmaf(omega, d.z, vc.z);
                    o.w = fmaf(omega, d.w, vc.w);
                }
                V::store(ynv, kz, o);
            }
        } else if (own) {
            const float4 up = pl[ty][tx], dn = pl[ty + 2][tx];
            float d0 = d0i, d12 = d12i, d3 = d3i;
            if (!pz && (z == 0 || z + 1 == g.nz)) {   // a z wall: fewer neighbours
                const int nz_ = (z > 0) + (z + 1 < g.nz);
                d0 = sdg[n0 + nz_];
                d12 = sdg[n12 + nz_];
                d3 = sdg[n3 + nz_];
            }
            float4 s;
            s.x = left + vc.y + up.x + dn.x + vdn.x + vup.x;
            s.y = vc.x + vc.z + up.y + dn.y + vdn.y + vup.y;
            s.z = vc.y + vc.w + up.z + dn.z + vdn.z + vup.z;
            s.w = vc.z + right + up.w + dn.w + vdn.w + vup.w;
            float4 o;
            o.x = fmaf(omega, vc.x - ypc.x + gamma * (rc.x - fmaf(d0, vc.x, -cf.ce * s.x)), ypc.x);
            o.y = fmaf(omega, vc.y - ypc.y + gamma * (rc.y - fmaf(d12, vc.y, -cf.ce * s.y)), ypc.y);
            o.z = fmaf(omega, vc.z - ypc.z + gamma * (rc.z - fmaf(d12, vc.z, -cf.ce * s.z)), ypc.z);
            o.w = fmaf(omega, vc.w - ypc.w + gamma * (rc.w - fmaf(d3, vc.w, -cf.ce * s.w)), ypc.w);
            V::store(ynv, kz, o);
        }
        __syncthreads();
        vdn = vc;
        vc = vup;
        vup = nup;
        ypc = nyp;
        rc = nr;
        hlo = nlo;
        hhi = nhi;
        hl = nl;
        hr = nrr;
    }
}

// The unrolled marches of two and four planes keep their queue in 76 to 80 registers, three
// blocks to an SM (at four blocks they spill): 128^3, 2 planes 6.39 -> 5.71 us per
// iteration, 3 fields, 4 planes 16.6 -> 13.3 us (2 planes 16.0 -> 14.1); periodic on every
// axis, 256 x 128 x 128, 4 planes 15.5 -> 13.9 us.
template <class TS, int ZFIX = 0, bool PER = false>
__global__ void __launch_bounds__(kThreads, ZFIX >= 2 ? 3 : 4) k_cheb_v4(Geo g, int zlen, int nzc, Coef32 cf,
                                                      float gamma, float omega,
                                                      const TS *__restrict__ y_all,
                                                      const TS *yprev_all,
                                                      const TS *__restrict__ r_all, TS *ynext_all) {
    chain_wait();
    chain_release();
    const int f = nzc == (int)gridDim.z ? 0 : (int)blockIdx.z / nzc;   // one field: no division
    const int z0 = ((int)blockIdx.z - f * nzc) * zlen;
    const int z1 = min(g.nz, z0 + zlen);
    const size_t off = (size_t)f * g.n;
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    __syncthreads();
    cheb_v4_tile<TS, Vec4, ZFIX, PER>(g, blockIdx.x, blockIdx.y, z0, z1, cf, sdg, gamma, omega, y_all + off,
                           yprev_all ? yprev_all + off : nullptr, r_all + off, ynext_all + off);
}

// ---------------------------------------------------------------- shared expansion
// The first refinement round of every implicit step of a run of steps, from ONE Chebyshev
// recurrence.  With A = I - ce L and u_i the steps' exact solutions, the increment of step
// i is u_{i+1} - u_i = h_i(L) u_0 for the rational h_i of the scheme (pred_plan), so all
// increments are combinations of the same vectors T_k(L) u_0, T_k the Chebyshev
// polynomials on the spectrum of L.  The recurrence runs in FP32 sweeps (k_cheb* without
// r: T_{k+1} = 2 (T_k - A' T_k) - T_{k-1}, A' = -2 L / mu_max), and k_pred_combine forms
// every step's increment.  Its FP32 rounding leaves a residual of 1e-9 to 1e-6 of ||b||
// (it scales with sum_k |coef|, at most 1.6 and mostly below 0.2), which is what an own
// inner solve per step leaves after its first round; the step's refinement goes on from
// there as before and its residual is checked as before.  The run's K sweeps take the place
// of one inner solve per step: at 128^3, 10 steps, b = 8 dx 77 sweeps for 350, b = 2 dx 20
// for 90.
constexpr int kPredMaxK = 160;     // highest T_k
constexpr int kPredMaxSteps = 20;  // steps per run (accumulators of k_pred_combine)

// One step of the recurrence in difference form, T_{k+1} = (T_k - T_{k-1}) + T_k + w D T_k
// with D the sum of the differences to the neighbours (T_1 = T_0 + w D T_0: tprev ==
// nullptr).  At the lower end of the spectrum the recurrence amplifies a rounding error
// by the number of steps left; in this form a constant field stays exactly constant and a
// smooth one nearly so, while a neighbour sum less nn times the value rounds in proportion
// to the value: the error of the final field (40 steps, b = 4 dx) is 4e-15 with the
// differences and 1e-13 without.  Vectorised (nx % 4 == 0): k_cheb_v4's tile.
template <int ZFIX, bool PER>
__global__ void __launch_bounds__(kThreads, 4) k_pred_v4(Geo g, int zlen, int nzc, float w,
                                                      const float *__restrict__ t_all,
                                                      const float *__restrict__ tprev_all,
                                                      float *__restrict__ tnext_all) {
    chain_wait();
    chain_release();
    const int f = nzc == (int)gridDim.z ? 0 : (int)blockIdx.z / nzc;
    const int z0 = ((int)blockIdx.z - f * nzc) * zlen;
    const int z1 = min(g.nz, z0 + zlen);
    const size_t off = (size_t)f * g.n;
    const float dg[8] = {};   // unused by the difference form
    cheb_v4_tile<float, Vec4, ZFIX, PER, true>(g, blockIdx.x, blockIdx.y, z0, z1, Coef32{}, dg, 0.f, w, t_all + off,
                                               tprev_all ? tprev_all + off : nullptr, nullptr, tnext_all + off);
}

// The same step on any mesh: the neighbour sum is carried as an FP32 pair (a TwoSum
// cascade), so that less nn times the value it is the sum of the differences to FP32
// accuracy.  Four planes per block (walls) or the z march (a periodic axis).
template <bool PER>
__global__ void __launch_bounds__(kThreads) k_pred_any(Geo g, int zlen, int nzc, float w,
                                                       const float *__restrict__ t_all,
                                                       const float *__restrict__ tprev_all,
                                                       float *__restrict__ tnext_all) {
    chain_wait();
    chain_release();
    const int f = blockIdx.z / nzc;
    const int z0 = (blockIdx.z - f * nzc) * zlen;
    const size_t off = (size_t)f * g.n;
    const float *t = t_all + off, *tp = tprev_all ? tprev_all + off : nullptr;
    float *tn = tnext_all + off;
    auto load = [&](int k) { return DF{t[k], 0.f}; };
    auto prev = [&](int k) { return tp ? tp[k] : 0.f; };
    auto use = [&](int k, DF v, DF s, int nn, float p) {
        const float d = df_f(df_lap(s, v, (float)nn));
        tn[k] = fmaf(w, d, tp ? (v.hi - p) + v.hi : v.hi);
    };
    if constexpr (PER) sweep25p<DF>(g, z0, min(g.nz, z0 + zlen), load, prev, use);
    else sweepzb<4, DF>(g, blockIdx.x, blockIdx.y, z0, load, prev, use);
}

// T_0: the hi parts of a double-float field (pair layout or one pair per cell).
__global__ void __launch_bounds__(kThreads) k_pred_start(size_t n, bool pairs, const DF *__restrict__ u,
                                                         float *__restrict__ t0) {
    chain_wait();
    chain_release();
    const size_t step = (size_t)gridDim.x * blockDim.x, i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (pairs) {
        for (size_t i = i0; i < n / 2; i += step) {
            const float4 v = reinterpret_cast<const float4 *>(u)[i];
            reinterpret_cast<float2 *>(t0)[i] = make_float2(v.x, v.y);
        }
    } else {
        for (size_t i = i0; i < n; i += step) t0[i] = u[i].hi;
    }
}

template <int NS> struct PredCoef {
    float a[(kPredMaxK + 1) * NS];
};

// d_i = sum_k a[k][i] T_k for NS steps: each T_k is read once for all of them.  Bound by
// HBM (K + 1 vectors read, NS written) and, for many steps, by the multiply-adds; four
// cells per thread, two cells to an instruction, four vectors' loads in flight.  The
// vectors are `stride` floats apart and padded to whole float4s.
template <int NS>
__global__ void __launch_bounds__(kThreads) k_pred_combine(size_t n4, size_t stride, int K,
                                                           const __grid_constant__ PredCoef<NS> cf,
                                                           const float *__restrict__ t,
                                                           float *__restrict__ d) {
    chain_wait();
    chain_release();
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < n4; i += (size_t)gridDim.x * kThreads) {
        float2 lo[NS], hi[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q) lo[q] = hi[q] = make_float2(0.f, 0.f);
        const float *tp = t + 4 * i;
#pragma unroll 4
        for (int k = 0; k <= K; ++k, tp += stride) {
            const float4 v = *reinterpret_cast<const float4 *>(tp);
            const float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                const float w = cf.a[k * NS + q];
                lo[q] = fma2(a, make_float2(w, w), lo[q]);
                hi[q] = fma2(b, make_float2(w, w), hi[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < NS; ++q)
            *reinterpret_cast<float4 *>(d + q * stride + 4 * i) = make_float4(lo[q].x, lo[q].y, hi[q].x, hi[q].y);
    }
}

// ---------------------------------------------------------------- two iterations per sweep
// Iterations k and k+1 of the Chebyshev recurrence in one launch (temporal blocking), for
// rows of at most 128 cells (nx <= 128, nx % 4 == 0: a warp holds a whole row, four cells
// per lane, so x needs no halo).  A block owns TY2 rows and a z-chunk; it also computes
// y_{k+1} on the row above and the row below (from y_k on two rows either side), which
// y_{k+2} needs.  It marches q over the chunk's planes plus one either side: y_{k+1} on
// plane q from y_k (register queue over q-1, q, q+1; rows from a shared plane), then
// y_{k+2} on plane q-1 from y_{k+1} (register queue, rows from a second shared plane).
// y_{k+1} and y_{k+2} go to two buffers that nothing in the launch reads, so the rows a
// block recomputes never race with their owners' writes (four buffers rotate across
// launches).  Arithmetic and its order per cell are those of k_cheb_v4.
constexpr int TY2 = 8;
constexpr int kCheb2Threads = 32 * (TY2 + 2);

// A value as the storage type holds it (y_{k+1} is used by iteration k+1 exactly as the
// one-iteration sweep would read it back from memory).
template <class TS> __device__ __forceinline__ float4 as_stored(float4 v) { return v; }
template <> __device__ __forceinline__ float4 as_stored<__nv_bfloat16>(float4 v) {
    return make_float4(__bfloat162float(__float2bfloat16_rn(v.x)), __bfloat162float(__float2bfloat16_rn(v.y)),
                       __bfloat162float(__float2bfloat16_rn(v.z)), __bfloat162float(__float2bfloat16_rn(v.w)));
}
constexpr int kPairCode = 200;   // sweep_shape 200 + z: two iterations per launch, z planes

template <class TS>
__global__ void __launch_bounds__(kCheb2Threads, 2)
    k_cheb2_v4(Geo g, int zlen, int nzc, Coef32 cf, float gamma, float om1, float om2,
               const TS *__restrict__ yk_all, const TS *__restrict__ ykm_all,
               const TS *__restrict__ r_all, TS *__restrict__ c_all, TS *__restrict__ d_all) {
    chain_wait();
    chain_release();
    using V = Vec4<TS>;
    __shared__ float4 Sk[TY2 + 4][32];   // y_k on plane q, rows y0-2 .. y0+TY2+1
    __shared__ float4 Su[TY2 + 2][32];   // y_{k+1} on plane q-1, rows y0-1 .. y0+TY2
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    const int f = blockIdx.z / nzc;
    const int z0 = (blockIdx.z - f * nzc) * zlen, z1 = min(g.nz, z0 + zlen);
    const size_t off = (size_t)f * g.n;
    const TS *yk = yk_all + off;
    const TS *ykm = ykm_all ? ykm_all + off : nullptr;
    const TS *r = r_all + off;
    TS *yc = c_all + off;
    TS *yd = d_all + off;
    const int tx = threadIdx.x, t = threadIdx.y;
    const int x = 4 * tx;
    const int y0 = blockIdx.y * TY2, y = y0 - 1 + t;
    const bool ownx = x < g.nx;
    const bool rowin = y >= 0 && y < g.ny && ownx;
    const bool inner = t >= 1 && t <= TY2 && y < g.ny && ownx;   // rows this block writes
    const bool hlo = t == 0 && y0 - 2 >= 0 && ownx;                // also loads row y0-2
    const bool hhi = t == TY2 + 1 && y0 + TY2 + 1 < g.ny && ownx;  // also loads row y0+TY2+1
    const int nyb = (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + (x > 0) + 1, n3 = nyb + 1 + (x + 4 < g.nx), n12 = nyb + 2;
    // 32-bit offsets within a field (a field has fewer than 2^31 cells)
    auto at = [&](int q, int yy) -> int { return (q * g.ny + yy) * g.nx + x; };
    const int qs = max(z0 - 1, 0);
    // queues at q = qs
    float4 vkm = f4zero(), vk0 = f4zero(), vkp = f4zero(), hk = f4zero();
    float4 ypq = f4zero(), rq = f4zero(), rprev = f4zero();
    if (rowin) {
        if (qs > 0) vkm = V::load(yk, at(qs - 1, y));
        vk0 = V::load(yk, at(qs, y));
        if (qs + 1 < g.nz) vkp = V::load(yk, at(qs + 1, y));
        if (ykm) ypq = V::load(ykm, at(qs, y));
        rq = V::load(r, at(qs, y));
    }
    if (hlo) hk = V::load(yk, at(qs, y0 - 2));
    if (hhi) hk = V::load(yk, at(qs, y0 + TY2 + 1));
    __syncthreads();   // the diagonal table
    // diagonals of the four cells on planes with both z neighbours (most planes)
    const float d0i = sdg[n0 + 2], d12i = sdg[n12 + 2], d3i = sdg[n3 + 2];
    float4 um = f4zero(), u0 = f4zero();
    for (int q = qs; q <= z1; ++q) {
        // loads for plane q+1 (y_k two planes ahead)
        float4 nvkp = f4zero(), nhk = f4zero(), nyp = f4zero(), nr = f4zero();
        if (q + 1 < g.nz) {
            if (rowin) {
                if (q + 2 < g.nz) nvkp = V::load(yk, at(q + 2, y));
                if (ykm) nyp = V::load(ykm, at(q + 1, y));
                nr = V::load(r, at(q + 1, y));
            }
            if (hlo) nhk = V::load(yk, at(q + 1, y0 - 2));
            if (hhi) nhk = V::load(yk, at(q + 1, y0 + TY2 + 1));
        }
        Sk[t + 1][tx] = vk0;
        if (t == 0) Sk[0][tx] = hk;
        if (t == TY2 + 1) Sk[TY2 + 3][tx] = hk;
        Su[t][tx] = u0;
        // x neighbours of y_k (plane q) and of y_{k+1} (plane q-1) across lanes
        const float kl = __shfl_up_sync(0xffffffffu, vk0.w, 1);
        const float kr = __shfl_down_sync(0xffffffffu, vk0.x, 1);
        const float ul = __shfl_up_sync(0xffffffffu, u0.w, 1);
        const float ur = __shfl_down_sync(0xffffffffu, u0.x, 1);
        __syncthreads();
        // y_{k+1} on plane q
        float4 un = f4zero();
        if (q < g.nz && rowin) {
            const float4 up = Sk[t][tx], dn = Sk[t + 2][tx];
            const float left = tx == 0 ? 0.f : kl, right = x + 4 < g.nx ? kr : 0.f;
            float d0 = d0i, d12 = d12i, d3 = d3i;
            if (q == 0 || q + 1 == g.nz) {   // a z wall: fewer neighbours
                const int nz_ = (q > 0) + (q + 1 < g.nz);
                d0 = sdg[n0 + nz_];
                d12 = sdg[n12 + nz_];
                d3 = sdg[n3 + nz_];
            }
            float4 s;
            s.x = left + vk0.y + up.x + dn.x + vkm.x + vkp.x;
            s.y = vk0.x + vk0.z + up.y + dn.y + vkm.y + vkp.y;
            s.z = vk0.y + vk0.w + up.z + dn.z + vkm.z + vkp.z;
            s.w = vk0.z + right + up.w + dn.w + vkm.w + vkp.w;
            un.x = fmaf(om1, vk0.x - ypq.x + gamma * (rq.x - fmaf(d0, vk0.x, -cf.ce * s.x)), ypq.x);
            un.y = fmaf(om1, vk0.y - ypq.y + gamma * (rq.y - fmaf(d12, vk0.y, -cf.ce * s.y)), ypq.y);
            un.z = fmaf(om1, vk0.z - ypq.z + gamma * (rq.z - fmaf(d12, vk0.z, -cf.ce * s.z)), ypq.z);
            un.w = fmaf(om1, vk0.w - ypq.w + gamma * (rq.w - fmaf(d3, vk0.w, -cf.ce * s.w)), ypq.w);
            un = as_stored<TS>(un);
            if (inner && q >= z0 && q < z1) V::store(yc, at(q, y), un);
        }
        // y_{k+2} on plane z = q-1
        const int z = q - 1;
        if (inner && z >= z0 && z < z1) {
            const float4 up = Su[t - 1][tx], dn = Su[t + 1][tx];
            const float left = tx == 0 ? 0.f : ul, right = x + 4 < g.nx ? ur : 0.f;
            float d0 = d0i, d12 = d12i, d3 = d3i;
            if (z == 0 || z + 1 == g.nz) {
                const int nz_ = (z > 0) + (z + 1 < g.nz);
                d0 = sdg[n0 + nz_];
                d12 = sdg[n12 + nz_];
                d3 = sdg[n3 + nz_];
            }
            float4 s, o;
            s.x = left + u0.y + up.x + dn.x + um.x + un.x;
            s.y = u0.x + u0.z + up.y + dn.y + um.y + un.y;
            s.z = u0.y + u0.w + up.z + dn.z + um.z + un.z;
            s.w = u0.z + right + up.w + dn.w + um.w + un.w;
            o.x = fmaf(om2, u0.x - vkm.x + gamma * (rprev.x - fmaf(d0, u0.x, -cf.ce * s.x)), vkm.x);
            o.y = fmaf(om2, u0.y - vkm.y + gamma * (rprev.y - fmaf(d12, u0.y, -cf.ce * s.y)), vkm.y);
            o.z = fmaf(om2, u0.z - vkm.z + gamma * (rprev.z - fmaf(d12, u0.z, -cf.ce * s.z)), vkm.z);
            o.w = fmaf(om2, u0.w - vkm.w + gamma * (rprev.w - fmaf(d3, u0.w, -cf.ce * s.w)), vkm.w);
            V::store(yd, at(z, y), o);
        }
        __syncthreads();
        um = u0;
        u0 = un;
        vkm = vk0;
        vk0 = vkp;
        vkp = nvkp;
        hk = nhk;
        ypq = nyp;
        rprev = rq;
        rq = nr;
    }
}

// ---------------------------------------------------------------- two iterations per sweep, long rows
// The pair recurrence of k_cheb2_v4 for rows of up to 512 cells (nx % 4 == 0), where one
// warp no longer holds a row.  A block holds whole rows: W = nx/4 threads to a row,
// rounded up to whole warps (at most four), and TYR = blockDim.y - 2 rows it writes, with
// y_{k+1} recomputed on the row either side as in k_cheb2_v4.  A thread's x neighbours
// come from the adjacent lanes by shuffle, and across a warp boundary from the staged
// plane.  Instead of a register queue, y_k, y_{k-1} and r of the planes ahead are staged
// in shared-memory rings by cp.async one plane ahead of the march: y_k in four slots
// (planes q-1 .. q+2, all TYR + 4 rows), y_{k-1} in two (q, q+1), r in four (three in use,
// q-1 .. q+1); planes and rows outside the mesh are staged as zeros.  A slot is refilled
// only after the barrier that ends the step which last read it.  The row width W is a
// template parameter and the march is unrolled by four, so every slot offset is a
// constant.  With the queue in shared memory a block of 1024 threads fits the
// 64-register budget, one block per SM.  Per
// cell the arithmetic and its order are those of k_cheb_v4, so the iterates are
// bit-identical.  It pays where the sweep is bound by HBM: two iterations move 20 bytes
// per cell (three reads, two writes) instead of 32.  A periodic x axis wraps within the
// block's rows (y and z must be walls).
constexpr int kRowsThreads = 1024;
constexpr int kRowsMaxNx = 512;

// a row vector of four cells as stored: 16 bytes in FP32, 8 in BF16
template <class TS> using RowV = typename std::conditional<sizeof(TS) == 4, float4, uint2>::type;
template <class TS> __device__ __forceinline__ float4 rowv_f4(const RowV<TS> &v) {
    if constexpr (sizeof(TS) == 4) {
        return v;
    } else {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
        return make_float4(a.x, a.y, b.x, b.y);
    }
}
// stage one row vector (ok) or zeros
template <class TS> __device__ __forceinline__ void rowv_stage(RowV<TS> *dst, const TS *src, bool ok) {
    if (ok) {
        if constexpr (sizeof(TS) == 4) cp_async16(dst, src);
        else cp_async8(dst, src);
    } else {
        *dst = RowV<TS>{};
    }
}
// threads per row, rows per block and dynamic shared memory of a launch
__host__ __device__ inline int rows_width(int nx) { return ((nx / 4 + 31) / 32) * 32; }
inline int rows_per_block(int nx) { return kRowsThreads / rows_width(nx) - 2; }
template <class TS> inline size_t rows_smem(int W, int tyr) {
    return (size_t)W * ((size_t)(4 * (tyr + 4) + 6 * (tyr + 2)) * sizeof(RowV<TS>) + (size_t)(tyr + 2) * 16);
}

template <class TS, int W>
__global__ void __launch_bounds__(kRowsThreads, 1)
    k_cheb2_rows(Geo g, int zlen, int nzc, Coef32 cf, float gamma, float om1, float om2,
                 const TS *__restrict__ yk_all, const TS *__restrict__ ykm_all,
                 const TS *__restrict__ r_all, TS *__restrict__ c_all, TS *__restrict__ d_all) {
    chain_wait();
    chain_release();
    using RV = RowV<TS>;
    using V = Vec4<TS>;
    extern __shared__ __align__(16) unsigned char rows_sm[];
    __shared__ float sdg[8];
    stage_table(sdg, cf.dg);
    constexpr int TYR = kRowsThreads / W - 2;   // rows written per block
    constexpr int KR = TYR + 4, MR = TYR + 2;
    RV *Kr = reinterpret_cast<RV *>(rows_sm);                   // y_k    [4][KR][W]
    RV *Mr = Kr + 4 * KR * W;                                   // y_{k-1} [2][MR][W]
    RV *Rr = Mr + 2 * MR * W;                                   // r      [4][MR][W]
    float4 *Su = reinterpret_cast<float4 *>(Rr + 4 * MR * W);   // y_{k+1} of plane q-1 [MR][W]
    const int f = blockIdx.z / nzc;
    const int z0 = (blockIdx.z - f * nzc) * zlen, z1 = min(g.nz, z0 + zlen);
    const size_t off = (size_t)f * g.n;
    const TS *yk = yk_all + off;
    const TS *ykm = ykm_all ? ykm_all + off : nullptr;
    const TS *r = r_all + off;
    TS *yc = c_all + off;
    TS *yd = d_all + off;
    const int tx = threadIdx.x, t = threadIdx.y, lane = tx & 31;
    const int x = 4 * tx;
    const int y0 = blockIdx.y * TYR, y = y0 - 1 + t;
    const bool ownx = x < g.nx;
    const bool rowin = y >= 0 && y < g.ny && ownx;
    const bool inner = t >= 1 && t <= TYR && y < g.ny && ownx;   // rows this block writes
    const bool hrow = t == 0 || t == TYR + 1;                    // also stages row y0-2 / y0+TYR+1
    const int yh = t == 0 ? y0 - 2 : y0 + TYR + 1;
    const bool hin = hrow && yh >= 0 && yh < g.ny && ownx;
    const int hslot = t == 0 ? 0 : KR - 1;
    // a periodic x axis (the only periodic axis this kernel takes): a row's first and last
    // cells are neighbours, both held by the block
    const bool px = (g.per & 1) != 0;
    const int xlast = g.nx / 4 - 1;   // the thread holding a row's last four cells
    const int nyb = (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + (px || x > 0) + 1, n3 = nyb + 1 + (px || x + 4 < g.nx), n12 = nyb + 2;
    // 32-bit offsets within a field (a field has fewer than 2^31 cells)
    const int kown = rowin ? y * g.nx + x : 0, khalo = hin ? yh * g.nx + x : 0;
    constexpr int KW = KR * W, MW = MR * W;
    // ring slots: plane p sits in slot (p - qs + 1) mod 4 of the y_k and r rings and mod 2 of
    // the y_{k-1} ring; the march is unrolled by four, so every slot index is a constant
    const int qs = max(z0 - 1, 0);
    RV *const kown_s = Kr + (t + 1) * W + tx;   // this thread's row in slot 0 of the y_k ring
    RV *const mown_s = Mr + t * W + tx;
    RV *const rown_s = Rr + t * W + tx;
    // staging of plane p (slot s): y_k up to plane z1 + 1, y_{k-1} and r up to plane z1
    auto stage_k = [&](int p, int sl) __attribute__((always_inline)) {
        if (p > z1 + 1) return;
        const bool pin = p >= 0 && p < g.nz;
        const int kp = pin ? p * g.nxy : 0;
        rowv_stage<TS>(kown_s + sl * KW, yk + (kp + kown), pin && rowin);
        if (hrow) rowv_stage<TS>(Kr + sl * KW + hslot * W + tx, yk + (kp + khalo), pin && hin);
    };
    auto stage_mr = [&](int p, int sm, int sr) __attribute__((always_inline)) {
        if (p > z1) return;
        const bool ok = p < g.nz && rowin;
        const int kp = (ok ? p * g.nxy : 0) + kown;
        if (ykm) rowv_stage<TS>(mown_s + sm * MW, ykm + kp, ok);
        rowv_stage<TS>(rown_s + sr * MW, r + kp, ok);
    };
    stage_k(qs - 1, 0);
    stage_k(qs, 1);
    stage_k(qs + 1, 2);
    stage_mr(qs, 1, 1);
    cp_async_commit();
    __syncthreads();   // the diagonal table
    // diagonals of the four cells on planes with both z neighbours (most planes)
    const float d0i = sdg[n0 + 2], d12i = sdg[n12 + 2], d3i = sdg[n3 + 2];
    // y_{k+1} of planes q - 2 and q - 1
    float4 um = f4zero(), u0 = f4zero();
    // step q (the march's step j of four, j = (q - qs) mod 4): y_{k+1} on plane q, y_{k+2} on
    // plane q - 1
    auto step = [&](const int q, auto jc) __attribute__((always_inline)) {
        constexpr int j = decltype(jc)::value;
        constexpr int sk_m = j, sk_0 = (j + 1) & 3, sk_p = (j + 2) & 3, sk_pp = (j + 3) & 3;
        constexpr int sm_0 = (j + 1) & 1, sm_p = j & 1;
        constexpr int sr_m = j, sr_0 = (j + 1) & 3, sr_p = (j + 2) & 3;
        stage_k(q + 2, sk_pp);
        stage_mr(q + 1, sm_p, sr_p);
        cp_async_commit();
        cp_async_wait<1>();   // this thread's copies of the planes step q reads
        Su[t * W + tx] = u0;
        __syncthreads();
        RV *const k0 = kown_s + sk_0 * KW;   // this thread's vector of plane q
        const float4 vk0 = rowv_f4<TS>(*k0);
        const float4 vkm = rowv_f4<TS>(*(kown_s + sk_m * KW));
        // x neighbours of y_k (plane q) and of y_{k+1} (plane q-1): lanes, or across a warp
        float kl = __shfl_up_sync(0xffffffffu, vk0.w, 1);
        float kr = __shfl_down_sync(0xffffffffu, vk0.x, 1);
        float ul = __shfl_up_sync(0xffffffffu, u0.w, 1);
        float ur = __shfl_down_sync(0xffffffffu, u0.x, 1);
        if (lane == 0 && tx > 0) {
            kl = rowv_f4<TS>(*(k0 - 1)).w;
            ul = Su[t * W + tx - 1].w;
        }
        if (lane == 31 && tx + 1 < W) {
            kr = rowv_f4<TS>(*(k0 + 1)).x;
            ur = Su[t * W + tx + 1].x;
        }
        if (px && tx == 0) {       // cell nx - 1
            kl = rowv_f4<TS>(*(k0 + xlast)).w;
            ul = Su[t * W + xlast].w;
        }
        if (px && tx == xlast) {   // cell 0
            kr = rowv_f4<TS>(*(k0 - tx)).x;
            ur = Su[t * W].x;
        }
        // y_{k+1} on plane q
        float4 un = f4zero();
        if (q < g.nz && rowin) {
            const float4 up = rowv_f4<TS>(*(k0 - W)), dn = rowv_f4<TS>(*(k0 + W));
            const float4 vkp = rowv_f4<TS>(*(kown_s + sk_p * KW));
            const float4 ypq = ykm ? rowv_f4<TS>(*(mown_s + sm_0 * MW)) : f4zero();
            const float4 rq = rowv_f4<TS>(*(rown_s + sr_0 * MW));
            const float left = (px || tx > 0) ? kl : 0.f, right = (px || x + 4 < g.nx) ? kr : 0.f;
            float d0 = d0i, d12 = d12i, d3 = d3i;
            if (q == 0 || q + 1 == g.nz) {   // a z wall: fewer neighbours
                const int nz_ = (q > 0) + (q + 1 < g.nz);
                d0 = sdg[n0 + nz_];
                d12 = sdg[n12 + nz_];
                d3 = sdg[n3 + nz_];
            }
            float4 s;
            s.x = left + vk0.y + up.x + dn.x + vkm.x + vkp.x;
            s.y = vk0.x + vk0.z + up.y + dn.y + vkm.y + vkp.y;
            s.z = vk0.y + vk0.w + up.z + dn.z + vkm.z + vkp.z;
            s.w = vk0.z + right + up.w + dn.w + vkm.w + vkp.w;
            un.x = fmaf(om1, vk0.x - ypq.x + gamma * (rq.x - fmaf(d0, vk0.x, -cf.ce * s.x)), ypq.x);
            un.y = fmaf(om1, vk0.y - ypq.y + gamma * (rq.y - fmaf(d12, vk0.y, -cf.ce * s.y)), ypq.y);
            un.z = fmaf(om1, vk0.z - ypq.z + gamma * (rq.z - fmaf(d12, vk0.z, -cf.ce * s.z)), ypq.z);
            un.w = fmaf(om1, vk0.w - ypq.w + gamma * (rq.w - fmaf(d3, vk0.w, -cf.ce * s.w)), ypq.w);
            un = as_stored<TS>(un);
            if (inner && q >= z0 && q < z1) V::store(yc, q * g.nxy + kown, un);
        }
        // y_{k+2} on plane z = q-1
        const int z = q - 1;
        if (inner && z >= z0 && z < z1) {
            const float4 up = Su[(t - 1) * W + tx], dn = Su[(t + 1) * W + tx];
            const float4 rp = rowv_f4<TS>(*(rown_s + sr_m * MW));
            const float left = (px || tx > 0) ? ul : 0.f, right = (px || x + 4 < g.nx) ? ur : 0.f;
            float d0 = d0i, d12 = d12i, d3 = d3i;
            if (z == 0 || z + 1 == g.nz) {
                const int nz_ = (z > 0) + (z + 1 < g.nz);
                d0 = sdg[n0 + nz_];
                d12 = sdg[n12 + nz_];
                d3 = sdg[n3 + nz_];
            }
            float4 s, o;
            s.x = left + u0.y + up.x + dn.x + um.x + un.x;
            s.y = u0.x + u0.z + up.y + dn.y + um.y + un.y;
            s.z = u0.y + u0.w + up.z + dn.z + um.z + un.z;
            s.w = u0.z + right + up.w + dn.w + um.w + un.w;
            o.x = fmaf(om2, u0.x - vkm.x + gamma * (rp.x - fmaf(d0, u0.x, -cf.ce * s.x)), vkm.x);
            o.y = fmaf(om2, u0.y - vkm.y + gamma * (rp.y - fmaf(d12, u0.y, -cf.ce * s.y)), vkm.y);
            o.z = fmaf(om2, u0.z - vkm.z + gamma * (rp.z - fmaf(d12, u0.z, -cf.ce * s.z)), vkm.z);
            o.w = fmaf(om2, u0.w - vkm.w + gamma * (rp.w - fmaf(d3, u0.w, -cf.ce * s.w)), vkm.w);
            V::store(yd, z * g.nxy + kown, o);
        }
        __syncthreads();   // the slots step q read are refilled from step q + 1 on
        um = u0;
        u0 = un;
    };
    using I0 = std::integral_constant<int, 0>;
    using I1 = std::integral_constant<int, 1>;
    using I2 = std::integral_constant<int, 2>;
    using I3 = std::integral_constant<int, 3>;
    for (int q = qs; q <= z1; q += 4) {
        step(q, I0{});
        if (q + 1 <= z1) step(q + 1, I1{});
        if (q + 2 <= z1) step(q + 2, I2{});
        if (q + 3 <= z1) step(q + 3, I3{});
    }
    cp_async_wait<0>();   // no copy outlives the block
}

// ---------------------------------------------------------------- on-chip resident sweep
constexpr int kResidentThreads = 1024;
constexpr int kResidentMaxIters = 128;
constexpr int kResidentCode = 300;   // sweep_shape of the resident inner solve
constexpr int kTmaCode = 400;        // sweep_shape 400 + z: TMA-staged sweep, z planes per block

// The m-1 Chebyshev iterations of one refinement round with the iterates held in shared
// memory, for a mesh whose two iterates fit in the SMs' shared memory (one field,
// nx % 4 == 0).  The mesh is cut into bricks of whole x-rows (by rows x bz planes), one
// brick per block, every block resident (cooperative launch, one block per SM).  Each
// shared array holds a brick with a one-row / one-plane halo in y and z and four zero
// cells of padding at both ends of every row (the x walls).  Per iteration a block
// computes y_{k+1} over its brick from y_k (neighbours from shared memory) and y_{k-1}
// (same cell, overwritten), r from global memory: first the brick's surface rows, whose
// four faces (y and z) it then publishes to global memory (two parities) before raising
// its flag to k+1 (a release store), then the inner rows while the faces travel; then it
// waits -- bounded -- until its up to four neighbours have raised theirs and copies their
// faces into its halo.  A neighbour cannot overwrite a face parity before this block has read it: it
// would first need this block's next face.  Halos on walls stay zero.  Arithmetic and
// its order are those of k_cheb_v4, so the iterates are bit-identical.
struct Brick {
    int by, bz, nby, nbz;   // rows / planes per brick, bricks along y / z
    int pitch;              // shared row pitch in floats (nx + 8)
    int fmax;               // floats per face slot (nx * max(by, bz))
};

struct ChebWeights {
    float w[kResidentMaxIters];   // omega_k, k = 1 .. m-1
};

// floor(n / d) as a multiply-high by ceil(2^32 / d): exact whenever n * d < 2^32, which
// holds for every index divided below (at most a few thousand times at most 1024).  d = 1
// (whose multiplier would not fit in 32 bits) divides trivially.
struct FastDiv {
    unsigned int m;
    int d;
    __device__ explicit FastDiv(int d_)
        : m(d_ > 1 ? (unsigned int)((0x100000000ull + d_ - 1) / d_) : 0u), d(d_) {}
    __device__ __forceinline__ int div(int n) const {
        return d > 1 ? (int)__umulhi((unsigned int)n, m) : n;
    }
};

// One Chebyshev update (y_{k+1} into Ynext) of a brick's surface rows (boundary = true)
// or of its inner rows, for k_cheb_resident; a warp always covers whole rows, so it
// skips a row together.
template <class TS>
__device__ __forceinline__ void resident_rows(const Geo &g, const float *__restrict__ sdg, float ce,
                                              float gam, float omega, const TS *__restrict__ r,
                                              const float *Ycur, float *Ynext, int tid, int nthr,
                                              int nq, int bys, int bzs, int y0, int z0, int RW,
                                              int P, int PL, bool warp_rows, bool boundary,
                                              FastDiv dq, FastDiv dy) {
    const int nrow_b = bys * bzs;
    for (int it = tid; it < nrow_b * nq; it += nthr) {
        const int row = dq.div(it), q = it - row * nq;
        const int zz = dy.div(row), yy = row - zz * bys;
        const bool surf = yy == 0 || yy == bys - 1 || zz == 0 || zz == bzs - 1;
        if (surf != boundary) continue;
        const int gy = y0 + yy, gz = z0 + zz, x = 4 * q;
        const int si = ((zz + 1) * RW + (yy + 1)) * P + 4 + x;
        const float4 vc = *reinterpret_cast<const float4 *>(Ycur + si);
        const float4 up = *reinterpret_cast<const float4 *>(Ycur + si - P);
        const float4 dn = *reinterpret_cast<const float4 *>(Ycur + si + P);
        const float4 vdn = *reinterpret_cast<const float4 *>(Ycur + si - PL);
        const float4 vup = *reinterpret_cast<const float4 *>(Ycur + si + PL);
        float left, right;
        if (warp_rows) {   // a warp covers 128 consecutive cells of one row
            const int lane = tid & 31;
            left = __shfl_up_sync(0xffffffffu, vc.w, 1);
            right = __shfl_down_sync(0xffffffffu, vc.x, 1);
            if (lane == 0) left = Ycur[si - 1];
            if (lane == 31) right = Ycur[si + 4];
        } else {
            left = Ycur[si - 1];
            right = Ycur[si + 4];
        }
        const float4 ypc = *reinterpret_cast<const float4 *>(Ynext + si);
        const float4 rc = Vec4<TS>::load(r, ((size_t)gz * g.ny + gy) * g.nx + x);
        const int nyb = (gy > 0) + (gy + 1 < g.ny);
        const int nz_ = (gz > 0) + (gz + 1 < g.nz);
        const int n0 = nyb + (x > 0) + 1, n3 = nyb + 1 + (x + 4 < g.nx), n12 = nyb + 2;
        float4 s;
        s.x = left + vc.y + up.x + dn.x + vdn.x + vup.x;
        s.y = vc.x + vc.z + up.y + dn.y + vdn.y + vup.y;
        s.z = vc.y + vc.w + up.z + dn.z + vdn.z + vup.z;
        s.w = vc.z + right + up.w + dn.w + vdn.w + vup.w;
        float4 o;
        o.x = fmaf(omega, vc.x - ypc.x + gam * (rc.x - fmaf(sdg[n0 + nz_], vc.x, -ce * s.x)), ypc.x);
        o.y = fmaf(omega, vc.y - ypc.y + gam * (rc.y - fmaf(sdg[n12 + nz_], vc.y, -ce * s.y)), ypc.y);
        o.z = fmaf(omega, vc.z - ypc.z + gam * (rc.z - fmaf(sdg[n12 + nz_], vc.z, -ce * s.z)), ypc.z);
        o.w = fmaf(omega, vc.w - ypc.w + gam * (rc.w - fmaf(sdg[n3 + nz_], vc.w, -ce * s.w)), ypc.w);
        *reinterpret_cast<float4 *>(Ynext + si) = o;
    }
}

template <class TS>
__global__ void __launch_bounds__(kResidentThreads, 1)
    k_cheb_resident(Geo g, Brick bk, Coef32 cf, float gamma, ChebWeights om, int m,
                    const TS *__restrict__ y1, const TS *__restrict__ r, TS *__restrict__ yout,
                    float *__restrict__ faces, unsigned int *flags, int *err, long long budget) {
    extern __shared__ float4 smem4[];
    __shared__ float sdg[8];
    __shared__ float somega[kResidentMaxIters];
    __shared__ int s_stop;
    float *sm = reinterpret_cast<float *>(smem4);
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int b = blockIdx.x;
    const int iy = b % bk.nby, iz = b / bk.nby;
    const int y0 = iy * bk.by, z0 = iz * bk.bz;
    const int bys = min(bk.by, g.ny - y0), bzs = min(bk.bz, g.nz - z0);
    const int P = bk.pitch, RW = bk.by + 2, PL = RW * P;
    const int arr = PL * (bk.bz + 2);
    float *A0 = sm, *A1 = sm + arr;
    const int nq = g.nx >> 2;
    const FastDiv dq(nq), dy(bys);
#pragma unroll
    for (int i = 0; i < 7; ++i)   // constant indices: the parameter is not copied to memory
        if (tid == i) sdg[i] = cf.dg[i];
    if (tid == 7) sdg[7] = 0.f;
#pragma unroll
    for (int i = 0; i < kResidentMaxIters; i += 32)
        if (tid < 32) somega[i + tid] = om.w[i + tid];
    if (tid == 0) s_stop = 0;
    // zero both arrays (walls, padding), then y1 over the brick and its halo
    for (int i = tid; i < 2 * arr / 4; i += nthr) smem4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    {
        const int ylo = max(y0 - 1, 0), yhi = min(y0 + bys + 1, g.ny);
        const int zlo = max(z0 - 1, 0), zhi = min(z0 + bzs + 1, g.nz);
        const int ny_ = yhi - ylo, nrows = ny_ * (zhi - zlo);
        const FastDiv dny(ny_);
        for (int it = tid; it < nrows * nq; it += nthr) {
            const int row = dq.div(it), q = it - row * nq;
            const int rz = dny.div(row);
            const int gy = ylo + (row - rz * ny_), gz = zlo + rz;
            const bool iny = gy >= y0 && gy < y0 + bys, inz = gz >= z0 && gz < z0 + bzs;
            if (!iny && !inz) continue;   // halo edges and corners are never read
            const size_t k = ((size_t)gz * g.ny + gy) * g.nx + 4 * q;
            const int si = ((gz - z0 + 1) * RW + (gy - y0 + 1)) * P + 4 + 4 * q;
            *reinterpret_cast<float4 *>(A0 + si) = Vec4<TS>::load(y1, k);
        }
    }
    __syncthreads();
    float *Yc = A0, *Yp = A1;
    const int nrow_b = bys * bzs;
    const size_t fslot = (size_t)bk.fmax;
    const bool warp_rows = (nq % 32 == 0) && (nthr % 32 == 0);
    const float ce = cf.ce, gam = gamma;
    for (int k = 1; k < m; ++k) {
        const bool last = k + 1 == m;
        const int par = (k + 1) & 1;
        // surface rows first, so that their faces travel while the inner rows are computed
        resident_rows<TS>(g, sdg, ce, gam, somega[k], r, Yc, Yp, tid, nthr, nq, bys, bzs, y0, z0,
                          RW, P, PL, warp_rows, true, dq, dy);
        __syncthreads();
        if (!last) {
            // faces of y_{k+1}: slot (b, parity, face), face 0/1 = rows y0 / y0+bys-1 (all
            // planes), 2/3 = planes z0 / z0+bzs-1 (all rows)
            float *fb = faces + ((size_t)b * 2 + par) * 4 * fslot;
            for (int it = tid; it < 2 * (bzs + bys) * nq; it += nthr) {
                int rr = dq.div(it), face, si;
                const int q = it - rr * nq;
                if (rr < 2 * bzs) {
                    face = rr >= bzs ? 1 : 0;
                    rr -= face * bzs;
                    si = ((rr + 1) * RW + (face == 0 ? 1 : bys)) * P + 4 + 4 * q;
                } else {
                    rr -= 2 * bzs;
                    face = rr >= bys ? 3 : 2;
                    rr -= (face - 2) * bys;
                    si = ((face == 2 ? 1 : bzs) * RW + rr + 1) * P + 4 + 4 * q;
                }
                __stcg(reinterpret_cast<float4 *>(fb + face * fslot + (size_t)rr * g.nx + 4 * q),
                       *reinterpret_cast<const float4 *>(Yp + si));
            }
            __syncthreads();
            if (tid == 0)   // release: the block's face stores above happen before the flag
                asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(flags + b), "r"((unsigned int)(k + 1))
                             : "memory");
        }
        resident_rows<TS>(g, sdg, ce, gam, somega[k], r, Yc, Yp, tid, nthr, nq, bys, bzs, y0, z0,
                          RW, P, PL, warp_rows, false, dq, dy);
        __syncthreads();
        float *t = Yc;
        Yc = Yp;
        Yp = t;
        if (last) break;
        // wait for the neighbours' faces of y_{k+1}
        if (tid < 4) {
            const int nb = tid == 0 ? (iy > 0 ? b - 1 : -1)
                         : tid == 1 ? (iy + 1 < bk.nby ? b + 1 : -1)
                         : tid == 2 ? (iz > 0 ? b - bk.nby : -1)
                                    : (iz + 1 < bk.nbz ? b + bk.nby : -1);
            if (nb >= 0) {
                const long long t0 = clock64();
                while (true) {
                    unsigned int f;
                    asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(f) : "l"(flags + nb) : "memory");
                    if (f >= (unsigned int)(k + 1)) break;
                    if (*(volatile int *)err) {
                        s_stop = 1;
                        break;
                    }
                    if (clock64() - t0 > budget) {
                        atomicExch(err, 1);
                        s_stop = 1;
                        break;
                    }
                    __nanosleep(20);
                }
            }
        }
        __syncthreads();
        if (s_stop) return;
        // halo rows / planes from the neighbours' opposite faces
        for (int it = tid; it < 2 * (bzs + bys) * nq; it += nthr) {
            int rr = dq.div(it), side, si, nb, face;
            const int q = it - rr * nq;
            if (rr < 2 * bzs) {
                side = rr >= bzs ? 1 : 0;   // 0: row y0-1 from the lower neighbour's top face
                rr -= side * bzs;
                if (side == 0 ? iy == 0 : iy + 1 == bk.nby) continue;
                nb = side == 0 ? b - 1 : b + 1;
                face = side == 0 ? 1 : 0;
                si = ((rr + 1) * RW + (side == 0 ? 0 : bys + 1)) * P + 4 + 4 * q;
            } else {
                rr -= 2 * bzs;
                side = rr >= bys ? 1 : 0;
                rr -= side * bys;
                if (side == 0 ? iz == 0 : iz + 1 == bk.nbz) continue;
                nb = side == 0 ? b - bk.nby : b + bk.nby;
                face = side == 0 ? 3 : 2;
                si = ((side == 0 ? 0 : bzs + 1) * RW + rr + 1) * P + 4 + 4 * q;
            }
            const float *src = faces + ((size_t)nb * 2 + par) * 4 * fslot + face * fslot;
            *reinterpret_cast<float4 *>(Yc + si) =
                __ldcg(reinterpret_cast<const float4 *>(src + (size_t)rr * g.nx + 4 * q));
        }
        __syncthreads();
    }
    // y_m over the brick
    for (int it = tid; it < nrow_b * nq; it += nthr) {
        const int row = dq.div(it), q = it - row * nq;
        const int zz = dy.div(row), yy = row - zz * bys;
        const int si = ((zz + 1) * RW + (yy + 1)) * P + 4 + 4 * q;
        Vec4<TS>::store(yout, ((size_t)(z0 + zz) * g.ny + (y0 + yy)) * g.nx + 4 * q,
                        *reinterpret_cast<const float4 *>(Yc + si));
    }
}

// ---------------------------------------------------------------- flat-plane Chebyshev
// The Chebyshev iteration of k_cheb_v4 on a flat-plane layout (a block owns
// kFlatCpt * kThreads consecutive cells of the flattened xy plane, thread t the four
// consecutive cells q0 + 4t .. q0 + 4t + 3, loaded and stored as one vector: the inner
// vectors of a flat-plane snapshot are stored with planes pts = nxy rounded up to a
// multiple of four cells apart), written with per-thread pointers that advance one plane
// per step.  The
// neighbour sum (x-, x+, y-, y+, z-, z+, a wall adding a zero) and the update are
// those of the other sweeps: the same bits.  L is the load policy (Vec4-style
// scalars: plain or L2-coherent).
template <class TS, bool COH>
__device__ __forceinline__ float fld(const TS *p) {
    if constexpr (COH) {
        return ldcg(p, 0);
    } else {
        return ld(p, 0);
    }
}

// Shared segment of a flat-plane tile with padded rows: slot of plane cell q is
// (q / nx - r0) (nx + 1) + q % nx + 1, so every row starts with a pad slot; the pad slots
// and the rows outside the plane are zeroed once and never written, so a wall neighbour
// (x- of x = 0, x+ of x = nx-1 through the next row's pad, y+-1 outside the plane) reads
// +0.0 -- what the other engines add for a wall -- without a test.
constexpr int kFlatSlots = kFlatCpt * kThreads + 4 * kFlatMaxNx + kFlatCpt * kThreads + 8;

// PRED: one step of the shared expansion's recurrence in difference form (see k_pred_v4)
// instead: omega its factor, no r; a wall's neighbour is the cell itself.
template <class TS, bool COH, bool PRED = false>
__device__ __forceinline__ void cheb_flat_tile(const Geo &g, int pts, int chunk, int z0, int z1,
                                               float ce, float gamma, float omega, const float *sdg,
                                               const TS *yv, const TS *ypv, const TS *rv,
                                               TS *ynv) {
    using V = Vec4<TS>;
    using LD = typename std::conditional<COH, Vec4cg<TS>, Vec4<TS>>::type;
    constexpr int C = kFlatCpt;
    constexpr int S = kThreads;   // stride between the halo cells a thread loads
    __shared__ float sp[kFlatSlots];
    const int t = threadIdx.y * TX + threadIdx.x;
    const int nx = g.nx, nxy = g.nxy, nz = g.nz;
    const int P = nx + 1;
    const int q0 = chunk * (C * S);
    const int qt = q0 + C * t;    // this thread's first cell (a multiple of four)
    const int r0 = q0 / nx - 1;   // first row of the segment (may be -1)
    auto slot = [&](int q) {
        const int r = q / nx;
        return (r - r0) * P + (q - r * nx) + 1;
    };
    const int nslots = ((q0 + C * S + nx - 1) / nx + 2 - r0) * P;
    for (int i = t; i < nslots; i += S) sp[i] = 0.0f;
    // per cell j (cell qt + j): its segment slot, and (packed) whether it is in the plane
    // and its number of x/y neighbours
    int so[C];
    unsigned ownm = 0u, nnp = 0u, inl = 0u, inr = 0u, inu = 0u, ind = 0u;
#pragma unroll
    for (int j = 0; j < C; ++j) {
        const int q = qt + j;
        if (q < nxy) ownm |= 1u << j;
        const int iy = q / nx, ix = q - iy * nx;
        nnp |= (unsigned)((ix > 0) + (ix + 1 < nx) + (iy > 0) + (iy + 1 < g.ny)) << (3 * j);
        if (ix > 0) inl |= 1u << j;        // x - 1 is in the row (for j > 0: the thread's cell j - 1)
        if (ix + 1 < nx) inr |= 1u << j;   // x + 1 is in the row (for j < 3: its cell j + 1)
        if (iy > 0) inu |= 1u << j;
        if (iy + 1 < g.ny) ind |= 1u << j;
        so[j] = slot(q);
    }
    auto own = [&](int j) { return (ownm >> j) & 1u; };
    const bool any = ownm != 0u;   // the thread's vector holds cells of the plane
    const int lo0 = max(q0 - nx, 0);
    const int hi0 = q0 + C * S, hi1 = min(hi0 + nx, nxy);
    const bool hl0 = lo0 + t < q0, hl1 = lo0 + t + S < q0;
    const bool hh0 = hi0 + t < hi1, hh1 = hi0 + t + S < hi1;
    const int sl0 = slot(lo0 + t), sl1 = slot(lo0 + t + S);
    const int sh0 = slot(hi0 + t), sh1 = slot(hi0 + t + S);
    // per-thread pointers at plane z (planes are pts apart, a multiple of four cells, so
    // a thread's four cells are one aligned vector); the halo cells relative to ph
    const size_t pz0 = (size_t)z0 * pts;
    const TS *py = yv + pz0 + qt;
    const TS *pp = ypv ? ypv + pz0 + qt : nullptr;
    const TS *pr = PRED ? nullptr : rv + pz0 + qt;
    TS *po = ynv + pz0 + qt;
    const TS *ph = yv + pz0;
    const int dl0 = lo0 + t, dl1 = lo0 + t + S, dh0 = hi0 + t, dh1 = hi0 + t + S;
    float4 vdn = make_float4(0.f, 0.f, 0.f, 0.f), vc = vdn, vup = vdn, yp = vdn, rc = vdn;
    float ha0 = 0.f, ha1 = 0.f, hb0 = 0.f, hb1 = 0.f;
    if (z0 < z1) {
        if (any) {
            if (z0 > 0) vdn = LD::load(py - pts, 0);
            vc = LD::load(py, 0);
            if (z0 + 1 < nz) vup = LD::load(py + pts, 0);
            if (pp) yp = LD::load(pp, 0);
            if constexpr (!PRED) rc = LD::load(pr, 0);
        }
        if (hl0) ha0 = fld<TS, COH>(ph + dl0);
        if (hl1) ha1 = fld<TS, COH>(ph + dl1);
        if (hh0) hb0 = fld<TS, COH>(ph + dh0);
        if (hh1) hb1 = fld<TS, COH>(ph + dh1);
    }
    __syncthreads();   // the zeroed segment before the first plane is published
    for (int z = z0; z < z1; ++z) {
        // loads for plane z+1: y at z+2, y_prev and r at z+1, the halo at z+1
        float4 nup = make_float4(0.f, 0.f, 0.f, 0.f), nyp = nup, nrc = nup;
        float na0 = 0.f, na1 = 0.f, nb0 = 0.f, nb1 = 0.f;
        if (z + 1 < z1) {
            if (any) {
                if (z + 2 < nz) nup = LD::load(py + 2 * pts, 0);
                if (pp) nyp = LD::load(pp + pts, 0);
                if constexpr (!PRED) nrc = LD::load(pr + pts, 0);
            }
            if (hl0) na0 = fld<TS, COH>(ph + pts + dl0);
            if (hl1) na1 = fld<TS, COH>(ph + pts + dl1);
            if (hh0) nb0 = fld<TS, COH>(ph + pts + dh0);
            if (hh1) nb1 = fld<TS, COH>(ph + pts + dh1);
        }
        const float vcs[C] = {vc.x, vc.y, vc.z, vc.w};
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (own(j)) sp[so[j]] = vcs[j];
        if (hl0) sp[sl0] = ha0;
        if (hl1) sp[sl1] = ha1;
        if (hh0) sp[sh0] = hb0;
        if (hh1) sp[sh1] = hb1;
        __syncthreads();
        if (any) {
            const int nnz = (z > 0) + (z + 1 < nz);
            const float vds[C] = {vdn.x, vdn.y, vdn.z, vdn.w}, vus[C] = {vup.x, vup.y, vup.z, vup.w};
            const float yps[C] = {yp.x, yp.y, yp.z, yp.w}, rcs[C] = {rc.x, rc.y, rc.z, rc.w};
            float o[C];
#pragma unroll
            for (int j = 0; j < C; ++j) {
                // a lane beyond the plane computes from the zero slots and its padding
                // values and is stored into the plane's padding, which nothing reads
                // x neighbours inside the thread's vector come from its registers (the same
                // values the segment holds; a row end is a wall, zero as its pad slot)
                const float *c = sp + so[j];
                if constexpr (PRED) {
                    const float v = vcs[j];
                    const float xl = j == 0 ? c[-1] : vcs[j > 0 ? j - 1 : 0];
                    const float xr = j == C - 1 ? c[1] : vcs[j < C - 1 ? j + 1 : j];
                    const float dxl = ((inl >> j) & 1u) ? xl - v : 0.0f, dxr = ((inr >> j) & 1u) ? xr - v : 0.0f;
                    const float dyl = ((inu >> j) & 1u) ? c[-P] - v : 0.0f, dyr = ((ind >> j) & 1u) ? c[P] - v : 0.0f;
                    const float dzl = z > 0 ? vds[j] - v : 0.0f, dzr = z + 1 < nz ? vus[j] - v : 0.0f;
                    const float d = (dxl + dxr) + (dyl + dyr) + (dzl + dzr);
                    o[j] = fmaf(omega, d, pp ? (v - yps[j]) + v : v);
                    continue;
                }
                float sm = j == 0 ? c[-1] : (((inl >> j) & 1u) ? vcs[j - 1] : 0.0f);
                sm += j == C - 1 ? c[1] : (((inr >> j) & 1u) ? vcs[j + 1] : 0.0f);
                sm += c[-P];
                sm += c[P];
                sm += vds[j];
                sm += vus[j];
                const float v = vcs[j];
                const float ay = fmaf(sdg[((nnp >> (3 * j)) & 7u) + nnz], v, -ce * sm);
                o[j] = fmaf(omega, v - yps[j] + gamma * (rcs[j] - ay), yps[j]);
            }
            V::store(po, 0, make_float4(o[0], o[1], o[2], o[3]));
        }
        __syncthreads();
        vdn = vc;
        vc = vup;
        vup = nup;
        yp = nyp;
        rc = nrc;
        ha0 = na0;
        ha1 = na1;
        hb0 = nb0;
        hb1 = nb1;
        py += pts;
        if (pp) pp += pts;
        if constexpr (!PRED) pr += pts;
        po += pts;
        ph += pts;
    }
}

// ---------------------------------------------------------------- batched snapshots
// Many independent snapshots (each its own hex mesh, bandwidth and Chebyshev count) are
// smoothed by one persistent cooperative launch in the double-float modes.  Phases:
// u^0 -> double-float; the first refinement pass of the first pseudo-step; then per
// pseudo-step R rounds of (m_s - 1 Chebyshev iterations, one refinement pass), the last
// of which also starts the next step; a bounded grid barrier after every phase.  Work items (tile x z-chunk x field of one snapshot) are dealt to
// blocks round-robin; a snapshot whose m_s is smaller than the longest idles in the
// remaining Chebyshev phases.  Buffer roles are fixed: the first Chebyshev iterate is
// in Ya and, m_s being even, the correction always ends in Yb; the first round writes X1, later
// rounds alternate X2/X1, and the last round (R >= 2) writes u^{n+1} over u^n in U
// (read there only at the cell itself).  Per-item residual partials of each step's
// last pass (and ||b||^2 partials of its first pass) are stored and reduced afterwards.
// With the shared expansion (pred) a step's first round has no inner solve: its
// refinement pass takes the expansion's increment, formed by k_bpred* launches before
// either schedule starts, and reduces ||b||^2; under implicit Euler no pass then starts
// the next step.
template <class TS>
struct SnapDesc {
    Geo g;
    int gx, gy, zlen, nzc;   // refinement items (scalar engine)
    int v4, gx4, zlen4, nzc4;// Chebyshev items (vectorised if v4)
    int flat, nch, nchr;     // flat-plane items: plane chunks per plane (Chebyshev, refinement)
    int pts;                 // plane pitch of the inner (TS) vectors: nxy, rounded up to a
                             // multiple of four cells on a flat-plane snapshot
    double vcu;              // the cell volume
    int m;                   // Chebyshev iterations per round (even)
    int scheme;
    float gamma;
    Coef32 cf32;
    CoefDF cfdf;
    const double *cells;     // u^0, field-major FP64
    DF *U, *X1, *X2, *B;
    TS *R, *Ya, *Yb;
    const float *omega;      // omega[k], k = 1 .. m-1
    // the shared expansion of the steps' first rounds (see k_pred_combine), where the batch
    // runs it: K steps of the recurrence with factor w, coefficients pc[k * steps + i], the
    // vectors T_k of one field (nz pts values each) and every step's increment D of all
    int K;
    float w;
    const float *pc;
    float *T, *D;
};

struct BItem {
    int snap, bx, by, zf;    // zf = field * nzc + z-chunk
};

__device__ __forceinline__ DF ldcg_df(const DF *p, int i) {
    float2 v = __ldcg(reinterpret_cast<const float2 *>(p + i));
    return DF{v.x, v.y};
}

// Loads of the batched phases: COH (the persistent launch) reads data that other blocks
// of the same launch wrote, so it bypasses L1; one launch per phase reads plainly.
template <bool COH> __device__ __forceinline__ DF bld_df(const DF *p, int i) {
    if constexpr (COH) {
        return ldcg_df(p, i);
    } else {
        return p[i];
    }
}
template <bool COH, class TS> __device__ __forceinline__ float bld(const TS *p, int i) {
    if constexpr (COH) {
        return ldcg(p, i);
    } else {
        return ld(p, i);
    }
}

// part: this item's ||r||^2 partial of a step's last pass (or ||b||^2 of its first pass).
// part_next (a step's last pass, not the call's last step): the pass also starts the next
// step, as the single-mesh path's last refinement pass does: with x = u^{n+1} it has A x at
// hand, so the next first residual is c L x = (x - A x) / theta (and the Crank-Nicolson
// right-hand side x + c/2 L x), and that step's ||b||^2 partial goes to part_next.
template <class TS, bool COH>
__device__ __forceinline__ void batched_refine(const SnapDesc<TS> &d, int nf, const BItem &it, bool first,
                                               int round, int R, double *part, double *part_next,
                                               int pstep = -1, double *part_b = nullptr) {
    // the descriptor lives in global memory: copy what the sweep reads into registers
    // (through a reference every store would force the compiler to reload it)
    const Geo g = d.g;
    const int scheme = d.scheme;
    const DF cf_c = d.cfdf.c, cf_half_c = d.cfdf.half_c, cf_ce = d.cfdf.ce;
    const int f = it.zf / d.nzc;
    const int zc = it.zf - f * d.nzc;
    const int z0 = zc * d.zlen, z1 = min(g.nz, z0 + d.zlen);
    const size_t off = (size_t)f * g.n;                 // the double-float vectors
    const size_t off_ts = (size_t)f * g.nz * d.pts;     // the inner vectors
    float acc = 0.0f, acc_b = 0.0f;
    const float gamma = d.gamma;
    TS *r = d.R + off_ts;
    TS *y1 = d.Ya + off_ts;
    // the flat-plane engine or the 2.5D tile engine (the same arithmetic per cell); load
    // and consume take a cell's index in the double-float and in the inner vectors (the
    // same on the 2.5D engine's snapshots, whose inner planes are nxy apart)
    const bool flat = d.flat != 0;
    const int pts = d.pts;
    auto engine = [&](auto load, auto finish, auto pre, auto consume) {
        if (flat)
            sweep_flat_at<DF, kFlatCptDF>(g, pts, it.bx, z0, z1, load, finish, pre, consume);
        else
            sweep25_lf<DF>(
                g, it.bx, it.by, z0, z1, [&](int k) { return load(k, k); }, finish, pre,
                [&](int k, DF v, DF sm, int nn, decltype(pre(0)) pt) { consume(k, k, v, sm, nn, pt); });
    };
    if (first) {
        const DF *u = d.U + off;
        DF *bo = d.B + off;
        engine(
            [&](int k, int) { return bld_df<COH>(u, k); }, [](DF v) { return v; },
            [](int) { return NoPre{}; },
            [&](int k, int kt, DF v, DF sm, int nn, NoPre) {
                const DF lx = df_lap(sm, v, (float)nn);
                DF bk = v;
                if (scheme == 1) {
                    bk = v + df_mul(cf_half_c, lx);
                    bo[k] = bk;
                }
                float bf = df_f(bk);
                acc = fmaf(bf, bf, acc);
                float rf = df_f(df_mul_un(cf_c, lx));
                st(r, kt, rf);
                st(y1, kt, gamma * rf);
            });
    } else {
        const DF *xin = (round == 1 ? d.U : ((round & 1) ? d.X2 : d.X1)) + off;
        DF *xout = (round == R ? d.U : ((round & 1) ? d.X1 : d.X2)) + off;
        const DF *b = (scheme == 1 ? d.B : d.U) + off;
        DF *bo = d.B + off;
        const TS *dd = d.Yb + off_ts;
        if constexpr (sizeof(TS) == 4)   // the step's first round: the increment from the expansion
            if (pstep >= 0) dd = d.D + (size_t)pstep * nf * g.nz * d.pts + off_ts;
        const bool next = part_next != nullptr, wantb = part_b != nullptr;
        engine(
            [&](int k, int kt) { return DFd{bld_df<COH>(xin, k), bld<COH>(dd, kt)}; },
            [](DFd v) { return df_add_f(v.x, v.d); }, [&](int k) { return bld_df<COH>(b, k); },
            [&](int k, int kt, DF v, DF sm, int nn, DF bk) {
                xout[k] = v;
                const DF lx = df_lap(sm, v, (float)nn);
                float rf = df_f(df_res(bk, v, cf_ce, lx));
                acc = fmaf(rf, rf, acc);
                if (wantb) {
                    const float bf = df_f(bk);
                    acc_b = fmaf(bf, bf, acc_b);
                }
                if (next) {
                    DF cl = df_mul(cf_ce, lx);        // = theta c L v
                    DF bn = v;
                    if (scheme == 1) {
                        bn = v + cl;                  // v + c/2 L v
                        cl = cl + cl;                 // c L v
                        bo[k] = bn;                   // read above at this cell only
                    }
                    const float bf = df_f(bn);
                    acc_b = fmaf(bf, bf, acc_b);
                    rf = df_f(cl);
                }
                st(r, kt, rf);
                st(y1, kt, gamma * rf);
            });
        const double tb = block_sum_f(acc_b);
        if (is_thread0() && next) *part_next = tb;
        if (is_thread0() && wantb) *part_b = tb;
    }
    double tot = block_sum_f(acc);
    if (is_thread0() && part) *part = tot;
}

// The merged pass of k_refine_mid for a flat-plane snapshot: the iterate alternates between U
// (even steps' u_s) and X2, so that no block writes what another still reads.
template <class TS, bool COH>
__device__ __forceinline__ void batched_mid(const SnapDesc<TS> &d, int nf, const BItem &it, int step, bool end,
                                            double *part, double *part_next) {
    const Geo g = d.g;
    const int scheme = d.scheme, pts = d.pts;
    const DF cf_ce = d.cfdf.ce;
    const int f = it.zf / d.nzc;
    const int zc = it.zf - f * d.nzc;
    const int z0 = zc * d.zlen, z1 = min(g.nz, z0 + d.zlen);
    const size_t off = (size_t)f * g.n, off_ts = (size_t)f * g.nz * pts, ds = (size_t)nf * g.nz * pts;
    const DF *u = ((step & 1) ? d.X2 : d.U) + off;
    DF *xout = ((step & 1) ? d.U : d.X2) + off;
    const DF *b = scheme == 1 ? d.B + off : u;
    DF *bo = d.B + off;
    const float *e = d.D + step * ds + off_ts, *en = e + ds;
    const TS *dd = d.Yb + off_ts;
    TS *r = d.R + off_ts, *y1 = d.Ya + off_ts;
    const float gamma = d.gamma;
    float acc = 0.0f, acc_b = 0.0f;
    sweep_flat_at<DFe, kFlatCptDF>(
        g, pts, it.bx, z0, z1,
        [&](int k, int kt) {
            return DFeRaw{bld_df<COH>(u, k), e[kt], bld<COH>(dd, kt), end ? 0.0f : en[kt]};
        },
        [](DFeRaw v) { return DFe{df_add_f(df_add_f(v.u, v.e), v.d), DF{v.en, 0.0f}}; },
        [&](int k) { return bld_df<COH>(b, k); },
        [&](int k, int kt, DFe v, DFe sm, int nn, DF bk) {
            xout[k] = v.x;
            const DF lx = df_lap(sm.x, v.x, (float)nn);
            const float rf = df_f(df_res(bk, v.x, cf_ce, lx));
            acc = fmaf(rf, rf, acc);
            if (!end) {
                const DF le = df_lap(sm.e, v.e, (float)nn);
                DF bn = v.x, m = lx;
                if (scheme == 1) {
                    bn = v.x + df_mul(cf_ce, lx);
                    bo[k] = bn;
                    m = DF{2.0f * lx.hi, 2.0f * lx.lo};
                }
                const float bf = df_f(bn);
                acc_b = fmaf(bf, bf, acc_b);
                const DF t = df_two_sum(m.hi, le.hi);
                const DF q = df_mul_un(cf_ce, DF{t.hi, (m.lo + le.lo) + t.lo});
                const DF w = df_two_sum(-v.e.hi, q.hi);
                const float rn = w.hi + (q.lo + w.lo);
                st(r, kt, rn);
                st(y1, kt, gamma * rn);
            }
        });
    const double tb = block_sum_f(acc_b), tot = block_sum_f(acc);
    if (is_thread0()) {
        *part = tot;
        if (!end) *part_next = tb;
    }
}

template <class TS, bool COH>
__device__ __forceinline__ void batched_cheb(const SnapDesc<TS> &d, const BItem &it, int k) {
    const Geo g = d.g;   // register copies of the descriptor's fields (see batched_refine)
    const float gamma = d.gamma, ce = d.cf32.ce;
    const int nzc = (d.v4 && !d.flat) ? d.nzc4 : d.nzc, zlen = (d.v4 && !d.flat) ? d.zlen4 : d.zlen;
    const int f = it.zf / nzc;
    const int zc = it.zf - f * nzc;
    const int z0 = zc * zlen, z1 = min(g.nz, z0 + zlen);
    const size_t off = (size_t)f * g.nz * d.pts;   // inner vectors: planes pts apart
    // y_k lives in Ya for odd k, in Yb for even k; y_{k+1} overwrites y_{k-1}
    const TS *yc = ((k & 1) ? d.Ya : d.Yb) + off;
    TS *yo = ((k & 1) ? d.Yb : d.Ya) + off;
    const TS *yp = k == 1 ? nullptr : yo;
    const TS *r = d.R + off;
    const float omega = d.omega[k];
    __shared__ float sdg[8];
    stage_table(sdg, d.cf32.dg);
    __syncthreads();
    if (d.flat) {
        cheb_flat_tile<TS, COH>(g, d.pts, it.bx, z0, z1, ce, gamma, omega, sdg, yc, yp, r, yo);
    } else if (d.v4) {
        if constexpr (COH)
            cheb_v4_tile<TS, Vec4cg>(g, it.bx, it.by, z0, z1, d.cf32, sdg, d.gamma, omega, yc, yp, r, yo);
        else
            cheb_v4_tile<TS, Vec4>(g, it.bx, it.by, z0, z1, d.cf32, sdg, d.gamma, omega, yc, yp, r, yo);
    } else {
        sweep25_at<float>(
            g, it.bx, it.by, z0, z1, [&](int q) { return bld<COH>(yc, q); },
            [&](int q) { return float2{yp ? bld<COH>(yp, q) : 0.0f, bld<COH>(r, q)}; },
            [&](int q, float v, float sm, int nn, float2 pt) {
                float ay = fmaf(sdg[nn], v, -d.cf32.ce * sm);
                st(yo, q, fmaf(omega, v - pt.x + d.gamma * (pt.y - ay), pt.x));
            });
    }
}

template <class TS>
__global__ void __launch_bounds__(kThreads, 4) k_batched(const SnapDesc<TS> *__restrict__ sd, int nsnap,
                                                      int nf, const BItem *__restrict__ ritems,
                                                      int nr, const BItem *__restrict__ citems,
                                                      int nc, int nsteps, int R, int mmax, int pred,
                                                      int cn, int mid, double *__restrict__ part_rr,
                                                      double *__restrict__ part_bb, GridBar *gb,
                                                      long long budget) {
    // phase 0: u^0 -> double-float (with the expansion it has run: k_bconvert)
    const size_t tid = (size_t)blockIdx.x * kThreads + threadIdx.y * TX + threadIdx.x;
    const size_t nthr = (size_t)gridDim.x * kThreads;
    for (int s = 0; s < (pred ? 0 : nsnap); ++s) {
        const size_t cnt = (size_t)sd[s].g.n * nf;
        const double *u = sd[s].cells;
        DF *U = sd[s].U;
        for (size_t i = tid; i < cnt; i += nthr) {
            U[i] = df_split(u[i]);
        }
    }
    if (!grid_sync(gb, gridDim.x, budget)) return;
    for (int step = 0; step < nsteps; ++step) {
        if (step == 0 && (!pred || cn)) {   // later steps were started by the previous step's last pass
            for (int i = blockIdx.x; i < nr; i += gridDim.x) {
                const BItem it = ritems[i];
                batched_refine<TS, true>(sd[it.snap], nf, it, true, 0, R, part_bb + i, nullptr);
            }
            if (!grid_sync(gb, gridDim.x, budget)) return;
        }
        for (int round = 1; round <= R; ++round) {
            const bool shared = pred && round == 1;
            if (shared && mid && step > 0) continue;   // the merged pass has started the step
            for (int k = 1; k < (shared ? 1 : mmax); ++k) {
                for (int i = blockIdx.x; i < nc; i += gridDim.x) {
                    const BItem it = citems[i];
                    if (k < sd[it.snap].m) batched_cheb<TS, true>(sd[it.snap], it, k);
                }
                if (!grid_sync(gb, gridDim.x, budget)) return;
            }
            for (int i = blockIdx.x; i < nr; i += gridDim.x) {
                const BItem it = ritems[i];
                if constexpr (sizeof(TS) == 4)
                    if (mid && round == R) {
                        batched_mid<TS, true>(sd[it.snap], nf, it, step, step + 1 == nsteps,
                                              part_rr + (size_t)step * nr + i,
                                              part_bb + (size_t)(step + 1 < nsteps ? step + 1 : step) * nr + i);
                        continue;
                    }
                batched_refine<TS, true>(sd[it.snap], nf, it, false, round, R,
                                   round == R ? part_rr + (size_t)step * nr + i : nullptr,
                                   round == R && step + 1 < nsteps && (!pred || cn)
                                       ? part_bb + (size_t)(step + 1) * nr + i
                                       : nullptr,
                                   shared ? step : -1,
                                   shared && !cn ? part_bb + (size_t)step * nr + i : nullptr);
            }
            if (step + 1 < nsteps || round < R)
                if (!grid_sync(gb, gridDim.x, budget)) return;
        }
    }
}

// The same schedule as k_batched with one launch per phase (the phased schedule): the
// launch boundary orders the phases, so there is no grid barrier, loads may use L1, and
// the hardware deals the work items (block i takes item i) to the SMs as they free up.
// A captured graph holds the whole sequence of launches.
template <class TS>
__global__ void __launch_bounds__(kThreads, 4) k_bconvert(const SnapDesc<TS> *__restrict__ sd, int nf) {
    chain_wait();
    chain_release();
    const SnapDesc<TS> &d = sd[blockIdx.y];
    const size_t cnt = (size_t)d.g.n * nf;
    const size_t tid = (size_t)blockIdx.x * kThreads + threadIdx.y * TX + threadIdx.x;
    for (size_t i = tid; i < cnt; i += (size_t)gridDim.x * kThreads) {
        d.U[i] = df_split(d.cells[i]);
    }
}

template <class TS>
__global__ void __launch_bounds__(kThreads, 3) k_bcheb(const SnapDesc<TS> *__restrict__ sd,
                                                    const BItem *__restrict__ citems, int k) {
    chain_wait();
    chain_release();
    const BItem it = citems[blockIdx.x];
    if (k < sd[it.snap].m) batched_cheb<TS, false>(sd[it.snap], it, k);
}

// first: a step's first pass (||b||^2 partial to part[i]); else round `round` of R
// (||r||^2 partial to part[i] when part, the next step's ||b||^2 to part_next[i]).
template <class TS>
__global__ void __launch_bounds__(kThreads, 3) k_brefine(const SnapDesc<TS> *__restrict__ sd, int nf,
                                                      const BItem *__restrict__ ritems, int first,
                                                      int round, int R, double *part,
                                                      double *part_next, int pstep, double *part_b) {
    chain_wait();
    chain_release();
    const int i = blockIdx.x;
    const BItem it = ritems[i];
    batched_refine<TS, false>(sd[it.snap], nf, it, first != 0, round, R, part ? part + i : nullptr,
                              part_next ? part_next + i : nullptr, pstep, part_b ? part_b + i : nullptr);
}

// A merged pass of every snapshot (see batched_mid).  64 snapshots x 5 fields: 1.49 ms at 128
// registers (2.6 TB/s, latency) in the place of two k_brefine passes of 1.00 ms each; the call 5
// ms less.
template <class TS>
__global__ void __launch_bounds__(kThreads, 2) k_bmid(const SnapDesc<TS> *__restrict__ sd, int nf,
                                                    const BItem *__restrict__ ritems, int step, int end,
                                                    double *part, double *part_next) {
    chain_wait();
    chain_release();
    const int i = blockIdx.x;
    const BItem it = ritems[i];
    batched_mid<TS, false>(sd[it.snap], nf, it, step, end != 0, part + i, part_next + i);
}

// The shared expansion of a batch, one field of every snapshot at a time (so that the
// vectors T_k take the room of one field): T_0, the recurrence's step k, the combination.
// 64 snapshots of 32 to 96 cells a side, 5 fields, b = 3 dx, 10 steps: 29 recurrence steps of
// 80 us per field (3.3 TB/s: the flat tile's barriers and neighbour tests) and 0.9 ms per
// combination (4.0 TB/s) take the place of 130 k_bcheb launches of 335 us; the call, with the
// merged pass, 112 -> 86.5 ms.
template <class TS>
__global__ void __launch_bounds__(kThreads) k_bpred_start(const SnapDesc<TS> *__restrict__ sd, int f) {
    chain_wait();
    chain_release();
    const SnapDesc<TS> &d = sd[blockIdx.y];
    const int n = d.g.n, nxy = d.g.nxy, pad = d.pts - nxy;
    const DF *u = d.U + (size_t)f * n;
    float *t = d.T;
    for (int i = blockIdx.x * kThreads + threadIdx.x; i < n; i += gridDim.x * kThreads)
        t[i + (pad ? i / nxy * pad : 0)] = u[i].hi;
}

template <class TS>
__global__ void __launch_bounds__(kThreads, 4) k_bpred(const SnapDesc<TS> *__restrict__ sd,
                                                    const BItem *__restrict__ items, int k) {
    chain_wait();
    chain_release();
    const BItem it = items[blockIdx.x];
    const SnapDesc<TS> &d = sd[it.snap];
    if (k >= d.K) return;
    const Geo g = d.g;
    const int z0 = it.zf * d.zlen, z1 = min(g.nz, z0 + d.zlen);
    const size_t stride = (size_t)g.nz * d.pts;
    const float *t = d.T + k * stride;
    cheb_flat_tile<float, false, true>(g, d.pts, it.bx, z0, z1, 0.f, 0.f, k ? 2.0f * d.w : d.w, nullptr, t,
                                       k ? t - stride : nullptr, nullptr, d.T + (k + 1) * stride);
}

// k_pred_combine for one field of every snapshot (blockIdx.y); the coefficients differ per
// snapshot and come through shared memory.
template <class TS, int NS>
__global__ void __launch_bounds__(kThreads) k_bpred_combine(const SnapDesc<TS> *__restrict__ sd, int nf, int f,
                                                            int steps) {
    chain_wait();
    chain_release();
    __shared__ float a[(kPredMaxK + 1) * NS];
    const SnapDesc<TS> &d = sd[blockIdx.y];
    const int K = d.K;
    const float *pc = d.pc;
    for (int i = threadIdx.x; i < (K + 1) * NS; i += kThreads) {
        const int k = i / NS, q = i - k * NS;
        a[i] = q < steps ? pc[k * steps + q] : 0.0f;
    }
    __syncthreads();
    const size_t stride = (size_t)d.g.nz * d.pts, dstride = stride * nf;
    const float *t = d.T;
    float *o = d.D + (size_t)f * stride;
    for (size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x; i < stride / 4; i += (size_t)gridDim.x * kThreads) {
        float2 lo[NS], hi[NS];
#pragma unroll
        for (int q = 0; q < NS; ++q) lo[q] = hi[q] = make_float2(0.f, 0.f);
        const float *tp = t + 4 * i;
#pragma unroll 4
        for (int k = 0; k <= K; ++k, tp += stride) {
            const float4 v = *reinterpret_cast<const float4 *>(tp);
            const float2 va = make_float2(v.x, v.y), vb = make_float2(v.z, v.w);
#pragma unroll
            for (int q = 0; q < NS; ++q) {
                const float w = a[k * NS + q];
                lo[q] = fma2(va, make_float2(w, w), lo[q]);
                hi[q] = fma2(vb, make_float2(w, w), hi[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < NS; ++q)
            if (q < steps)
                *reinterpret_cast<float4 *>(o + q * dstride + 4 * i) = make_float4(lo[q].x, lo[q].y, hi[q].x, hi[q].y);
    }
}

// hist[(step * nsnap + s) * nf + f] = (sum of ||r||^2 partials, sum of ||b||^2 partials)
// over the snapshot-field's items, in item order.  One block per (step, s, f).  A step
// whose ||r||^2 exceeds tol2 ||b||^2 (or is not a number) increments *bad.
__global__ void k_batched_hist(const int *__restrict__ first_item, int nsnap, int nf, int nr,
                               const double *__restrict__ part_rr,
                               const double *__restrict__ part_bb, double2 *__restrict__ hist,
                               double tol2, unsigned int *bad) {
    const int sf = blockIdx.x % (nsnap * nf);
    const int step = blockIdx.x / (nsnap * nf);
    const int i0 = first_item[sf], i1 = first_item[sf + 1];
    double a = 0.0, b = 0.0;
    for (int i = i0 + threadIdx.x; i < i1; i += kThreads) {
        a += part_rr[(size_t)step * nr + i];
        b += part_bb[(size_t)step * nr + i];
    }
    double A = block_sum(a), B = block_sum(b);
    if (threadIdx.x == 0) {
        hist[blockIdx.x] = make_double2(A, B);
        if (!(A <= tol2 * B)) atomicAdd(bad, 1u);
    }
}

// u^{n} -> the caller's FP64 arrays, only when every step of every snapshot-field met
// the tolerance (otherwise the inputs stay intact for a run with more rounds).
template <class TS>
__global__ void k_batched_final(const SnapDesc<TS> *__restrict__ sd, int nf, double *const *cells,
                                const unsigned int *__restrict__ bad, int in_x2) {
    if (*bad != 0u) return;
    const SnapDesc<TS> &d = sd[blockIdx.y];
    const size_t cnt = (size_t)d.g.n * nf;
    double *out = cells[blockIdx.y];
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < cnt;
         i += (size_t)gridDim.x * blockDim.x) {
        const DF v = in_x2 ? d.X2[i] : d.U[i];
        out[i] = df_join(v.hi, v.lo);
    }
}

// sum_k V_c u_k of every snapshot's field (the caller's FP64 arrays): one block per
// (snapshot, field), out[s * nf + f]
template <class TS>
__global__ void k_mass_batched(const SnapDesc<TS> *__restrict__ sd, int nf, double *__restrict__ out) {
    const int s = blockIdx.x / nf, f = blockIdx.x - s * nf;
    const SnapDesc<TS> &d = sd[s];
    const int n = d.g.n;
    const double *u = d.cells + (size_t)f * n;
    const double vcu = d.vcu;
    double acc = 0.0;
    for (int k = threadIdx.x; k < n; k += kThreads) acc += vcu * u[k];
    const double v = block_sum(acc);
    if (threadIdx.x == 0) out[blockIdx.x] = v;
}

// sum_k V_k u_k per field (any mesh).  Few blocks of many cells each: a block's FP64 reduction and the
// last block's sum of the partials cost more than its cells on a small mesh (GB300 issues a
// warp's FP64 instruction in 16 cycles).
__global__ void k_mass(int n, const double *__restrict__ u_all, const double *__restrict__ vc,
                       double vcu, double *__restrict__ partials_all, unsigned int *tickets,
                       double *__restrict__ out) {
    const int f = blockIdx.y;
    const double *u = u_all + (size_t)f * n;
    double s = 0.0;
    grid_stride<8>(
        n, blockIdx.x * kThreads + threadIdx.x, gridDim.x * kThreads,
        [&](uint32_t k, uint32_t step) {   // eight cells in flight
            double x[8], v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                x[j] = u[k + j * step];
                v[j] = vc ? vc[k + j * step] : vcu;
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) s += v[j] * x[j];
        },
        [&](uint32_t k) { s += (vc ? vc[k] : vcu) * u[k]; });
    double v = block_sum(s);
    double *partials = partials_all + (size_t)f * gridDim.x;
    if (arrive(partials, 1, &v, blockIdx.x, gridDim.x, &tickets[f])) {
        double S = finish_sum(partials, 0, gridDim.x);
        if (is_thread0()) {
            out[f] = S;
            tickets[f] = 0;
        }
    }
}

inline size_t align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

int stencil_grid(int n) {
    int b = (n + kThreads - 1) / kThreads;
    int cap = num_sms() * 8;
    return b < cap ? (b < 1 ? 1 : b) : cap;
}

// The double-float vectors of a mesh are in the pair layout of the two-cells-per-thread
// refinement kernel when that kernel runs (nx even, no periodic axis but x), else one
// (hi, lo) per cell.  Conversions of n values (all fields) in the layout of geometry g:
inline bool df_pairs(const Geo &g) { return g.nx % 2 == 0 && (g.per & ~1) == 0; }
inline void launch_to_df(const Geo &g, size_t n, const double *u, DF *x, cudaStream_t st) {
    if (df_pairs(g))
        k_to_df_pairs<<<stencil_grid((int)(n / 2)), kThreads, 0, st>>>(n / 2, u, reinterpret_cast<float4 *>(x));
    else
        k_to_df<<<stencil_grid((int)n), kThreads, 0, st>>>(n, u, x);
}
inline void launch_from_df(const Geo &g, size_t n, const DF *x, double *u, cudaStream_t st) {
    if (df_pairs(g))
        k_from_df_pairs<<<stencil_grid((int)(n / 2)), kThreads, 0, st>>>(
            n / 2, reinterpret_cast<const float4 *>(x), u);
    else
        k_from_df<<<stencil_grid((int)n), kThreads, 0, st>>>(n, x, u);
}

// Blocks of a cooperative launch: all must be co-resident (at most 4 per SM here).
template <class K> int coop_blocks(K kernel) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0) != cudaSuccess)
        per_sm = 1;
    per_sm = per_sm < 1 ? 1 : (per_sm > 4 ? 4 : per_sm);
    return per_sm * num_sms();
}

// Work items (xy tile x z-chunk x field) for a persistent sweep over G blocks.
struct Items {
    int gx, gy, zlen, nzc, n;
};
Items make_items(const Geo &g, int nf, int G) {
    Items it;
    it.gx = (g.nx + TX - 1) / TX;
    it.gy = (g.ny + TY - 1) / TY;
    long long cols = (long long)it.gx * it.gy * nf;
    int nzc = (int)((G + cols - 1) / cols);
    if (nzc < 1) nzc = 1;
    it.zlen = (g.nz + nzc - 1) / nzc;
    it.nzc = (g.nz + it.zlen - 1) / it.zlen;
    it.n = (int)(cols * it.nzc);
    return it;
}

DF split(double v) {
    float hi = (float)v;
    return DF{hi, (float)(v - (double)hi)};
}

CoefDF coefdf(double c, double ce) {
    CoefDF k;
    k.c = split(c);
    k.half_c = split(0.5 * c);
    k.ce = split(ce);
    for (int q = 0; q < 7; ++q) k.dg[q] = split(1.0 + ce * q);
    return k;
}

Coef64 coef64(double ce) {
    Coef64 c;
    c.ce = ce;
    for (int q = 0; q < 7; ++q) c.dg[q] = 1.0 + ce * q;
    return c;
}

Coef32 coef32(double ce) {
    Coef32 c;
    c.ce = (float)ce;
    for (int q = 0; q < 7; ++q) c.dg[q] = (float)(1.0 + ce * q);
    return c;
}

// ---------------------------------------------------------------- TMA-staged sweep
// The vectorised Chebyshev iteration with its planes staged by the Tensor Memory
// Accelerator: one thread issues, per plane, 2D tile copies (cp.async.bulk.tensor) of
// y_k with a one-row and four-column halo (136 x 10 floats), y_{k-1} and r (128 x 8
// each) into a ring of kTmaStages shared-memory stages, each completing on its own
// mbarrier; the block reads planes z-1, z and z+1 of y_k from the ring, so no thread
// spends registers or address arithmetic on prefetching.  Cells outside the mesh come
// back as zeros from the copy (zero flux: they add nothing and are not counted).  The
// arithmetic is the vectorised tile's, term for term, so the results are the same bits.
// Waits are bounded by `budget` clock cycles; a wait that gives up sets *err and the
// block finishes without its copies in flight.
constexpr int kTmaStages = 4;
constexpr int kTmaW = 4 * TX + 8;                              // 136 floats per halo row
constexpr int kTmaYBytes = (TY + 2) * kTmaW * 4;               // 5440
constexpr int kTmaYSlot = (kTmaYBytes + 127) / 128 * 128;      // 5504
constexpr int kTmaTBytes = TY * 4 * TX * 4;                    // 4096 (y_{k-1}, r)
constexpr int kTmaStageBytes = kTmaYSlot + 2 * kTmaTBytes;     // 13696
constexpr int kTmaSmem = kTmaStages * kTmaStageBytes;          // 54784

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void tma_load4(unsigned dst, const CUtensorMap *map, int c0, int c1, int c2,
                                          int c3, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(dst), "l"(reinterpret_cast<unsigned long long>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, long long budget) {
    const long long t0 = clock64();
    for (;;) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > budget) return false;
    }
}

__global__ void __launch_bounds__(kThreads, 4) k_cheb_tma(Geo g, int zlen, int nzc, Coef32 cf, float gamma,
                                                       float omega, const __grid_constant__ CUtensorMap ty_map,
                                                       const __grid_constant__ CUtensorMap tp_map,
                                                       const __grid_constant__ CUtensorMap tr_map, int has_yp,
                                                       float *ynext_all, int *err, long long budget) {
    chain_wait();
    chain_release();
    extern __shared__ __align__(128) unsigned char tma_smem[];
    __shared__ __align__(8) unsigned long long bar[kTmaStages];
    __shared__ float sdg[8];
    __shared__ int abort_flag;
    const int f = nzc == (int)gridDim.z ? 0 : (int)blockIdx.z / nzc;
    const int z0 = ((int)blockIdx.z - f * nzc) * zlen;
    const int z1 = min(g.nz, z0 + zlen);
    const int tx = threadIdx.x, ty = threadIdx.y;
    const bool leader = tx == 0 && ty == 0;
    const int x0 = blockIdx.x * (4 * TX), yb0 = blockIdx.y * TY;
    const int x = x0 + 4 * tx, y = yb0 + ty;
    const bool own = (x < g.nx) && (y < g.ny);
    const int nyb = (y > 0) + (y + 1 < g.ny);
    const int n0 = nyb + (x > 0) + 1, n3 = nyb + 1 + (x + 4 < g.nx), n12 = nyb + 2;
    const unsigned sbase = smem_u32(tma_smem), bbase = smem_u32(bar);
    const int nload = (z1 - z0) + 2;   // planes z0-1 .. z1 (outside the mesh: zeros)
    const unsigned tbytes = kTmaYBytes + (has_yp ? 2 : 1) * kTmaTBytes;
    if (leader) {
        for (int s = 0; s < kTmaStages; ++s)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bbase + 8 * s) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        abort_flag = 0;
    }
    stage_table(sdg, cf.dg);
    __syncthreads();
    // plane z0 - 1 + j into stage j % kTmaStages (leader only)
    auto issue = [&](int j) {
        const int st = j % kTmaStages, p = z0 - 1 + j;
        const unsigned b = bbase + 8 * st, d = sbase + st * kTmaStageBytes;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(tbytes) : "memory");
        tma_load4(d, &ty_map, x0 - 4, yb0 - 1, p, f, b);
        if (has_yp) tma_load4(d + kTmaYSlot, &tp_map, x0, yb0, p, f, b);
        tma_load4(d + kTmaYSlot + kTmaTBytes, &tr_map, x0, yb0, p, f, b);
    };
    int issued = 0;
    if (leader)
        for (; issued < min(kTmaStages, nload); ++issued) issue(issued);
    int waited = 0;   // stages this thread has waited for
    bool ok = true;
    auto wait_upto = [&](int j) {   // planes up to j have landed
        for (; waited <= j; ++waited)
            if (ok && !mbar_wait(bbase + 8 * (waited % kTmaStages), (waited / kTmaStages) & 1, budget)) {
                ok = false;
                atomicExch(err, 1);
                abort_flag = 1;
            }
    };
    for (int i = 0; i < z1 - z0; ++i) {
        const int z = z0 + i;
        wait_upto(i + 2);
        const float *ym = reinterpret_cast<const float *>(tma_smem + (i % kTmaStages) * kTmaStageBytes);
        const unsigned char *cur = tma_smem + ((i + 1) % kTmaStages) * kTmaStageBytes;
        const float *yc = reinterpret_cast<const float *>(cur);
        const float *yq = reinterpret_cast<const float *>(tma_smem + ((i + 2) % kTmaStages) * kTmaStageBytes);
        const float *tp = reinterpret_cast<const float *>(cur + kTmaYSlot);
        const float *tr = reinterpret_cast<const float *>(cur + kTmaYSlot + kTmaTBytes);
        const int c = 4 + 4 * tx;   // this thread's first cell in a halo row
        const float4 vc = *reinterpret_cast<const float4 *>(yc + (ty + 1) * kTmaW + c);
        const float4 vdn = *reinterpret_cast<const float4 *>(ym + (ty + 1) * kTmaW + c);
        const float4 vup = *reinterpret_cast<const float4 *>(yq + (ty + 1) * kTmaW + c);
        const float4 up = *reinterpret_cast<const float4 *>(yc + ty * kTmaW + c);
        const float4 dn = *reinterpret_cast<const float4 *>(yc + (ty + 2) * kTmaW + c);
        const float4 ypc = has_yp ? *reinterpret_cast<const float4 *>(tp + ty * 4 * TX + 4 * tx) : f4zero();
        const float4 rc = *reinterpret_cast<const float4 *>(tr + ty * 4 * TX + 4 * tx);
        float left = __shfl_up_sync(0xffffffffu, vc.w, 1);
        float right = __shfl_down_sync(0xffffffffu, vc.x, 1);
        if (tx == 0) left = yc[(ty + 1) * kTmaW + 3];
        if (tx == TX - 1) right = yc[(ty + 1) * kTmaW + c + 4];
        if (own && ok) {
            const int nz_ = (z > 0) + (z + 1 < g.nz);
            const float d0 = sdg[n0 + nz_], d12 = sdg[n12 + nz_], d3 = sdg[n3 + nz_];
            float4 s4;
            s4.x = left + vc.y + up.x + dn.x + vdn.x + vup.x;
            s4.y = vc.x + vc.z + up.y + dn.y + vdn.y + vup.y;
            s4.z = vc.y + vc.w + up.z + dn.z + vdn.z + vup.z;
            s4.w = vc.z + right + up.w + dn.w + vdn.w + vup.w;
            float4 o;
            o.x = fmaf(omega, vc.x - ypc.x + gamma * (rc.x - fmaf(d0, vc.x, -cf.ce * s4.x)), ypc.x);
            o.y = fmaf(omega, vc.y - ypc.y + gamma * (rc.y - fmaf(d12, vc.y, -cf.ce * s4.y)), ypc.y);
            o.z = fmaf(omega, vc.z - ypc.z + gamma * (rc.z - fmaf(d12, vc.z, -cf.ce * s4.z)), ypc.z);
            o.w = fmaf(omega, vc.w - ypc.w + gamma * (rc.w - fmaf(d3, vc.w, -cf.ce * s4.w)), ypc.w);
            *reinterpret_cast<float4 *>(ynext_all + (size_t)f * g.n + (size_t)y * g.nx + x +
                                        (size_t)z * g.nxy) = o;
        }
        __syncthreads();   // stage i is no longer read: refill it with plane i + kTmaStages
        if (abort_flag) break;
        if (leader && issued < nload) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue(issued++);
        }
    }
    if (abort_flag && leader)   // let the copies still in flight land before the block ends
        for (int j = max(0, issued - kTmaStages); j < issued; ++j)
            mbar_wait(bbase + 8 * (j % kTmaStages), (j / kTmaStages) & 1, budget);
}

// Tensor maps of the TMA-staged sweep: a field-major [nf][nz][ny][nx] FP32 array as a 4D
// tensor (x fastest), box 136 x 10 (halo) or 128 x 8 (tile), zeros outside.
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn tma_encoder() {
    // looked up once per process (a function-local static is initialised exactly once,
    // also when several library threads get here together)
    static const EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return (EncodeTiledFn)p;
        cudaGetLastError();
        return nullptr;
    }();
    return fn;
}

bool tma_sweep_fits(const Geo &g) { return g.nx % 4 == 0 && g.per == 0 && tma_encoder() != nullptr; }

bool tma_map(CUtensorMap *map, const Geo &g, int nf, const float *base, bool halo) {
    const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)nf};
    const cuuint64_t strides[3] = {(cuuint64_t)g.nx * 4, (cuuint64_t)g.nxy * 4, (cuuint64_t)g.n * 4};
    const cuuint32_t box[4] = {halo ? (cuuint32_t)kTmaW : (cuuint32_t)(4 * TX), halo ? (cuuint32_t)(TY + 2) : (cuuint32_t)TY,
                               1, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return tma_encoder()(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float *>(base), dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

__device__ int g_tma_err;   // set by a TMA-staged sweep whose wait gave up (one word per device:
                            // concurrent problems share it, so any of them may report it)
constexpr long long kTmaBudget = 4000000000LL;   // clock cycles (about two seconds)

// Chebyshev iteration count for a residual reduction eps on spectrum [1, lmax].
int cheb_iters(double lmax, double eps) {
    if (lmax <= 1.0 + 1e-12) return 1;
    double kappa = lmax;
    double rho = (std::sqrt(kappa) - 1.0) / (std::sqrt(kappa) + 1.0);
    int m = (int)std::ceil(std::log(2.0 * std::sqrt(kappa) / eps) / std::log(1.0 / rho));
    return m < 1 ? 1 : (m > 400 ? 400 : m);
}

// One launch of the TMA-staged sweep (FP32 storage): zlen planes per block.  The tensor
// maps are encoded for this launch's buffers (inside a captured graph they are part of
// the recorded parameters).  A map that cannot be encoded runs the vectorised kernel,
// which computes the same bits.
// Per host thread: the device address of the error word, once the kernel's shared
// memory limit is raised (tma_prepare, called before any stream capture).
static thread_local int *t_tma_errp = nullptr;
void tma_prepare() {
    if (t_tma_errp) return;
    int *p = nullptr;
    if (cudaFuncSetAttribute(k_cheb_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, kTmaSmem) == cudaSuccess &&
        cudaGetSymbolAddress((void **)&p, g_tma_err) == cudaSuccess)
        t_tma_errp = p;
    else
        cudaGetLastError();
}

template <class TS>
void launch_cheb_tma(int zlen, const Geo &g, int nf, const Coef32 &cf, float gamma, float omega,
                     const TS *y, const TS *yp, const TS *r, TS *yn, cudaStream_t st) {
    const int nzc = (g.nz + zlen - 1) / zlen;
    const dim3 grid((g.nx + 4 * TX - 1) / (4 * TX), (g.ny + TY - 1) / TY, nzc * nf);
    if constexpr (std::is_same<TS, float>::value) {
        int *errp = t_tma_errp;
        CUtensorMap my, mp, mr;
        if (errp && tma_sweep_fits(g) && tma_map(&my, g, nf, y, true) && tma_map(&mr, g, nf, r, false) &&
            tma_map(&mp, g, nf, yp ? yp : r, false)) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = grid;
            cfg.blockDim = dim3(TX, TY);
            cfg.dynamicSmemBytes = kTmaSmem;
            cfg.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
            at[0].val.programmaticStreamSerializationAllowed = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            cudaLaunchKernelEx(&cfg, k_cheb_tma, g, zlen, nzc, cf, gamma, omega, my, mp, mr, yp ? 1 : 0,
                               (float *)yn, errp, kTmaBudget);
            return;
        }
    }
    launch_chain(k_cheb_v4<TS>, grid, dim3(TX, TY), st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
}

// The TMA wait error word: returns (and clears) whether a TMA-staged sweep gave up a wait.
bool tma_wait_failed(cudaStream_t st) {
    int h = 0;
    if (cudaMemcpyFromSymbolAsync(&h, g_tma_err, sizeof(int), 0, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (h) {
        const int zero = 0;
        cudaMemcpyToSymbolAsync(g_tma_err, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, st);
        cudaStreamSynchronize(st);
    }
    return h != 0;
}

// One Chebyshev iteration launch in a tuned shape: code > 0 = register-blocked engine
// with ZB = code planes per block, code < 0 = z-marching engine with -code planes per
// block.
template <class TS>
void launch_cheb(int code, const Geo &g, int nf, const Coef32 &cf, float gamma, float omega,
                 const TS *y, const TS *yp, const TS *r, TS *yn, cudaStream_t st) {
    const dim3 blk(TX, TY);
    const int gx = (g.nx + TX - 1) / TX, gy = (g.ny + TY - 1) / TY;
    if (code >= kTmaCode) {
        launch_cheb_tma<TS>(code - kTmaCode, g, nf, cf, gamma, omega, y, yp, r, yn, st);
    } else if (code >= 100) {
        const int zlen = code - 100;
        const int nzc = (g.nz + zlen - 1) / zlen;
        const dim3 grid((g.nx + 4 * TX - 1) / (4 * TX), gy, nzc * nf);
        if (g.per && zlen == 4)
            launch_chain(k_cheb_v4<TS, 4, true>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else if (g.per && zlen == 2)
            launch_chain(k_cheb_v4<TS, 2, true>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else if (g.per)   // periodic axes: the wrapping variant
            launch_chain(k_cheb_v4<TS, 0, true>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else if (zlen == 1)
            launch_chain(k_cheb_v4<TS, 1>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else if (zlen == 2)
            launch_chain(k_cheb_v4<TS, 2>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else if (zlen == 4)
            launch_chain(k_cheb_v4<TS, 4>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
        else
            launch_chain(k_cheb_v4<TS>, grid, blk, st, g, zlen, nzc, cf, gamma, omega, y, yp, r, yn);
    } else if (code > 0) {
        const int nzb = (g.nz + code - 1) / code;
        const dim3 grid(gx, gy, nzb * nf);
        if (code == 2) launch_chain(k_cheb_zb<2, TS>, grid, blk, st, g, nzb, cf, gamma, omega, y, yp, r, yn);
        else if (code == 4) launch_chain(k_cheb_zb<4, TS>, grid, blk, st, g, nzb, cf, gamma, omega, y, yp, r, yn);
        else launch_chain(k_cheb_zb<8, TS>, grid, blk, st, g, nzb, cf, gamma, omega, y, yp, r, yn);
    } else {
        const Sweep sw = make_sweep_z(g, nf, -code);
        k_cheb<TS><<<sw.grid, blk, 0, st>>>(g, sw.zlen, sw.nzc, cf, gamma, omega, y, yp, r, yn);
    }
}

// Chebyshev iterations k and k+1 in one launch (k_cheb2_v4): zlen planes per block.
inline bool cheb2_fits(const Geo &g) {
    return g.nx % 4 == 0 && g.nx <= kRowsMaxNx && (g.per & ~1) == 0;   // periodic: x only
}

// The shared-memory limit of the long-row pair kernel, raised before any stream capture
// that may launch it (a host call outside the stream; cheap, so it is simply repeated).
template <class TS> cudaError_t rows_prepare() {
    cudaError_t e = cudaSuccess;
    auto raise = [&](auto kernel, int W) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)rows_smem<TS>(W, kRowsThreads / W - 2));
    };
    raise(k_cheb2_rows<TS, 32>, 32);
    raise(k_cheb2_rows<TS, 64>, 64);
    raise(k_cheb2_rows<TS, 96>, 96);
    raise(k_cheb2_rows<TS, 128>, 128);
    return e;
}

// One launch of two iterations: rows of at most 128 cells as one warp each (k_cheb2_v4),
// longer rows (up to 512 cells) and x-periodic meshes as whole-row blocks with staged
// planes (k_cheb2_rows).
template <class TS>
void launch_cheb2(int zlen, const Geo &g, int nf, const Coef32 &cf, float gamma, float om1,
                  float om2, const TS *yk, const TS *ykm, const TS *r, TS *yc, TS *yd,
                  cudaStream_t st) {
    zlen = std::max(1, std::min(zlen, g.nz));
    const int nzc = (g.nz + zlen - 1) / zlen;
    if (g.nx <= 128 && g.per == 0) {
        const dim3 grid(1, (g.ny + TY2 - 1) / TY2, nzc * nf);
        launch_chain(k_cheb2_v4<TS>, grid, dim3(32, TY2 + 2), st, g, zlen, nzc, cf, gamma, om1, om2,
                     yk, ykm, r, yc, yd);
        return;
    }
    const int W = rows_width(g.nx), tyr = rows_per_block(g.nx);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, (g.ny + tyr - 1) / tyr, nzc * nf);
    cfg.blockDim = dim3(W, tyr + 2);
    cfg.dynamicSmemBytes = rows_smem<TS>(W, tyr);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    switch (W) {
    case 32: cudaLaunchKernelEx(&cfg, k_cheb2_rows<TS, 32>, g, zlen, nzc, cf, gamma, om1, om2, yk, ykm, r, yc, yd); break;
    case 64: cudaLaunchKernelEx(&cfg, k_cheb2_rows<TS, 64>, g, zlen, nzc, cf, gamma, om1, om2, yk, ykm, r, yc, yd); break;
    case 96: cudaLaunchKernelEx(&cfg, k_cheb2_rows<TS, 96>, g, zlen, nzc, cf, gamma, om1, om2, yk, ykm, r, yc, yd); break;
    default: cudaLaunchKernelEx(&cfg, k_cheb2_rows<TS, 128>, g, zlen, nzc, cf, gamma, om1, om2, yk, ykm, r, yc, yd); break;
    }
}

// The m-1 Chebyshev iterations of a round from y1 (y_0 = 0), two per launch; a last odd
// iteration runs alone in the vectorised sweep (code 100 + zlen).  Four buffers rotate:
// each pair launch writes its two iterates to the two buffers it does not read.
// `pool` holds y1's buffer first and three spares; returns the buffer holding y_m.
template <class TS>
TS *cheb_pairs(int zlen, const Geo &g, int nf, const Coef32 &cf, float gamma, double sigma, int m,
               TS *const pool[4], const TS *r, cudaStream_t st) {
    TS *cur = pool[0], *prev = nullptr;
    double om = 1.0;
    auto omega_next = [&](int k) {
        if (sigma > 0.0)
            om = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma * sigma))
                          : 1.0 / (1.0 - om / (4.0 * sigma * sigma));
        return (float)om;
    };
    int k = 1;
    while (k < m) {
        if (k + 1 < m) {
            const float o1 = omega_next(k), o2 = omega_next(k + 1);
            TS *n1 = nullptr, *n2 = nullptr;
            for (int i = 0; i < 4; ++i) {
                if (pool[i] == cur || pool[i] == prev) continue;
                if (!n1) n1 = pool[i];
                else if (!n2) n2 = pool[i];
            }
            CGK_LAUNCH_UNTIMED(st, launch_cheb2<TS>(zlen, g, nf, cf, gamma, o1, o2, cur, prev, r,
                                                    n1, n2, st));
            prev = n1;
            cur = n2;
            k += 2;
        } else {
            const float o1 = omega_next(k);
            TS *yn = prev;
            if (!yn)
                for (int i = 0; i < 4 && !yn; ++i)
                    if (pool[i] != cur) yn = pool[i];
            CGK_LAUNCH_UNTIMED(st, launch_cheb<TS>(100 + zlen, g, nf, cf, gamma, o1, cur, prev, r,
                                                   yn, st));
            prev = cur;
            cur = yn;
            k += 1;
        }
    }
    return cur;
}

// A double-float refinement pass of mode kMode: the two-cells-per-thread kernel when nx
// is even (and no axis but x is periodic), the scalar one otherwise; both use the z-chunks
// of sw (same partial slots).
template <class TS, int kMode, class TD = TS>
void launch_refine_df(const Geo &g, const Sweep &sw, int nf, const CoefDF &cf, int scheme,
                      const DF *xin, const TD *d, const DF *b, DF *xout, DF *bout, TS *r, TS *y1,
                      float gamma, double *partials, RefScal *sc, RefScal *sc_next,
                      cudaStream_t st) {
    const dim3 blk(TX, TY);
    if (df_pairs(g)) {
        const dim3 grid((g.nx + 2 * TX - 1) / (2 * TX), sw.grid.y, sw.grid.z);
        launch_chain(k_refine_df2<TS, kMode, TD>, grid, blk, st, g, sw.zlen, sw.nzc, cf,
                     scheme, xin, d, b, xout, bout, r, y1, gamma, partials, sc, sc_next);
    } else {
        launch_chain(k_refine_df<TS, kMode, TD>, sw.grid, blk, st, g, sw.zlen, sw.nzc, cf, scheme, xin,
                     d, b, xout, bout, r, y1, gamma, partials, sc, sc_next);
    }
}

// Whether the merged pass has a form for the call: the packed form is implicit Euler only.
inline bool mid_fits(const Geo &g, int scheme) { return scheme == 0 || !df_pairs(g); }

// Its launch geometry: three blocks to an SM, and a block pays about two planes besides its
// own (the planes either side and its start), so the chunk of at most 16 planes that minimises
// waves x (planes + 2): longer ones leave SMs idle at the end (3 fields of 128^3 in one wave of
// 32 planes 81.7 us, in two or more 76).
inline Sweep mid_sweep(const Geo &g, int nf) {
    const long long slots = 3LL * num_sms();
    const int w = df_pairs(g) ? 2 * TX : TX;
    const long long cols = (long long)((g.nx + w - 1) / w) * ((g.ny + TY - 1) / TY) * nf;
    int best = 1;
    long long cost = -1;
    for (int z = std::min(16, g.nz); z >= 1; --z) {
        const int nzc = (g.nz + z - 1) / z;
        if ((g.nz + nzc - 1) / nzc != z || !grid_z_fits(g, nf, z)) continue;   // (no even chunks of z)
        const long long c = (cols * nzc + slots - 1) / slots * (z + 2);
        if (cost < 0 || c < cost) {
            cost = c;
            best = z;
        }
    }
    return make_sweep_z(g, nf, best);
}

// One merged pass (en == nullptr: the call's last).
inline void launch_refine_mid(const Geo &g, const Sweep &sw, const CoefDF &cf, int scheme, const DF *u,
                              const float *e, const float *d, const float *en, const DF *b, DF *xout, DF *bout,
                              float *r, float *y1, float gamma, double *partials, RefScal *sc, RefScal *sc_next,
                              cudaStream_t st) {
    const dim3 blk(TX, TY);
    if (df_pairs(g)) {
        const dim3 grid((g.nx + 2 * TX - 1) / (2 * TX), sw.grid.y, sw.grid.z);
        launch_chain(en ? k_refine_mid2<false> : k_refine_mid2<true>, grid, blk, st, g, sw.zlen, sw.nzc, cf, u, e, d,
                     en, xout, r, y1, gamma, partials, sc, sc_next);
    } else {
        launch_chain(en ? k_refine_mid<false> : k_refine_mid<true>, sw.grid, blk, st, g, sw.zlen, sw.nzc, cf, scheme,
                     u, e, d, en, b, xout, bout, r, y1, gamma, partials, sc, sc_next);
    }
}

// Brick decomposition for k_cheb_resident: the smallest brick (rows x planes) such that
// the bricks fit on the SMs one per SM and two padded brick arrays fit in one block's
// shared memory.  Not available (ok = false) for several fields, nx % 4 != 0, more
// iterations than the weight table holds, or a mesh too large for the SMs.
struct ResidentPlan {
    bool ok = false;
    Brick bk{};
    int nblocks = 0;
    size_t smem = 0;       // dynamic shared memory per block
    size_t ws_bytes = 0;   // flags | error word | faces
};

template <class TS>
ResidentPlan plan_resident(const Geo &g, int nf, int m_it) {
    ResidentPlan rp;
    if (nf != 1 || g.nx % 4 != 0 || m_it < 2 || m_it > kResidentMaxIters) return rp;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
        cudaGetLastError();
        return rp;
    }
    const int nsm = num_sms();
    const size_t limit = (size_t)optin > 2048 ? (size_t)optin - 2048 : 0;   // static shared
    const int P = g.nx + 8;
    long long best_rows = -1;
    int best_halo = 0;
    for (int by = 1; by <= std::min(g.ny, 64); ++by)
        for (int bz = 1; bz <= std::min(g.nz, 64); ++bz) {
            const int nby = (g.ny + by - 1) / by, nbz = (g.nz + bz - 1) / bz;
            if ((long long)nby * nbz > nsm) continue;
            const size_t smem = 2ull * P * (by + 2) * (bz + 2) * 4;
            if (smem > limit) continue;
            const long long rows = (long long)by * bz;
            if (best_rows < 0 || rows < best_rows || (rows == best_rows && by + bz < best_halo)) {
                best_rows = rows;
                best_halo = by + bz;
                rp.bk = Brick{by, bz, nby, nbz, P, g.nx * std::max(by, bz)};
                rp.smem = smem;
                rp.nblocks = nby * nbz;
            }
        }
    if (best_rows < 0) return rp;
    // the attribute is raised to the device limit once for all meshes (a captured launch
    // of another mesh may need more than this one)
    if (cudaFuncSetAttribute(k_cheb_resident<TS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)limit) != cudaSuccess) {
        cudaGetLastError();
        return rp;
    }
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cheb_resident<TS>, kResidentThreads,
                                                      rp.smem) != cudaSuccess) {
        cudaGetLastError();
        return rp;
    }
    if (per_sm < 1 || rp.nblocks > per_sm * nsm) return rp;
    rp.ws_bytes = align_up((size_t)(rp.nblocks + 1) * 4) + (size_t)rp.nblocks * 8 * rp.bk.fmax * 4;
    rp.ok = true;
    return rp;
}

// One round's m-1 Chebyshev iterations as one resident launch; the flags are cleared
// first (ws: flags | error word | faces, ws_bytes of plan_resident).  The error word is
// left alone so that it collects every launch since the caller cleared it.
template <class TS>
cudaError_t launch_resident(const Geo &g, const ResidentPlan &rp, const Coef32 &cf, float gamma,
                            double sigma, int m, const TS *y1, const TS *r, TS *yout, char *ws,
                            long long budget, cudaStream_t st) {
    unsigned int *flags = (unsigned int *)ws;
    int *err = (int *)(ws + (size_t)rp.nblocks * 4);
    float *faces = (float *)(ws + align_up((size_t)(rp.nblocks + 1) * 4));
    ChebWeights om{};
    double o = 1.0;
    om.w[0] = 1.0f;
    for (int k = 1; k < m; ++k) {
        if (sigma > 0.0)
            o = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma * sigma))
                         : 1.0 / (1.0 - o / (4.0 * sigma * sigma));
        om.w[k] = (float)o;
    }
    cudaError_t e = cudaMemsetAsync(ws, 0, (size_t)rp.nblocks * 4, st);
    if (e != cudaSuccess) return e;
    Geo ga = g;
    Brick bk = rp.bk;
    Coef32 cfa = cf;
    float ga_ = gamma;
    int ma = m;
    const TS *y1a = y1, *ra = r;
    TS *ya = yout;
    long long bu = budget;
    void *args[] = {&ga, &bk, &cfa, &ga_, &om, &ma, &y1a, &ra, &ya, &faces, &flags, &err, &bu};
    return cudaLaunchCooperativeKernel((const void *)k_cheb_resident<TS>, dim3(rp.nblocks),
                                       dim3(kResidentThreads), args, rp.smem, st);
}

// Where the last of the m-1 streamed Chebyshev iterates lands (y_{k+1} over y_{k-1},
// the first over `other`).
template <class TS>
TS *cheb_final_buffer(TS *y1, TS *other, int m) {
    TS *yc = y1, *yp = nullptr;
    for (int k = 1; k < m; ++k) {
        TS *yn = yp ? yp : other;
        yp = yc;
        yc = yn;
    }
    return yc;
}

// Resident or streamed inner solve for m iterations: both are captured as CUDA graphs on
// the caller's buffers (the round's whole Chebyshev loop, as the solver runs it), and
// the faster replay (best of three after a warm-up) is kept per mesh, field count,
// storage type and m.
// Tuning results shared by every mesh of the process: a mesh with the dimensions, periodic
// axes and tuning key (field count and storage type; for the resident solve, the
// iteration count) of one tuned before takes that choice without timing it again, and one
// thread times at a time.  Problems that run concurrently on other threads would
// otherwise disturb each other's timings, and a disturbed timing can pick a shape that is
// much slower in the solve (one plane per block against two at 128^3: 7.3 against 8.5 ms
// for ten implicit steps at b = 8 dx).
struct TuneKey {
    int nx, ny, nz, per, key, dev;
    bool operator==(const TuneKey &o) const {
        return nx == o.nx && ny == o.ny && nz == o.nz && per == o.per && key == o.key && dev == o.dev;
    }
};
std::mutex g_tune_mu;
std::vector<std::pair<TuneKey, int>> g_tuned;

template <class TS>
cg_status tune_resident(cg_mesh *m, const Geo &g, const ResidentPlan &rp, int code, int m_it,
                        const Coef32 &cf, TS *ya, TS *yb, TS *yc4, TS *yd4, const TS *r, char *ws,
                        cudaStream_t st, bool *use) {
    const int key = -((m_it * 64 + 1) * 4 + (int)sizeof(TS));
    for (auto &e : m->tuned)
        if (e.first == key) {
            *use = e.second != 0;
            return CG_OK;
        }
    int dev = 0;
    CGK_CUDA(cudaGetDevice(&dev));
    const TuneKey tk{g.nx, g.ny, g.nz, g.per, key * 1024 + (code + 512), dev};   // code in -16 .. 416
    std::lock_guard<std::mutex> lock(g_tune_mu);
    for (auto &e : g_tuned)
        if (e.first == tk) {
            m->tuned.push_back({key, e.second});
            *use = e.second != 0;
            return CG_OK;
        }
    if (!m->capture_stream)
        CGK_CUDA(cudaStreamCreateWithFlags(&m->capture_stream, cudaStreamNonBlocking));
    cudaEvent_t e0, e1;
    CGK_CUDA(cudaEventCreate(&e0));
    CGK_CUDA(cudaEventCreate(&e1));
    float t[2] = {1e30f, 1e30f};
    CGK_CUDA(cudaMemsetAsync(ws + (size_t)rp.nblocks * 4, 0, 4, st));
    cudaError_t ce = cudaSuccess;
    for (int variant = 0; variant < 2 && ce == cudaSuccess; ++variant) {
        cudaStream_t cs = m->capture_stream;
        cudaGraph_t graph = nullptr;
        cudaGraphExec_t exec = nullptr;
        cudaError_t le = cudaSuccess;
        ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (ce == cudaSuccess) {
            if (variant == 0 && code >= kPairCode && code < kResidentCode) {
                TS *const pool[4] = {ya, yb, yc4, yd4};
                cheb_pairs<TS>(code - kPairCode, g, 1, cf, 0.5f, 0.0, m_it, pool, r, cs);
            } else if (variant == 0) {
                TS *yc = ya, *yp = nullptr;
                for (int k = 1; k < m_it; ++k) {
                    TS *yn = yp ? yp : yb;
                    launch_cheb<TS>(code, g, 1, cf, 0.5f, 1.0f, yc, yp, r, yn, cs);
                    yp = yc;
                    yc = yn;
                }
            } else {
                le = launch_resident<TS>(g, rp, cf, 0.5f, 0.0, m_it, ya, r, yb, ws, 2000000000LL, cs);
            }
            ce = cudaStreamEndCapture(cs, &graph);
            if (ce == cudaSuccess) ce = le;
        }
        if (ce == cudaSuccess) ce = cudaGraphInstantiate(&exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        for (int rep = 0; rep < 4 && ce == cudaSuccess; ++rep) {
            cudaEventRecord(e0, st);
            ce = cudaGraphLaunch(exec, st);
            cudaEventRecord(e1, st);
            if (ce == cudaSuccess) ce = cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0) t[variant] = std::min(t[variant], ms);
        }
        if (exec) cudaGraphExecDestroy(exec);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (ce != cudaSuccess) return cuda_fail(ce, "resident autotuner", __FILE__, __LINE__);
    int errh = 0;
    CGK_CUDA(cudaMemcpy(&errh, ws + (size_t)rp.nblocks * 4, 4, cudaMemcpyDeviceToHost));
    if (errh) return fail(CG_ETIMEOUT, "cg_diffuse: a wait of the resident inner solve gave up");
    *use = t[1] < t[0];
    m->tuned.push_back({key, *use ? 1 : 0});
    g_tuned.push_back({tk, *use ? 1 : 0});
    return CG_OK;
}

// Autotuner of the Chebyshev sweep's shape (vectorised, register-blocked with 2, 4 or 8
// planes per block, z-marching with 1..16 planes per block): times ten iterations of
// each candidate on the caller's buffers (all scratch at this point) and keeps the
// fastest.  The choice is cached per mesh, field count and storage type, and shared with
// every mesh of the same geometry (the process-wide table below).  (The
// two-iterations-per-launch sweep is not a candidate: inside the solver's graph it
// measured no faster per iteration than the one-iteration sweep; sweep_shape selects it.)
template <class TS>
cg_status tune_cheb(cg_mesh *m, const Geo &g, int nf, const Coef32 &cf, TS *ya, TS *yb, TS *yc,
                    TS *yd, const TS *r, cudaStream_t st, int *code_out) {
    const int key = (nf * 4 + (int)sizeof(TS)) * 8 + g.per;
    for (auto &e : m->tuned)
        if (e.first == key) {
            *code_out = e.second;
            return CG_OK;
        }
    int dev = 0;
    CGK_CUDA(cudaGetDevice(&dev));
    const TuneKey tk{g.nx, g.ny, g.nz, g.per, key, dev};
    std::lock_guard<std::mutex> lock(g_tune_mu);
    for (auto &e : g_tuned)
        if (e.first == tk) {
            m->tuned.push_back({key, e.second});
            *code_out = e.second;
            return CG_OK;
        }
    if (!m->capture_stream)
        CGK_CUDA(cudaStreamCreateWithFlags(&m->capture_stream, cudaStreamNonBlocking));
    // candidates: code, and how many launches make 10 iterations
    std::vector<std::pair<int, int>> cands;
    const bool v4 = g.nx % 4 == 0;   // vectorised shapes need whole 4-cell vectors per row
    for (int c : {101, 102, 104, 108, 116, 2, 4, 8, -1, -4, -16})
        if ((c < 100 || v4) && (g.per == 0 || c < 0 || c >= 100))   // periodic: z-marching or vectorised
            cands.push_back({c, 10});
    if (sizeof(TS) == 4 && tma_sweep_fits(g)) {        // TMA-staged sweep: FP32 storage
        tma_prepare();
        for (int c : {401, 402, 404, 408}) cands.push_back({c, 10});
    }
    // two iterations per launch (five launches make ten) where the rows are longer than one
    // warp holds: there a sweep leaves L2 sooner and the whole-row kernel halves its traffic
    // (on rows of a warp, where the working set stays in L2, whole solves measured no gain)
    if (cheb2_fits(g) && g.nx > 128) {
        std::vector<int> zs = {8, 16, 32};
        {   // one block per SM, so also the chunk that minimises waves of blocks x planes a
            // block marches (its chunk and the plane either side)
            int sms = 0;
            CGK_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            const int tyr = rows_per_block(g.nx);
            const long long yb = (long long)((g.ny + tyr - 1) / tyr) * nf;
            int best_z = g.nz;
            long long best_cost = -1;
            for (int c = 1; c <= g.nz; ++c) {
                const int zc = (g.nz + c - 1) / c;
                const long long blocks = yb * ((g.nz + zc - 1) / zc);
                const long long cost = (blocks + sms - 1) / sms * (zc + 2);
                if (best_cost < 0 || cost < best_cost) {
                    best_cost = cost;
                    best_z = zc;
                }
            }
            zs.push_back(best_z);
        }
        for (int z : zs) {
            const int c = kPairCode + std::max(1, std::min({z, g.nz, 99}));
            bool dup = false;
            for (auto &cd : cands) dup = dup || cd.first == c;
            if (!dup) cands.push_back({c, 5});
        }
    }
    // per shape: 10 iterations captured as a CUDA graph (as the solver runs them) and
    // replayed once to warm up; then three rounds that replay every shape in turn, each
    // shape keeping its fastest replay (interleaving spreads a transient disturbance over
    // all shapes instead of one); the vectorised shape is kept unless another is more
    // than 3 % faster
    std::vector<cudaGraphExec_t> execs(cands.size(), nullptr);
    cudaError_t ce = cudaSuccess;
    for (size_t i = 0; i < cands.size() && ce == cudaSuccess; ++i) {
        const int code = cands[i].first;
        cudaStream_t cs = m->capture_stream;
        cudaGraph_t graph = nullptr;
        ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (ce == cudaSuccess) {
            for (int q = 0; q < cands[i].second; ++q) {
                if (code >= kPairCode && code < kResidentCode)
                    launch_cheb2<TS>(code - kPairCode, g, nf, cf, 0.5f, 1.0f, 1.0f, ya, yb, r, yc,
                                     yd, cs);
                else
                    launch_cheb<TS>(code, g, nf, cf, 0.5f, 1.0f, ya, yb, r, yb, cs);
            }
            ce = cudaStreamEndCapture(cs, &graph);
        }
        if (ce == cudaSuccess) ce = cudaGraphInstantiate(&execs[i], graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (ce == cudaSuccess) ce = cudaGraphLaunch(execs[i], st);   // warm-up replay
    }
    std::vector<std::pair<float, int>> timing;
    for (auto &cand : cands) timing.push_back({1e30f, cand.first});
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (ce == cudaSuccess) ce = cudaEventCreate(&e0);
    if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
    for (int round = 0; round < 3 && ce == cudaSuccess; ++round)
        for (size_t i = 0; i < cands.size() && ce == cudaSuccess; ++i) {
            cudaEventRecord(e0, st);
            ce = cudaGraphLaunch(execs[i], st);
            cudaEventRecord(e1, st);
            if (ce == cudaSuccess) ce = cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            timing[i].first = std::min(timing[i].first, ms);
        }
    for (cudaGraphExec_t ex : execs)
        if (ex) cudaGraphExecDestroy(ex);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (ce != cudaSuccess) return cuda_fail(ce, "sweep autotuner", __FILE__, __LINE__);
    if (tma_wait_failed(st)) return fail(CG_ETIMEOUT, "cg_diffuse: a wait of the TMA-staged sweep gave up");
    std::sort(timing.begin(), timing.end());
    int best_code = timing[0].second;
    if (v4) {
        float best_v4 = 1e30f;
        int code_v4 = 0;
        for (auto &tc : timing)
            if (tc.second >= 100 && tc.second < kPairCode && tc.first < best_v4) {
                best_v4 = tc.first;
                code_v4 = tc.second;
            }
        if (code_v4 && best_v4 <= 1.03f * timing[0].first) best_code = code_v4;
    }
    m->tuned.push_back({key, best_code});
    g_tuned.push_back({tk, best_code});
    *code_out = best_code;
    return CG_OK;
}

// ---------------------------------------------------------------- solid velocity
__global__ void k_solid_velocity(int64_t n, int ncomp, const double *__restrict__ eps,
                                 const double *__restrict__ mom, double eps_min,
                                 double *__restrict__ out) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        const double e = eps[k];
        const bool solid = e > eps_min;
        for (int c = 0; c < ncomp; ++c)
            out[(int64_t)c * n + k] = solid ? __ddiv_rn(mom[(int64_t)c * n + k], e) : 0.0;
    }
}

}  // namespace

// ============================================================================ host side
cg_status solid_velocity_run(int64_t n, int ncomp, const double *eps, const double *mom,
                             double eps_min, double *u_out, cudaStream_t st) {
    if (n > 0) {
        CGK_LAUNCH("solid_velocity", (double)n * (8 + 16.0 * ncomp), st,
                   k_solid_velocity<<<stencil_grid(n), kThreads, 0, st>>>(n, ncomp, eps, mom,
                                                                         eps_min, u_out));
        CGK_CUDA(cudaGetLastError());
    }
    CGK_CUDA(cudaStreamSynchronize(st));
    return CG_OK;
}

// Launches the mass reduction of one mesh's fields and the copy of its result into the
// mesh's pinned readback buffer (complete once the stream has synchronised).
// keep: device doubles that take the masses instead of the pinned readback buffer.
static cg_status field_mass_launch(cg_mesh *m, int nf, const double *cells, cudaStream_t st,
                                   double *keep = nullptr) {
    int n = (int)m->ncells;
    // a block per 2048 cells, at most four to an SM over all fields
    const int G = std::max(1, std::min((n + 2047) / 2048, std::max(1, 4 * num_sms() / nf)));
    size_t need = align_up((size_t)nf * G * 8) + 64 * 8 + 64 * 4;
    CGK_TRY(m->ws_small.ensure(4096 + need, kSmallRoom));
    char *base = m->ws_small.as<char>() + 4096;
    double *partials = (double *)base;
    double *out = (double *)(base + align_up((size_t)nf * G * 8));
    unsigned int *tickets = (unsigned int *)(out + 64);
    if (keep) out = keep;
    CGK_CUDA(cudaMemsetAsync(tickets, 0, 64 * 4, st));
    const double *vc = m->kind != MESH_STRUCTURED ? m->tet.vc : nullptr;
    double vcu = (m->dx * m->dx) * m->dx;
    CGK_LAUNCH("mass", (double)n * nf * 8, st,
               k_mass<<<dim3(G, nf), kThreads, 0, st>>>(n, cells, vc, vcu, partials, tickets, out));
    CGK_CUDA(cudaGetLastError());
    if (keep) return CG_OK;
    CGK_TRY(m->h_small.ensure(4096));
    CGK_CUDA(cudaMemcpyAsync(m->h_small.as<char>() + 2048, out, nf * 8, cudaMemcpyDeviceToHost, st));
    return CG_OK;
}

// Without waiting or copying: the masses stay in device memory (the mesh's location
// workspace, which no diffusion touches), slot 0 or 1; field_mass_read waits and copies.
cg_status field_mass_keep(cg_mesh *m, int nf, const double *cells, int slot, cudaStream_t st) {
    CGK_TRY(m->ws_locate.ensure(4096));
    return field_mass_launch(m, nf, cells, st, m->ws_locate.as<double>() + 64 * slot);
}
cg_status field_mass_read(cg_mesh *m, int nf, double *slot0, double *slot1, cudaStream_t st) {
    CGK_TRY(m->h_small.ensure(4096));
    double *h = (double *)(m->h_small.as<char>() + 2048);
    CGK_CUDA(cudaMemcpyAsync(h, m->ws_locate.as<double>(), 128 * 8, cudaMemcpyDeviceToHost, st));
    CGK_CUDA(cudaStreamSynchronize(st));
    for (int f = 0; f < nf; ++f) {
        slot0[f] = h[f];
        if (slot1) slot1[f] = h[64 + f];
    }
    return CG_OK;
}

// The masses of several meshes' fields (distinct meshes: each uses its own buffers): every
// reduction is launched before one synchronisation; mass_host[s * nf + f].
cg_status field_mass_many(int nmesh, cg_mesh *const *ms, int nf, const double *const *cells,
                          double *mass_host, cudaStream_t st) {
    for (int s = 0; s < nmesh; ++s) CGK_TRY(field_mass_launch(ms[s], nf, cells[s], st));
    CGK_CUDA(cudaStreamSynchronize(st));
    for (int s = 0; s < nmesh; ++s)
        for (int f = 0; f < nf; ++f)
            mass_host[(size_t)s * nf + f] = ((double *)(ms[s]->h_small.as<char>() + 2048))[f];
    return CG_OK;
}

// FP64 CG as one cooperative launch (k_cg_coop) where a field's cells fit in the SMs'
// registers; *solved stays false where it does not apply or a wait gave up, and the
// caller's field is then untouched.
template <int NT, int C>
static cudaError_t launch_cg_coop(int groups, int blocks, Geo g, int per_block, double c, Coef64 cf, int scheme,
                                  int nf, int nsteps, int max_it, double tol2, const double *cells, double *X,
                                  double *V, size_t vstride, double2 *part, Scal *hist, CoopBar *bars,
                                  cudaStream_t st) {
    long long budget = 2000000000LL;   // clock cycles a wait may take (about one second)
    void *args[] = {&g, &blocks, &per_block, &c, &cf, &scheme, &nf, &nsteps, &max_it, &tol2, &cells, &X, &V,
                    &vstride, &part, &hist, &bars, &budget};
    return cudaLaunchCooperativeKernel((const void *)k_cg_coop<NT, C>, dim3(groups * blocks), dim3(NT), args, 0, st);
}

static cg_status fp64_coop(cg_mesh *m, const Geo &g, int nf, double *cells, const cg_params *p, double c,
                           const Coef64 &cf, cg_report *rep, cudaStream_t st, bool *solved) {
    const int n = g.n;
    // A block per SM, but at least 64 cells to a block (8^3 on 8 blocks: 7.5 us per iteration);
    // up to 12 cells for each of 512 threads on every SM (933,888 cells on 152 SMs), where the
    // cooperative form is still twice as fast as the two-launch form (30.7 against 58.7 us at 96^3).  Small meshes take
    // blocks of fewer threads, so that the solves of several streams share the SMs: blocks of
    // 512 threads at any size ran six concurrent 32^3 calls one after another, 15.2 ms
    // against 8.6 with the two-launch form (now 5.4; 64^3 20.3 -> 16.2 ms).
    const int grid = std::max(1, std::min(num_sms(), (n + 63) / 64));
    const int per_block = (n + grid - 1) / grid;
    const int nt = per_block <= 128 * 4 ? 128 : per_block <= 256 * 8 ? 256 : 512;
    const int need = (per_block + nt - 1) / nt;
    if (need > kCoopMaxC) return CG_OK;
    // Groups of fields side by side: up to four blocks of 128 threads on an SM, evened out over the
    // turns.  Blocks of 256 threads run one field at a time: an SM holds two of them, and a second
    // problem's fill that place as well as a second field would (four problems of 48^3 x 3 fields
    // at a time 19.2 ms, 26.9 with two groups each).
    const int cap = nt == 128 ? std::min(nf, 4 * num_sms() / grid) : 1, turns = (nf + cap - 1) / cap;
    const int groups = (nf + turns - 1) / turns;
    // Many fields of a small mesh take so many turns of about 8.5 us an iteration that the two-launch
    // form, one pair of launches for all of them, is the faster one: it costs about 24 us and, per
    // million cells, 19 us more than the turns' arithmetic.  Measured per iteration, this form
    // against that one: 16^3 x 16 fields 17.5 and 23.9 us, x 32 34.0 and 27.5; 32^3 x 8 23.4 and 29.6,
    // x 16 46.4 and 42.8; 48^3 x 3 35.8 and 35.8, x 4 47.8 and 42.5; 64^3 x 5 79.6 and 79.9, x 8 127 and 112.
    if (8.5 * turns > 24.0 + 1.9e-5 * nf * n) return CG_OK;
    const size_t vec = align_up((size_t)n * nf * 8), one = align_up((size_t)n * 8);
    const size_t hist_n = (size_t)p->nsteps * nf;
    const size_t part_b = align_up((size_t)2 * groups * grid * sizeof(double2));
    const size_t bars_b = align_up((size_t)(groups + 1) * sizeof(CoopBar));
    if (hist_n > (1u << 20) || m->ws_diffuse.ensure(vec + groups * one) != CG_OK ||
        m->ws_small.ensure(4096 + part_b + bars_b + hist_n * sizeof(Scal)) != CG_OK ||
        m->h_small.ensure(4096 + bars_b + hist_n * sizeof(Scal)) != CG_OK)
        return CG_OK;
    double *X = m->ws_diffuse.as<double>(), *V = (double *)(m->ws_diffuse.as<char>() + vec);
    double2 *part = (double2 *)(m->ws_small.as<char>() + 4096);
    CoopBar *bars = (CoopBar *)(m->ws_small.as<char>() + 4096 + part_b);
    Scal *hist = (Scal *)((char *)bars + bars_b);
    CGK_CUDA(cudaMemsetAsync(bars, 0, bars_b + hist_n * sizeof(Scal), st));
    // the two-launch form checks its iteration cap every eight iterations
    const int max_it = p->max_iter > 0x7ffffff0 ? 0x7ffffff0 : (p->max_iter + 7) / 8 * 8;
    const double tol2 = p->tol * p->tol;
    cudaError_t e = cudaSuccess;
#define CGK_COOP(NT, C)                                                                                    \
    CGK_LAUNCH("cg64_coop", (double)n * nf * 16, st,                                                       \
               e = launch_cg_coop<NT, C>(groups, grid, g, per_block, c, cf, p->scheme, nf, p->nsteps, max_it,  \
                                     tol2, cells, X, V, one / 8, part, hist, bars, st))
    if (nt == 128) {
        if (need <= 1) CGK_COOP(128, 1);
        else if (need <= 2) CGK_COOP(128, 2);
        else CGK_COOP(128, 4);
    } else if (nt == 256) {
        if (need <= 4) CGK_COOP(256, 4);
        else CGK_COOP(256, 8);
    } else {
        if (need <= 8) CGK_COOP(512, 8);
        else CGK_COOP(512, 12);
    }
#undef CGK_COOP
    if (e != cudaSuccess) {   // not launched: the two-launch form takes the call
        cudaGetLastError();
        return CG_OK;
    }
    CGK_LAUNCH("cg64_coop_out", (double)n * nf * 16, st,
               k_cg_coop_out<<<stencil_grid((int)std::min<size_t>((size_t)n * nf, 1u << 30)), kThreads, 0, st>>>(
                   (size_t)n * nf, X, cells, bars));
    CGK_CUDA(cudaGetLastError());
    char *hb = m->h_small.as<char>() + 4096;
    CGK_CUDA(cudaMemcpyAsync(hb, bars, bars_b + hist_n * sizeof(Scal), cudaMemcpyDeviceToHost, st));
    CGK_CUDA(cudaStreamSynchronize(st));
    if (((CoopBar *)hb)->err) return CG_OK;
    const Scal *h = (const Scal *)(hb + bars_b);
    long long total_iters = 0;
    double worst = 0.0;
    int bad = -1;
    for (int s = 0; s < p->nsteps && bad < 0; ++s)
        for (int f = 0; f < nf; ++f) {
            const Scal &S = h[(size_t)s * nf + f];
            total_iters += S.iters + 1;
            worst = std::max(worst, S.bb > 0 ? std::sqrt(S.rr / S.bb) : 0.0);
            if (S.breakdown ? S.rr > tol2 * S.bb : !S.done) bad = s;
        }
    if (rep) {
        rep->iters = total_iters;
        rep->cell_updates = total_iters * (long long)n;
        rep->final_rel_residual = worst;
    }
    *solved = true;
    if (bad >= 0) return fail(CG_ENOCONV, "cg_diffuse: FP64 CG did not reach tol in step %d", bad);
    return CG_OK;
}

static cg_status diffuse_fp64(cg_mesh *m, int nf, double *cells, const cg_params *p, double T,
                              cg_report *rep, cudaStream_t st) {
    const int n = (int)m->ncells;
    Geo g{m->nx, m->ny, m->nz, m->nx * m->ny, n, m->per};
    const double dtau = T / p->nsteps;
    const double c = dtau / (m->dx * m->dx);
    const double ce = p->scheme == CG_SCHEME_CRANK_NICOLSON ? 0.5 * c : c;
    const double tol2 = p->tol * p->tol;
    const Sweep sw = make_sweep(g, nf);
    const int G = sw.nb;
    const Coef64 cf = coef64(ce);
    const dim3 blk(TX, TY);
    bool solved = false;
    CGK_TRY(fp64_coop(m, g, nf, cells, p, c, cf, rep, st, &solved));
    if (solved) return CG_OK;
    const size_t vec = align_up((size_t)n * nf * 8);
    CGK_TRY(m->ws_diffuse.ensure(3 * vec));
    double *r = (double *)m->ws_diffuse.as<char>();
    double *P[2] = {(double *)(m->ws_diffuse.as<char>() + vec),
                    (double *)(m->ws_diffuse.as<char>() + 2 * vec)};
    const int ub = std::min(G, std::max(1, std::min((n + 4 * kThreads - 1) / (4 * kThreads), num_sms() * 8)));
    CGK_TRY(m->ws_small.ensure(4096 + align_up((size_t)nf * 2 * G * 8) + 64 * sizeof(Scal)));
    double *partials = (double *)(m->ws_small.as<char>() + 4096);
    Scal *sc = (Scal *)(m->ws_small.as<char>() + 4096 + align_up((size_t)nf * 2 * G * 8));
    CGK_CUDA(cudaMemsetAsync(sc, 0, nf * sizeof(Scal), st));
    CGK_TRY(m->h_small.ensure(4096 + 64 * sizeof(Scal)));
    Scal *hsc = (Scal *)(m->h_small.as<char>() + 4096);
    // a fourth vector keeps A p between the passes; where it may not be held the second pass
    // forms A p again
    OptUse opt;
    double *Q = opt.take(m->ws_opt, vec) ? m->ws_opt.as<double>() : nullptr;
    long long total_iters = 0;
    double worst = 0.0;
    const int chunk = 8;
    for (int s = 0; s < p->nsteps; ++s) {
        CGK_LAUNCH("cg64_init", (double)n * nf * 24, st,
                   k_cg_init<<<sw.grid, blk, 0, st>>>(g, sw.zlen, sw.nzc, c, p->scheme, cells, r,
                                                      P[0], partials, sc, tol2));
        CGK_CUDA(cudaGetLastError());
        int it = 0;
        bool all_done = false;
        while (true) {
            for (int q = 0; q < chunk; ++q, ++it) {
                CGK_LAUNCH("cg64_pass1", (double)n * nf * (Q ? 32 : 24), st,
                           k_cg_pass1<<<sw.grid, blk, 0, st>>>(g, sw.zlen, sw.nzc, cf, r,
                                                               P[it & 1], P[(it + 1) & 1], Q,
                                                               partials, sc));
                if (Q)
                    CGK_LAUNCH("cg64_update", (double)n * nf * 48, st,
                               k_cg_update<<<dim3(ub, nf), kThreads, 0, st>>>(n, G, P[(it + 1) & 1], Q, cells,
                                                                              r, partials, sc, tol2));
                else
                    CGK_LAUNCH("cg64_pass2", (double)n * nf * 40, st,
                               k_cg_pass2<<<sw.grid, blk, 0, st>>>(g, sw.zlen, sw.nzc, cf,
                                                                   P[(it + 1) & 1], cells, r,
                                                                   partials, sc, tol2));
            }
            CGK_CUDA(cudaGetLastError());
            CGK_CUDA(cudaMemcpyAsync(hsc, sc, nf * sizeof(Scal), cudaMemcpyDeviceToHost, st));
            CGK_CUDA(cudaStreamSynchronize(st));
            all_done = true;
            for (int f = 0; f < nf; ++f) all_done = all_done && hsc[f].done;
            if (all_done || it >= p->max_iter) break;
        }
        for (int f = 0; f < nf; ++f) {
            total_iters += hsc[f].iters + 1;
            double rel = hsc[f].bb > 0 ? std::sqrt(hsc[f].rr / hsc[f].bb) : 0.0;
            if (rel > worst) worst = rel;
            if (hsc[f].breakdown && hsc[f].rr > tol2 * hsc[f].bb) all_done = false;
        }
        if (!all_done) {
            if (rep) {
                rep->iters = total_iters;
                rep->cell_updates = total_iters * (long long)n;
                rep->final_rel_residual = worst;
            }
            return fail(CG_ENOCONV, "cg_diffuse: FP64 CG did not reach tol in step %d", s);
        }
    }
    if (rep) {
        rep->iters = total_iters;
        rep->cell_updates = total_iters * (long long)n;
        rep->final_rel_residual = worst;
    }
    return CG_OK;
}

// One launch of k_explicit_tb<K>: kt explicit steps (1 <= kt <= 4) from a to b.
// Resident blocks per SM of k_explicit_tb<K> (queried once per thread: the library's
// calls may run on several host threads at a time).
template <int K> static int explicit_tb_blocks_per_sm(size_t smem) {
    static thread_local int cached = 0;
    if (!cached) {
        cudaFuncSetAttribute(k_explicit_tb<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_explicit_tb<K>, kEBlock.x * kEBlock.y, smem) !=
                cudaSuccess || nb < 1)
            nb = 1;
        cached = nb;
    }
    return cached;
}

template <int K> static int explicit_tb4_blocks_per_sm(size_t smem) {
    static thread_local int cached = 0;
    if (!cached) {
        cudaFuncSetAttribute(k_explicit_tb4<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int nb = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_explicit_tb4<K>, 1024, smem) != cudaSuccess ||
            nb < 1)
            nb = 1;
        cached = nb;
    }
    return cached;
}

// z-chunk length of a blocked explicit launch: a block of a chunk of zlen planes runs
// zlen + 2K pipeline iterations and the launch takes ceil(blocks / resident blocks)
// waves; the chunk length that minimises waves x (zlen + 2K).
static int explicit_zlen(const Geo &g, long long cols, long long slots, int kt) {
    int zlen = g.nz;
    long long best = -1;
    for (int zl = 1; zl <= g.nz; ++zl) {
        const long long nzc = (g.nz + zl - 1) / zl;
        if (zl > 1 && (g.nz + zl - 2) / (zl - 1) == nzc) continue;   // same chunk count, shorter zl wins
        const long long waves = (cols * nzc + slots - 1) / slots;
        const long long cost = waves * (zl + 2 * kt);
        if (best < 0 || cost < best) best = cost, zlen = zl;
    }
    return zlen;
}

// One launch of the four-cells-per-thread kernel k_explicit_tb4<K> (nx % 4 == 0).
static cg_status launch_explicit_tb4(const Geo &g, int nf, int kt, float c, const float *a, float *b,
                                     cudaStream_t st) {
    const int OY = kE4H - 2 * kt;
    // tiles per axis: at walls the first and the last tile need no halo outside
    const bool px = g.per & 1, py = (g.per >> 1) & 1;
    const int gx = px ? (g.nx + kE4OX - 1) / kE4OX : std::max(1, (g.nx - 8 + kE4OX - 1) / kE4OX);
    const int gy = py ? (g.ny + OY - 1) / OY : std::max(1, (g.ny - 2 * kt + OY - 1) / OY);
    const size_t smem = explicit_tb4_smem(kt);
    const int per_sm = kt == 1 ? explicit_tb4_blocks_per_sm<1>(smem)
                     : kt == 2 ? explicit_tb4_blocks_per_sm<2>(smem)
                     : kt == 3 ? explicit_tb4_blocks_per_sm<3>(smem) : explicit_tb4_blocks_per_sm<4>(smem);
    const long long cols = (long long)gx * gy * nf;
    const int zlen = explicit_zlen(g, cols, (long long)num_sms() * per_sm, kt);
    const int nzc = (g.nz + zlen - 1) / zlen;
    const dim3 grid(gx, gy, nzc * nf);
    const double bytes = (double)g.n * nf * 8;
    switch (kt) {
    case 1:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb4<1><<<grid, kE4Block, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    case 2:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb4<2><<<grid, kE4Block, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    case 3:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb4<3><<<grid, kE4Block, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    default:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb4<4><<<grid, kE4Block, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    }
    CGK_CUDA(cudaGetLastError());
    return CG_OK;
}

static cg_status launch_explicit_tb(const Geo &g, int nf, int kt, float c, const float *a, float *b,
                                    cudaStream_t st) {
    if (g.nx % 4 == 0) return launch_explicit_tb4(g, nf, kt, c, a, b, st);
    const int OX = kEW - 2 * kt, OY = kEH - 2 * kt;
    const int gx = (g.nx + OX - 1) / OX, gy = (g.ny + OY - 1) / OY;
    const size_t smem = explicit_tb_smem(kt);
    const int per_sm = kt == 1 ? explicit_tb_blocks_per_sm<1>(smem)
                     : kt == 2 ? explicit_tb_blocks_per_sm<2>(smem)
                     : kt == 3 ? explicit_tb_blocks_per_sm<3>(smem) : explicit_tb_blocks_per_sm<4>(smem);
    const long long cols = (long long)gx * gy * nf;
    const int zlen = explicit_zlen(g, cols, (long long)num_sms() * per_sm, kt);
    const int nzc = (g.nz + zlen - 1) / zlen;
    const dim3 grid(gx, gy, nzc * nf);
    const double bytes = (double)g.n * nf * 8;
    switch (kt) {
    case 1:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb<1><<<grid, kEBlock, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    case 2:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb<2><<<grid, kEBlock, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    case 3:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb<3><<<grid, kEBlock, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    default:
        CGK_LAUNCH("explicit_tb", bytes, st, k_explicit_tb<4><<<grid, kEBlock, smem, st>>>(g, zlen, nzc, c, a, b));
        break;
    }
    CGK_CUDA(cudaGetLastError());
    return CG_OK;
}

// Explicit Euler in FP32 with K = fused_k steps per launch (the last launch takes the
// remainder).
static cg_status explicit_blocked(const Geo &g, int nf, double *cells, int nsteps, int K, float c,
                                  cg_mesh *m, cg_report *rep, cudaStream_t st) {
    if (K > 4) return fail(CG_EINVAL, "cg_diffuse: fused_k must be 0..4 (got %d)", K);
    const size_t cnt = (size_t)g.n * nf;
    const size_t vec = align_up(cnt * 4);
    CGK_TRY(m->ws_diffuse.ensure(2 * vec));
    float *a = m->ws_diffuse.as<float>(), *b = (float *)(m->ws_diffuse.as<char>() + vec);
    CGK_LAUNCH("to_f32", (double)cnt * 12, st, k_to_f32<<<stencil_grid(cnt), kThreads, 0, st>>>(cnt, cells, a));
    for (int s = 0; s < nsteps;) {
        const int kt = std::min(K, nsteps - s);
        CGK_TRY(launch_explicit_tb(g, nf, kt, c, a, b, st));
        std::swap(a, b);
        s += kt;
    }
    CGK_LAUNCH("from_f32", (double)cnt * 12, st, k_from_f32<<<stencil_grid(cnt), kThreads, 0, st>>>(cnt, a, cells));
    CGK_CUDA(cudaGetLastError());
    CGK_CUDA(cudaStreamSynchronize(st));
    if (rep) {
        rep->iters = (long long)nsteps * nf;
        rep->cell_updates = rep->iters * (long long)g.n;
        rep->final_rel_residual = 0.0;
    }
    return CG_OK;
}

static cg_status diffuse_explicit(cg_mesh *m, int nf, double *cells, const cg_params *p, double T,
                                  cg_report *rep, cudaStream_t st) {
    const int n = (int)m->ncells;
    Geo g{m->nx, m->ny, m->nz, m->nx * m->ny, n, m->per};
    const double dtau = T / p->nsteps;
    const double c = dtau / (m->dx * m->dx);
    if (c > 1.0 / 6.0 + 1e-15)
        return fail(CG_EINVAL, "cg_diffuse: explicit Euler needs dtau <= dx^2/6 (dtau/dx^2 = %g)", c);
    const size_t vec = align_up((size_t)n * nf * 8);
    if (p->fused_k > 0) return explicit_blocked(g, nf, cells, p->nsteps, p->fused_k, (float)c, m, rep, st);
    const Sweep sw = make_sweep(g, nf);
    const dim3 blk(TX, TY);
    const bool df = (p->precision == CG_PREC_FP32_DF_REFINE || p->precision == CG_PREC_BF16_DF_REFINE) &&
                    m->nx % 2 == 0 && m->per == 0;
    if (df) {
        // double-float steps (FP64-class accuracy on the FP32 units), two cells per thread
        CGK_TRY(m->ws_diffuse.ensure(2 * vec));
        DF *A = m->ws_diffuse.as<DF>(), *Bf = (DF *)(m->ws_diffuse.as<char>() + vec);
        const CoefDF cfdf = coefdf(c, c);
        const dim3 grid((g.nx + 2 * TX - 1) / (2 * TX), sw.grid.y, sw.grid.z);
        CGK_LAUNCH("to_double_float", (double)n * nf * 16, st,
                   launch_to_df(g, (size_t)n * nf, cells, A, st));
        for (int s = 0; s < p->nsteps; ++s) {
            CGK_LAUNCH("explicit_df", (double)n * nf * 16, st,
                       launch_chain(k_refine_df2<float, 3>, grid, blk, st, g, sw.zlen, sw.nzc, cfdf,
                                    p->scheme, (const DF *)A, (const float *)nullptr,
                                    (const DF *)nullptr, Bf, (DF *)nullptr, (float *)nullptr,
                                    (float *)nullptr, 0.0f, (double *)nullptr, (RefScal *)nullptr,
                                    (RefScal *)nullptr));
            std::swap(A, Bf);
        }
        CGK_LAUNCH("from_double_float", (double)n * nf * 16, st,
                   launch_from_df(g, (size_t)n * nf, A, cells, st));
        CGK_CUDA(cudaGetLastError());
        CGK_CUDA(cudaStreamSynchronize(st));
        if (rep) {
            rep->iters = (long long)p->nsteps * nf;
            rep->cell_updates = rep->iters * (long long)n;
            rep->final_rel_residual = 0.0;
        }
        return CG_OK;
    }
    CGK_TRY(m->ws_diffuse.ensure(vec));
    double *tmp = m->ws_diffuse.as<double>();
    double *a = cells, *b = tmp;
    for (int s = 0; s < p->nsteps; ++s) {
        CGK_LAUNCH("explicit64", (double)n * nf * 16, st,
                   k_explicit<<<sw.grid, blk, 0, st>>>(g, sw.zlen, sw.nzc, c, a, b));
        std::swap(a, b);
    }
    CGK_CUDA(cudaGetLastError());
    if (a != cells)
        CGK_CUDA(cudaMemcpyAsync(cells, a, (size_t)n * nf * 8, cudaMemcpyDeviceToDevice, st));
    CGK_CUDA(cudaStreamSynchronize(st));
    if (rep) {
        rep->iters = (long long)p->nsteps * nf;
        rep->cell_updates = rep->iters * (long long)n;
        rep->final_rel_residual = 0.0;
    }
    return CG_OK;
}

// The expansions of a call's increments.  Step i of a run (i = 0, 1, ..) starting at u_0:
// implicit Euler u_i = (1 + c mu)^-i u_0, so h_i = -c mu (1 + c mu)^-(i+1); Crank-Nicolson
// u_i = g^i u_0 with g = (1 - c mu / 2) / (1 + c mu / 2), so h_i = (g - 1) g^i; mu >= 0 the
// eigenvalues of -L, up to mu_max.  Coefficients by Gauss-Chebyshev quadrature on enough
// nodes that they have decayed; K where the rest adds at most a third of the FP32 rounding
// of the sum to the residual: lmax tail_i <= 0.3 * 9e-8 S_i A_rms with S_i = sum |a|,
// A_rms = 1 + 6.5 ce (the diagonal dominates on rounding noise).
//
// Whether it pays: in units of one sweep (16 B per cell) a call's own inner solves take
// 2 (m - 1) per step and the predicted ones about half of that plus, per run, K recurrence
// sweeps of 12 B and the combination (K + 1 vectors read, `len` written).  By that count two
// steps cost as much either way and three are worth it; measured (whole diffusions, own
// rounds -> expansion): 128^3, 3 steps, c = 0.025 0.436 -> 0.392 ms, c = 0.4 0.813 -> 0.749 ms;
// 10 steps 1.10 -> 0.83 and 2.36 -> 1.78 ms; 32^3, 3 steps, c = 0.1 0.234 -> 0.196 ms.
static void pred_build(PredPlan &pl) {
    const double ce = pl.scheme == CG_SCHEME_CRANK_NICOLSON ? 0.5 * pl.c : pl.c;
    const double mu_max = (pl.lmax - 1.0) / ce;
    pl.use = false;
    if (!(mu_max > 0.0) || pl.nsteps < 2) return;
    const int groups = (pl.nsteps + kPredMaxSteps - 1) / kPredMaxSteps;
    const double arms = 1.0 + 6.5 * ce;
    double cost = 0.0;
    std::vector<std::vector<double>> sums;   // S_i per run
    for (int q = 0, s0 = 0; q < groups; ++q) {
        const int len = (pl.nsteps - s0 + groups - q - 1) / (groups - q);
        if (q > 0 && len == pl.len[q - 1]) {   // runs of one length share their coefficients
            pl.coef.push_back(pl.coef[q - 1]);
            pl.K.push_back(pl.K[q - 1]);
        } else {
            std::vector<double> a;   // [k][i]
            int K = -1, N = 32;
            for (; N <= 4 * kPredMaxK && K < 0; N *= 2) {
                const int kc = std::min(N / 2, kPredMaxK + 40);
                std::vector<double> cs(4 * N);
                for (int j = 0; j < 4 * N; ++j) cs[j] = std::cos(M_PI * j / (2.0 * N));
                a.assign((size_t)(kc + 1) * len, 0.0);
                std::vector<double> h(len);
                for (int j = 0; j < N; ++j) {   // x_j = cos(pi (j + 1/2) / N), mu = mu_max (1 - x) / 2
                    const double cm = pl.c * 0.5 * mu_max * (1.0 - cs[2 * j + 1]);
                    double g, w;
                    if (pl.scheme == CG_SCHEME_CRANK_NICOLSON) {
                        g = (1.0 - 0.5 * cm) / (1.0 + 0.5 * cm);
                        w = -cm / (1.0 + 0.5 * cm);   // g - 1
                    } else {
                        g = 1.0 / (1.0 + cm);
                        w = -cm * g;
                    }
                    for (int i = 0; i < len; ++i, w *= g) h[i] = w * 2.0 / N;
                    for (int k = 0; k <= kc; ++k) {
                        const double f = (k ? 1.0 : 0.5) * cs[(int)((long long)(2 * j + 1) * k % (4 * N))];
                        for (int i = 0; i < len; ++i) a[(size_t)k * len + i] += f * h[i];
                    }
                }
                std::vector<double> S(len, 0.0), tail(len, 0.0);
                for (int k = 0; k <= kc; ++k)
                    for (int i = 0; i < len; ++i) S[i] += std::fabs(a[(size_t)k * len + i]);
                int k = kc;
                for (; k > 0; --k) {   // drop T_k while every step's rest stays below its bound
                    bool drop = true;
                    for (int i = 0; i < len; ++i)
                        drop = drop && pl.lmax * (tail[i] + std::fabs(a[(size_t)k * len + i])) <= 2.7e-8 * S[i] * arms;
                    if (!drop) break;
                    for (int i = 0; i < len; ++i) tail[i] += std::fabs(a[(size_t)k * len + i]);
                }
                if (k <= kc - 4 && k <= kPredMaxK) K = std::max(k, 1);
            }
            if (K < 0) return;
            std::vector<float> f((size_t)(K + 1) * len);
            for (size_t j = 0; j < f.size(); ++j) f[j] = (float)a[j];
            for (int i = 0; i < len; ++i) {   // h_i(0) = 0 also for the rounded coefficients
                double sum = 0.0;
                for (int k = 1; k <= K; ++k) sum += f[(size_t)k * len + i];
                f[i] = (float)-sum;
            }
            pl.coef.push_back(f);
            pl.K.push_back(K);
            std::vector<double> S(len, 0.0);
            for (int k = 0; k <= K; ++k)
                for (int i = 0; i < len; ++i) S[i] += std::fabs(a[(size_t)k * len + i]);
            sums.push_back(S);
        }
        if (sums.size() < pl.coef.size()) sums.push_back(sums.back());
        pl.start.push_back(s0);
        pl.len.push_back(len);
        pl.maxK = std::max(pl.maxK, pl.K.back());
        pl.maxlen = std::max(pl.maxlen, len);
        cost += 0.75 * pl.K.back() + 0.25 * (pl.K.back() + 1 + len);
        s0 += len;
    }
    // The iterations of the round that follows: from the residual that rounding leaves in
    // step i, 9e-8 S_i A_rms ||u_0||, to half of what a double-float residual resolves,
    // with ||u_i|| / ||u_0|| of a field of white noise (a deposited field of few particles;
    // smoother fields decay less).  A mode's decay per step depends on mu alone: sampled at
    // the midpoints of 8^3 frequencies.
    double mus[120], wts[120];
    int ns = 0;
    for (int a = 0; a < 8; ++a)
        for (int b = a; b < 8; ++b)
            for (int d = b; d < 8; ++d) {
                auto l = [](int q) { const double v = std::sin(M_PI * (q + 0.5) / 16.0); return 4.0 * v * v; };
                mus[ns] = std::min(l(a) + l(b) + l(d), mu_max);
                wts[ns++] = a == d ? 1.0 : (a == b || b == d) ? 3.0 : 6.0;
            }
    std::vector<double> amp(ns, 1.0), norm(pl.nsteps);
    for (int s = 0; s < pl.nsteps; ++s) {
        double e = 0.0;
        for (int q = 0; q < ns; ++q) {
            e += wts[q] * amp[q] * amp[q];
            const double cm = pl.c * mus[q];
            amp[q] *= pl.scheme == CG_SCHEME_CRANK_NICOLSON ? (1.0 - 0.5 * cm) / (1.0 + 0.5 * cm) : 1.0 / (1.0 + cm);
        }
        norm[s] = std::sqrt(e / 512.0);
    }
    const double sg = (std::sqrt(pl.lmax) - 1.0) / (std::sqrt(pl.lmax) + 1.0);
    double own = 0.0;
    for (size_t q = 0; q < pl.start.size(); ++q)
        for (int i = 0; i < pl.len[q]; ++i) {
            const int s = pl.start[q] + i;
            const double est = 9e-8 * sums[q][i] * arms * norm[pl.start[q]] / norm[s];
            const double target = 1.8e-15 * arms;
            int mi = (int)std::ceil(std::log(2.0 * std::max(est / target, 1.0)) / -std::log(sg));
            mi = std::max(2, std::min(mi, 400));
            pl.m.push_back(mi);
            pl.maxm = std::max(pl.maxm, mi);
            cost += mi - 1;
            own += 2.0 * (pl.m_it - 1);
        }
    pl.use = cost <= 0.9 * own;
}

// A round's iterations where a step has R - 1 rounds of them.  The estimate is for one; a field that
// decays faster than white noise (the highest frequencies alone) needs a second, and each
// then has 0.65 of it: together (2 sg^(0.65 m))^2 instead of 2 sg^m, 4e-11 instead of 2e-8 at
// c = 0.225.  (With 0.6 a checkerboard of 128^3 at
// c = 0.8 took a third round.)  Checkerboards, 128^3, ten steps, two rounds of all m iterations
// against this: c = 0.225 2.53 -> 2.00 ms, c = 0.4 3.20 -> 2.47 ms.
static int pred_round_m(int m, int R) { return R > 2 ? std::max(2, (13 * m + 19) / 20) : m; }

static const PredPlan &pred_plan(cg_mesh *m, int scheme, int nsteps, int m_it, double c, double lmax) {
    for (const PredPlan &q : m->preds)
        if (q.scheme == scheme && q.nsteps == nsteps && q.m_it == m_it && q.c == c && q.lmax == lmax) return q;
    if (m->preds.size() >= 16) m->preds.erase(m->preds.begin());
    PredPlan pl;
    pl.scheme = scheme;
    pl.nsteps = nsteps;
    pl.m_it = m_it;
    pl.c = c;
    pl.lmax = lmax;
    pred_build(pl);
    m->preds.push_back(std::move(pl));
    return m->preds.back();
}

template <int NS>
static void launch_pred_combine(size_t n, size_t stride, const PredPlan &pl, int q, const float *t, float *d,
                                cudaStream_t st) {
    PredCoef<NS> cf;
    const int K = pl.K[q], len = pl.len[q];
    for (int k = 0; k <= K; ++k)
        for (int i = 0; i < NS; ++i) cf.a[k * NS + i] = i < len ? pl.coef[q][(size_t)k * len + i] : 0.f;
    const size_t n4 = (n + 3) / 4;
    const unsigned grid = (unsigned)std::min<size_t>((n4 + kThreads - 1) / kThreads, 1u << 30);
    launch_chain(k_pred_combine<NS>, dim3(grid), dim3(kThreads), st, n4, stride, K, cf, t, d);
}

// Planes per block of the vectorised sweep, unrolled (the register queue rotates by
// renaming) in 64 registers, four blocks to an SM: 128^3 4.7 us (1 plane 6.0; 4 planes at three
// blocks 5.5, 8 at two 7.0), 512 x 256 x 256 70.5 us = 5.7 TB/s (1 plane 96.9; 4 planes 73.4, 8 72.2).
constexpr int kPredPlanes = 2;
static int pred_sweep_planes(const Geo &g, int nf) {
    return g.nx % 4 == 0 ? kPredPlanes : g.per ? make_sweep(g, nf).zlen : 4;
}
static void launch_pred_sweep(const Geo &g, int nf, float w, const float *t, const float *tp, float *tn,
                              cudaStream_t st) {
    const dim3 blk(TX, TY);
    const int gy = (g.ny + TY - 1) / TY;
    const int zl = pred_sweep_planes(g, nf), nzc = (g.nz + zl - 1) / zl;
    if (g.nx % 4 == 0) {
        const dim3 grid((g.nx + 4 * TX - 1) / (4 * TX), gy, nzc * nf);
        if (g.per) launch_chain(k_pred_v4<kPredPlanes, true>, grid, blk, st, g, kPredPlanes, nzc, w, t, tp, tn);
        else launch_chain(k_pred_v4<kPredPlanes, false>, grid, blk, st, g, kPredPlanes, nzc, w, t, tp, tn);
    } else {
        const dim3 grid((g.nx + TX - 1) / TX, gy, nzc * nf);
        if (g.per) launch_chain(k_pred_any<true>, grid, blk, st, g, zl, nzc, w, t, tp, tn);
        else launch_chain(k_pred_any<false>, grid, blk, st, g, zl, nzc, w, t, tp, tn);
    }
}

// The increments of run q of the plan, from u (double-float): K sweeps, then the
// combination.  T: (K + 1) vectors of `stride` floats, D: len vectors.
static void launch_pred(const PredPlan &pl, int q, const Geo &g, int nf, const DF *u, float *T, float *D,
                        size_t stride, cudaStream_t st) {
    const size_t n = (size_t)g.n * nf;
    const double ce = pl.scheme == CG_SCHEME_CRANK_NICOLSON ? 0.5 * pl.c : pl.c;
    const float e = (float)(2.0 * ce / (pl.lmax - 1.0));   // T_1 = (1 + 2 L / mu_max) T_0
    CGK_LAUNCH("pred_start", (double)n * 12, st,
               launch_chain(k_pred_start, dim3(stencil_grid((int)std::min<size_t>(n, 1u << 30))), dim3(kThreads), st, n,
                            df_pairs(g), u, T));
    {
        CGK_TIMED(loop_, "pred_sweep", (double)n * (8.0 + 12.0 * (pl.K[q] - 1)), st, pl.K[q]);
        for (int k = 0; k < pl.K[q]; ++k)
            CGK_LAUNCH_UNTIMED(st, launch_pred_sweep(g, nf, k ? 2.0f * e : e, T + k * stride,
                                                     k ? T + (k - 1) * stride : nullptr, T + (k + 1) * stride, st));
    }
    const int len = pl.len[q];
    CGK_LAUNCH("pred_combine", (double)n * 4 * (pl.K[q] + 1 + len), st, {
        if (len <= 2) launch_pred_combine<2>(n, stride, pl, q, T, D, st);
        else if (len <= 5) launch_pred_combine<5>(n, stride, pl, q, T, D, st);
        else if (len <= 8) launch_pred_combine<8>(n, stride, pl, q, T, D, st);
        else if (len <= 10) launch_pred_combine<10>(n, stride, pl, q, T, D, st);
        else if (len <= 13) launch_pred_combine<13>(n, stride, pl, q, T, D, st);
        else if (len <= 16) launch_pred_combine<16>(n, stride, pl, q, T, D, st);
        else launch_pred_combine<kPredMaxSteps>(n, stride, pl, q, T, D, st);
    });
}
// (vectors of D a combination of NS >= len steps writes)
static int pred_vectors(int len) {
    for (int ns : {2, 5, 8, 10, 13, 16})
        if (len <= ns) return ns;
    return kPredMaxSteps;
}

// Mixed-precision implicit steps: TS is the storage type of the inner solve (float or
// bf16), XT the type of the iterate and of the refinement residual (IEEE double, or
// the double-float pair DF).
template <class TS, class XT>
static cg_status diffuse_mixed(cg_mesh *m, int nf, double *cells, const cg_params *p, double T,
                               cg_report *rep, cudaStream_t st) {
    constexpr bool kDF = std::is_same<XT, DF>::value;
    static_assert(sizeof(XT) == 8, "iterate types are 8 bytes");
    const int n = (int)m->ncells;
    Geo g{m->nx, m->ny, m->nz, m->nx * m->ny, n, m->per};
    const bool cn = p->scheme == CG_SCHEME_CRANK_NICOLSON;
    const double dtau = T / p->nsteps;
    const double c = dtau / (m->dx * m->dx);
    const double ce = cn ? 0.5 * c : c;
    const double tol2 = p->tol * p->tol;
    const Sweep sw = make_sweep(g, nf);
    const int G = sw.nb;
    const dim3 blk(TX, TY);
    const Coef64 cf64 = coef64(ce);
    const Coef32 cf32 = coef32(ce);
    const CoefDF cfdf = coefdf(c, ce);

    // spectrum of A = I - ce L: [1, lmax] (a periodic axis of even length reaches 4 ce)
    const int dims[3] = {m->nx, m->ny, m->nz};
    double lmax = 1.0;
    for (int a = 0; a < 3; ++a) {
        double sv = std::sin(M_PI * (dims[a] - 1) / (2.0 * dims[a]));
        if (((m->per >> a) & 1) && dims[a] % 2 == 0) sv = 1.0;
        lmax += 4.0 * ce * sv * sv;
    }
    const double theta = 0.5 * (lmax + 1.0), delta = 0.5 * (lmax - 1.0);
    const double gamma = 1.0 / theta;
    const double eps_inner = sizeof(TS) == 2 ? 2e-3 : 1e-6;
    int m_it = cheb_iters(lmax, eps_inner);
    if (p->max_iter > 0 && m_it > p->max_iter) m_it = p->max_iter;
    double sigma_d = delta > 0.0 ? theta / delta : 0.0;
    const int coopG = coop_blocks(k_cheb_loop<TS>);
    const Items items = make_items(g, nf, coopG);
    // barrier_budget > 0: the whole inner solve as one cooperative launch with bounded
    // grid barriers between iterations; otherwise one launch per iteration.
    // (with sweep_shape = the resident code, barrier_budget bounds the resident waits)
    const bool persistent = p->barrier_budget > 0 && p->sweep_shape != kResidentCode;
    const long long budget = persistent ? p->barrier_budget : 0;

    // buffers: X0 (double-float copy of u^0), X1, X2, B (XT); R, Ya, Yb (TS)
    const size_t v64 = align_up((size_t)n * nf * 8), vts = align_up((size_t)n * nf * sizeof(TS));
    // the resident inner solve (whole mesh in shared memory) where it fits; its flags and
    // faces follow the vectors
    const ResidentPlan rp = (persistent || m->per) ? ResidentPlan{} : plan_resident<TS>(g, nf, m_it);
    CGK_TRY(m->ws_diffuse.ensure(4 * v64 + 5 * vts + (rp.ok ? rp.ws_bytes : 0)));
    char *wb = m->ws_diffuse.as<char>();
    char *rws = wb + 4 * v64 + 5 * vts;
    XT *X1 = (XT *)wb, *X2 = (XT *)(wb + v64), *B = (XT *)(wb + 2 * v64), *X0 = (XT *)(wb + 3 * v64);
    TS *R = (TS *)(wb + 4 * v64), *Ya = (TS *)(wb + 4 * v64 + vts), *Yb = (TS *)(wb + 4 * v64 + 2 * vts);
    // two more iterate buffers for two-iterations-per-launch sweeps
    TS *Yc = (TS *)(wb + 4 * v64 + 3 * vts), *Yd = (TS *)(wb + 4 * v64 + 4 * vts);
    TS *const R_ = R;
    // small workspace: partials | scalars | barrier | per-step residual history
    const size_t hist_off = 4096 + align_up((size_t)nf * 2 * G * 8) + 64 * sizeof(RefScal) + 256;
    const size_t hist_n = (size_t)p->nsteps * nf;
    CGK_TRY(m->ws_small.ensure(hist_off + hist_n * sizeof(RefScal)));
    double *partials = (double *)(m->ws_small.as<char>() + 4096);
    RefScal *sc = (RefScal *)(m->ws_small.as<char>() + 4096 + align_up((size_t)nf * 2 * G * 8));
    GridBar *gbar = (GridBar *)((char *)sc + 64 * sizeof(RefScal));
    RefScal *hist = (RefScal *)(m->ws_small.as<char>() + hist_off);
    CGK_CUDA(cudaMemsetAsync(sc, 0, nf * sizeof(RefScal), st));
    CGK_CUDA(cudaMemsetAsync(gbar, 0, sizeof(GridBar), st));
    CGK_TRY(m->h_small.ensure(4096 + std::max<size_t>(64 * sizeof(RefScal) + 256,
                                                      hist_n * sizeof(RefScal))));
    RefScal *hsc = (RefScal *)(m->h_small.as<char>() + 4096);
    GridBar *hgb = (GridBar *)((char *)hsc + 64 * sizeof(RefScal));
    // the shared expansion of the steps' first rounds, where it pays, nothing caps the
    // iterations, and its vectors may be held: T_k, the increments, the merged pass's partials
    const PredPlan *pred = nullptr;
    const size_t vpd = align_up((size_t)n * nf * 4);   // one FP32 vector of the expansion
    Sweep sw_mid = sw;
    OptUse opt;
    float *PT = nullptr, *PD = nullptr;
    double *mid_part = nullptr;
    if (kDF && !persistent) {
        const PredPlan &q = pred_plan(m, p->scheme, p->nsteps, cheb_iters(lmax, 1e-6), c, lmax);
        // (a round cap that the own rounds' start would exceed is refused as ever; a mesh whose
        // sweeps of two or four planes a block would exceed a grid's z extent keeps the own rounds)
        if (q.use && grid_z_fits(g, nf, pred_sweep_planes(g, nf)) &&
            p->max_iter >= std::max(q.maxm, q.maxK) && q.maxm <= kResidentMaxIters &&
            (p->max_rounds <= 0 || p->max_rounds >= (sizeof(TS) == 2 ? 5 : 2))) {
            sw_mid = mid_sweep(g, nf);
            const size_t nt = (size_t)(q.maxK + 1), nd = (size_t)pred_vectors(q.maxlen);
            if (opt.take(m->ws_opt, (nt + nd) * vpd + (size_t)nf * 2 * sw_mid.nb * 8)) {
                pred = &q;
                PT = m->ws_opt.as<float>();
                PD = PT + nt * (vpd / 4);
                mid_part = (double *)(PD + nd * (vpd / 4));
            }
        }
    }

    int cheb_code = p->sweep_shape;
    bool resident = false;
    if (m->per && cheb_code > 0 && !(cheb_code >= 100 && cheb_code < kPairCode) &&
        !(m->per == 1 && cheb_code >= kPairCode && cheb_code < kResidentCode))
        return fail(CG_EINVAL, "sweep_shape %d: with periodic axes only the z-marching and vectorised "
                    "sweeps (sweep_shape < 0 or 100 + z, or 0 for autotuning) apply, and two "
                    "iterations per launch (200 + z) with x the only periodic axis", cheb_code);
    if (cheb_code == kResidentCode) {
        if (!rp.ok)
            return fail(CG_EINVAL, "sweep_shape %d needs one field, nx %% 4 == 0, at most %d inner "
                        "iterations, one-launch solves and a mesh that fits in shared memory",
                        kResidentCode, kResidentMaxIters);
        resident = true;
    } else {
        if ((cheb_code > kResidentCode && cheb_code < kTmaCode) || cheb_code >= kTmaCode + 100)
            return fail(CG_EINVAL, "unknown sweep_shape %d", cheb_code);
        if (cheb_code >= kTmaCode &&
            (sizeof(TS) != 4 || !tma_sweep_fits(g) || cheb_code - kTmaCode < 1))
            return fail(CG_EINVAL, "sweep_shape %d needs FP32 inner storage, nx %% 4 == 0, no periodic axis and "
                        "1..99 planes", cheb_code);
        if (cheb_code >= kPairCode && cheb_code < kResidentCode && (!cheb2_fits(g) || cheb_code - kPairCode < 1))
            return fail(CG_EINVAL, "sweep_shape %d needs nx %% 4 == 0, nx <= %d and 1..99 planes",
                        cheb_code, kRowsMaxNx);
        if (cheb_code >= 100 && cheb_code < kPairCode && (m->nx % 4 != 0 || cheb_code - 100 < 1))
            return fail(CG_EINVAL, "sweep_shape %d needs nx %% 4 == 0 and 1..99 planes", cheb_code);
        if (cheb_code != 0 && cheb_code != 2 && cheb_code != 4 && cheb_code != 8 && cheb_code > -1 &&
            cheb_code < 100)
            return fail(CG_EINVAL, "unknown sweep_shape %d", cheb_code);
        const bool auto_shape = cheb_code == 0;
        // (before any capture that may launch the long-row pair kernel)
        if (auto_shape || (cheb_code >= kPairCode && cheb_code < kResidentCode))
            CGK_CUDA(rows_prepare<TS>());
        if (auto_shape) CGK_TRY(tune_cheb<TS>(m, g, nf, cf32, Ya, Yb, Yc, Yd, R, st, &cheb_code));
        if (auto_shape && rp.ok)
            CGK_TRY(tune_resident<TS>(m, g, rp, cheb_code, m_it, cf32, Ya, Yb, Yc, Yd, R, rws, st,
                                      &resident));
    }
    const int shape_used = resident ? kResidentCode : cheb_code;
    if (cheb_code >= kTmaCode) tma_prepare();
    // clock cycles a resident wait may take (about one second by default)
    const long long rbudget = (resident && p->barrier_budget > 0) ? p->barrier_budget : 2000000000LL;

    // ---- double-float modes: a fixed schedule captured as a CUDA graph.  The whole call
    // (conversion, every step's passes and inner iterations, R refinement rounds per
    // step) is captured once per signature and buffer set and replayed; the per-step
    // residuals it records are checked afterwards.  If a step fell short, the call runs
    // again from the untouched input (cells is written only after the check) with one
    // more round per step, and that count is remembered for the signature.  The same
    // input therefore always follows the same schedule.  (Persistent inner solves use
    // the adaptive host-driven loop below.)
    if constexpr (kDF) {
        // rounds per step: remembered for this signature, else an a-priori start (two
        // FP32 inner solves of ~1e-6 each, the first of them the shared expansion's where
        // it runs, reach 1e-13 from a residual below |b|)
        const int max_r = p->max_rounds > 0 ? p->max_rounds : 12;
        // (BF16 rounds gain about 2.5 digits each: five from r = c L u, three and the shared
        // expansion's from there)
        int R = sizeof(TS) == 2 ? (pred ? 4 : 5) : 2;
        RoundsEntry *remembered = nullptr;
        for (RoundsEntry &re : m->rounds)
            if (re.nf == nf && re.precision == p->precision && re.scheme == p->scheme &&
                re.nsteps == p->nsteps && re.T == T && re.tol == p->tol && re.predicted == (pred != nullptr) &&
                re.m_it == m_it) {
                R = re.rounds;
                remembered = &re;
            }
        if (!remembered) {
            m->rounds.push_back(
                RoundsEntry{nf, p->precision, p->scheme, p->nsteps, T, p->tol, R, pred != nullptr, m_it});
            remembered = &m->rounds.back();
        }
        XT *last_result = nullptr;
        for (; !persistent && R <= max_r; R = ++remembered->rounds) {
            const bool prof = prof_on();
            GraphEntry *ge = nullptr;
            for (auto it = m->graphs.begin(); it != m->graphs.end();) {
                if (it->batched) {
                    ++it;
                    continue;
                }
                if (it->gen_diffuse != m->ws_diffuse.gen || it->gen_small != m->ws_small.gen ||
                    (it->predicted && it->gen_opt != m->ws_opt.b.gen)) {
                    graph_release(*it);
                    it = m->graphs.erase(it);
                    continue;
                }
                if (it->nf == nf && it->precision == p->precision && it->scheme == p->scheme &&
                    it->nsteps == p->nsteps && it->rounds == R && it->T == T && it->tol == p->tol &&
                    it->cells == cells && it->profiled == prof && it->code == shape_used &&
                    it->predicted == (pred != nullptr) && it->m_it == m_it &&
                    it->wait_budget == rbudget)
                    ge = &*it;
                ++it;
            }
            XT *result = nullptr;
            if (!ge) {
                if (!m->capture_stream)
                    CGK_CUDA(cudaStreamCreateWithFlags(&m->capture_stream, cudaStreamNonBlocking));
                cudaStream_t cs = m->capture_stream;
                GraphEntry e;
                e.nf = nf;
                e.precision = p->precision;
                e.scheme = p->scheme;
                e.nsteps = p->nsteps;
                e.rounds = R;
                e.T = T;
                e.tol = p->tol;
                e.cells = cells;
                e.gen_diffuse = m->ws_diffuse.gen;
                e.gen_small = m->ws_small.gen;
                e.gen_opt = m->ws_opt.b.gen;
                e.profiled = prof;
                e.predicted = pred != nullptr;
                e.m_it = m_it;
                e.code = shape_used;
                e.wait_budget = rbudget;
                prof_capture_begin(&e.records, &e.kernels);
                cudaError_t cap_err = cudaSuccess;   // a launch refused while capturing
                cudaError_t ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
                if (ce == cudaSuccess) {
                    cudaMemsetAsync(hist, 0, hist_n * sizeof(RefScal), cs);
                    if (resident) cudaMemsetAsync(rws + (size_t)rp.nblocks * 4, 0, 4, cs);
                    CGK_LAUNCH("to_double_float", (double)n * nf * 16, cs,
                               launch_to_df(g, (size_t)n * nf, cells, (DF *)X0, cs));
                    XT *u = X0, *f1 = X1, *f2 = X2;
                    TS *y1_start = Ya;
                    int run = -1;   // the current run of the shared expansion
                    // merged passes between the steps of a run (one inner solve per step)
                    const bool mid = sizeof(TS) == 4 && pred && R == 2 && mid_fits(g, p->scheme);
                    bool merged_in = false;   // the step was started by a merged pass
                    for (int s2 = 0; s2 < p->nsteps; ++s2) {
                        RefScal *slot = hist + (size_t)s2 * nf;
                        const XT *bp_ = cn ? B : u;
                        TS *y1 = y1_start;
                        // the first step starts with its own pass; later steps were started
                        // by the previous step's last pass
                        const bool run_start = pred && run + 1 < (int)pred->start.size() &&
                                               pred->start[run + 1] == s2;
                        if ((s2 == 0 || (mid && run_start)) && (!pred || cn))
                            CGK_LAUNCH("refine_df_first", (double)n * nf * (8 + (cn ? 8 : 0) + 2 * sizeof(TS)), cs,
                                       launch_refine_df<TS, 0>(g, sw, nf, cfdf, p->scheme,
                                                               (const DF *)u, (const TS *)nullptr,
                                                               (const DF *)nullptr, (DF *)nullptr,
                                                               (DF *)B, R_, y1, (float)gamma,
                                                               partials, slot, slot, cs));
                        XT *xc = u;
                        if (pred) {   // the step's first round
                            if (run_start) launch_pred(*pred, ++run, g, nf, (const DF *)u, PT, PD, vpd / 4, cs);
                            const float *d0 = PD + (size_t)(s2 - pred->start[run]) * (vpd / 4);
                            // (a merged pass at the end of the step before has left this
                            // step's first residual, and u + d0 is formed where it is read)
                            if (merged_in) {
                            } else if (cn)
                                CGK_LAUNCH("refine_df", (double)n * nf * (24 + 3 * sizeof(TS)), cs,
                                           launch_refine_df<TS, 1, float>(g, sw, nf, cfdf, p->scheme, (const DF *)u, d0,
                                                                   (const DF *)bp_, (DF *)f1, (DF *)nullptr, R_, y1,
                                                                   (float)gamma, partials, slot, slot, cs));
                            else
                                CGK_LAUNCH("refine_df", (double)n * nf * (24 + 3 * sizeof(TS)), cs,
                                           launch_refine_df<TS, 4, float>(g, sw, nf, cfdf, p->scheme, (const DF *)u, d0,
                                                                   (const DF *)bp_, (DF *)f1, (DF *)nullptr, R_, y1,
                                                                   (float)gamma, partials, slot, slot, cs));
                            if (!merged_in) xc = f1;
                        }
                        const int mi = pred && sizeof(TS) == 4 ? pred_round_m(pred->m[s2], R) : m_it;   // inner iterations of a round
                        for (int r = pred ? 1 : 0; r < R; ++r) {
                            TS *yc = y1, *yp = nullptr, *yo = (y1 == Ya) ? Yb : Ya;
                            double om = 1.0;
                            if (mi > 1 && resident) {
                                TS *yf = cheb_final_buffer(yc, yo, mi);
                                CGK_LAUNCH(sizeof(TS) == 2 ? "cheb_resident_bf16" : "cheb_resident_fp32",
                                           (double)n * nf * sizeof(TS) * (3.0 + 4.0 * (mi - 2)), cs,
                                           {
                                               cudaError_t le = launch_resident<TS>(
                                                   g, rp, cf32, (float)gamma, sigma_d, mi, yc, R_,
                                                   yf, rws, rbudget, cs);
                                               if (cap_err == cudaSuccess) cap_err = le;
                                           });
                                yc = yf;
                            } else if (mi > 1 && cheb_code >= kPairCode && cheb_code < kResidentCode) {
                                const int np = (mi - 1) / 2, ns = (mi - 1) % 2;
                                CGK_TIMED(loop_, sizeof(TS) == 2 ? "cheb2_bf16" : "cheb2_fp32",
                                          (double)n * nf * sizeof(TS) *
                                              (np > 0 ? 4.0 + 5.0 * (np - 1) : 0.0) +
                                              (double)n * nf * sizeof(TS) * 4.0 * ns,
                                          cs, np + ns);
                                TS *const pool[4] = {yc, yo, Yc, Yd};   // y1 is Ya or Yb
                                yc = cheb_pairs<TS>(cheb_code - kPairCode, g, nf, cf32, (float)gamma,
                                                    sigma_d, mi, pool, R_, cs);
                            } else if (mi > 1) {
                                CGK_TIMED(loop_, sizeof(TS) == 2 ? "cheb_bf16" : "cheb_fp32",
                                          (double)n * nf * sizeof(TS) * (3.0 + 4.0 * (mi - 2)),
                                          cs, mi - 1);
                                for (int k = 1; k < mi; ++k) {
                                    if (sigma_d > 0.0)
                                        om = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma_d * sigma_d))
                                                      : 1.0 / (1.0 - om / (4.0 * sigma_d * sigma_d));
                                    TS *yn = yp ? yp : yo;
                                    CGK_LAUNCH_UNTIMED(cs, launch_cheb<TS>(cheb_code, g, nf, cf32,
                                                                           (float)gamma, (float)om,
                                                                           yc, yp, R_, yn, cs));
                                    yp = yc;
                                    yc = yn;
                                }
                            }
                            XT *xn = (xc == f1) ? f2 : f1;
                            // the next step's first Chebyshev iterate goes to Ya: it must not
                            // be the buffer holding this round's correction
                            const bool last = r == R - 1;
                            if constexpr (sizeof(TS) == 4)
                                if (last && mid) {
                                    const int i = s2 - pred->start[run];
                                    const float *e0 = PD + (size_t)i * (vpd / 4);
                                    merged_in = i + 1 < pred->len[run];
                                    y1 = (yc == Ya) ? Yb : Ya;
                                    if (merged_in) y1_start = y1;
                                    CGK_LAUNCH(merged_in ? "refine_mid" : "refine_mid_end",
                                               (double)n * nf * ((merged_in ? 36 : 24) + (cn ? 16 : 0)), cs,
                                               launch_refine_mid(g, sw_mid, cfdf, p->scheme, (const DF *)u, e0,
                                                                 (const float *)yc,
                                                                 merged_in ? e0 + vpd / 4 : nullptr, (const DF *)bp_,
                                                                 (DF *)xn, (DF *)B, (float *)R_, (float *)y1,
                                                                 (float)gamma, mid_part, slot, slot + nf, cs));
                                    xc = xn;
                                    break;
                                }
                            const bool emit = last && (s2 + 1 < p->nsteps) && (!pred || cn);
                            y1 = (yc == Ya) ? Yb : Ya;
                            if (emit) y1_start = y1;    // where the next step's y1 is
                            if (last && !emit)   // nothing follows from this pass's r
                                CGK_LAUNCH("refine_df_end", (double)n * nf * (24 + sizeof(TS)), cs,
                                           launch_refine_df<TS, 5>(g, sw, nf, cfdf, p->scheme,
                                                                   (const DF *)xc, (const TS *)yc,
                                                                   (const DF *)bp_, (DF *)xn,
                                                                   (DF *)nullptr, R_, y1,
                                                                   (float)gamma, partials, slot,
                                                                   slot, cs));
                            else if (emit)
                                CGK_LAUNCH("refine_df_last", (double)n * nf * (24 + 3 * sizeof(TS) + (cn ? 8 : 0)), cs,
                                           launch_refine_df<TS, 2>(g, sw, nf, cfdf, p->scheme,
                                                                   (const DF *)xc, (const TS *)yc,
                                                                   (const DF *)bp_, (DF *)xn,
                                                                   (DF *)B, R_, y1, (float)gamma,
                                                                   partials, slot, slot + nf, cs));
                            else
                                CGK_LAUNCH("refine_df", (double)n * nf * (24 + 3 * sizeof(TS)), cs,
                                           launch_refine_df<TS, 1>(g, sw, nf, cfdf, p->scheme,
                                                                   (const DF *)xc, (const TS *)yc,
                                                                   (const DF *)bp_, (DF *)xn,
                                                                   (DF *)nullptr, R_, y1,
                                                                   (float)gamma, partials, slot,
                                                                   slot, cs));
                            xc = xn;
                        }
                        XT *old_u = u, *other = (xc == f1) ? f2 : f1;
                        u = xc;
                        f1 = old_u;
                        f2 = other;
                    }
                    result = u;
                    cudaGraph_t graph = nullptr;
                    ce = cudaStreamEndCapture(cs, &graph);
                    if (ce == cudaSuccess) ce = cap_err;
                    if (ce == cudaSuccess) ce = cudaGraphInstantiate(&e.exec, graph, 0);
                    if (graph) cudaGraphDestroy(graph);
                }
                prof_capture_end();
                if (ce != cudaSuccess || !e.exec) {
                    graph_release(e);
                    cudaGetLastError();
                    return cuda_fail(ce == cudaSuccess ? cudaErrorUnknown : ce, "graph capture",
                                     __FILE__, __LINE__);
                }
                e.result = result;
                m->graphs.push_back(e);
                ge = &m->graphs.back();
            }
            result = (XT *)ge->result;
            CGK_CUDA(cudaGraphLaunch(ge->exec, st));
            RefScal *hh = (RefScal *)(m->h_small.as<char>() + 4096);
            CGK_CUDA(cudaMemcpyAsync(hh, hist, hist_n * sizeof(RefScal), cudaMemcpyDeviceToHost, st));
            int *herr = (int *)(m->h_small.as<char>() + 1024);
            *herr = 0;
            if (resident)
                CGK_CUDA(cudaMemcpyAsync(herr, rws + (size_t)rp.nblocks * 4, 4, cudaMemcpyDeviceToHost, st));
            CGK_CUDA(cudaStreamSynchronize(st));
            prof_account_replay(*ge);
            if (*herr)
                return fail(CG_ETIMEOUT, "cg_diffuse: a wait of the resident inner solve gave up");
            if (cheb_code >= kTmaCode && tma_wait_failed(st))
                return fail(CG_ETIMEOUT, "cg_diffuse: a wait of the TMA-staged sweep gave up");
            bool ok = true;
            double worst_g = 0.0;
            for (size_t i = 0; i < hist_n; ++i) {
                ok = ok && (hh[i].rr <= tol2 * hh[i].bb);
                worst_g = std::max(worst_g, hh[i].bb > 0 ? std::sqrt(hh[i].rr / hh[i].bb) : 0.0);
            }
            if (ok) {
                CGK_LAUNCH("from_double_float", (double)n * nf * 16, st,
                           launch_from_df(g, (size_t)n * nf, (const DF *)result, cells, st));
                CGK_CUDA(cudaGetLastError());
                CGK_CUDA(cudaStreamSynchronize(st));
                if (rep) {
                    long long apps = 1 + (long long)p->nsteps * R * m_it;
                    if (pred) {   // expansions, then per step one pass and R - 1 rounds
                        apps = (cn ? 1 : 0) + p->nsteps;
                        for (int K : pred->K) apps += K;
                        for (int mi : pred->m)
                            apps += (long long)(R - 1) * (sizeof(TS) == 4 ? pred_round_m(mi, R) : m_it);
                    }
                    rep->iters = apps * nf;
                    rep->refine_rounds = (long long)p->nsteps * R;
                    rep->cell_updates = apps * nf * (long long)n;
                    rep->final_rel_residual = worst_g;
                    rep->inner_iters_per_round = pred && sizeof(TS) == 4 ? pred_round_m(pred->maxm, R) : m_it;
                    rep->sweep_shape_used = shape_used;
                }
                return CG_OK;
            }
            // a step needed more rounds than the schedule: try again with one more
            last_result = result;
        }
        if (!persistent) {
            remembered->rounds = max_r;
            if (last_result) {   // leave the last iterate in place
                CGK_LAUNCH("from_double_float", (double)n * nf * 16, st,
                           launch_from_df(g, (size_t)n * nf, (const DF *)last_result, cells, st));
                CGK_CUDA(cudaStreamSynchronize(st));
            }
            return fail(CG_ENOCONV, "cg_diffuse: refinement did not reach tol with %d rounds "
                                    "per step", max_r);
        }
    }

    const int max_rounds = p->max_rounds > 0 ? p->max_rounds : 12;
    int sched = 2;   // rounds before the first convergence check of a step
    long long applications = 0, rounds_total = 0;
    double worst = 0.0;
    XT *ubuf = (XT *)cells;                  // u^n (also b for implicit Euler)
    if (kDF) {
        CGK_LAUNCH("to_double_float", (double)n * nf * 16, st,
                   launch_to_df(g, (size_t)n * nf, cells, (DF *)X0, st));
        ubuf = X0;
    }
    XT *F1 = X1, *F2 = X2;                   // the two buffers not holding u^n
    if (resident) CGK_CUDA(cudaMemsetAsync(rws + (size_t)rp.nblocks * 4, 0, 4, st));
    bool converged = true, timed_out = false;
    int s = 0;
    for (; s < p->nsteps; ++s) {
        const XT *bptr = cn ? B : ubuf;
        TS *y1buf = Ya;
        if constexpr (kDF)
            CGK_LAUNCH("refine_df_first", (double)n * nf * (8 + (cn ? 8 : 0) + 2 * sizeof(TS)), st,
                       (launch_refine_df<TS, 0>(g, sw, nf, cfdf, p->scheme, (const DF *)ubuf,
                                                (const TS *)nullptr, (const DF *)nullptr,
                                                (DF *)nullptr, (DF *)B, R, y1buf, (float)gamma,
                                                partials, sc, sc, st)));
        else
            CGK_LAUNCH("refine64_first", (double)n * nf * (8 + (cn ? 8 : 0) + 2 * sizeof(TS)), st,
                       (k_refine<TS, true><<<sw.grid, blk, 0, st>>>(
                           g, sw.zlen, sw.nzc, c, cf64, p->scheme, ubuf, nullptr, nullptr, nullptr,
                           B, R, y1buf, (float)gamma, partials, sc)));
        CGK_CUDA(cudaGetLastError());
        applications += 1;
        XT *xcur = ubuf;
        int rounds = 0;
        converged = false;
        while (rounds < max_rounds) {
            // inner Chebyshev solve of A d = r, starting from y1 = gamma r: one cooperative
            // launch runs iterations 2..m with grid barriers in between
            TS *ycur = y1buf, *yprev = nullptr, *yother = (y1buf == Ya) ? Yb : Ya;
            if (m_it > 1 && persistent) {
                CGK_CUDA(cudaMemsetAsync(gbar, 0, sizeof(GridBar), st));
                Geo ga = g;
                int a_zlen = items.zlen, a_nzc = items.nzc, a_gx = items.gx, a_gy = items.gy;
                int a_n = items.n, a_m = m_it;
                float a_gamma = (float)gamma;
                Coef32 a_cf = cf32;
                TS *a_y1 = y1buf, *a_oth = yother;
                const TS *a_r = R;
                long long a_budget = budget;
                void *args[] = {&ga,      &a_zlen, &a_nzc, &a_gx,  &a_gy,  &a_n,   &a_cf,   &a_gamma,
                                &sigma_d, &a_m,    &a_y1,  &a_oth, &a_r,   &gbar,  &a_budget};
                CGK_LAUNCH(sizeof(TS) == 2 ? "cheb_loop_bf16" : "cheb_loop_fp32",
                           (double)n * nf * sizeof(TS) * (3.0 + 4.0 * (m_it - 2)), st,
                           CGK_CUDA(cudaLaunchCooperativeKernel((const void *)k_cheb_loop<TS>,
                                                                dim3(coopG), dim3(TX, TY), args, 0,
                                                                st)));
            }
            if (m_it > 1 && !persistent && !resident && cheb_code >= kPairCode && cheb_code < kResidentCode) {
                const int np = (m_it - 1) / 2, ns = (m_it - 1) % 2;
                CGK_TIMED(loop_, sizeof(TS) == 2 ? "cheb2_bf16" : "cheb2_fp32",
                          (double)n * nf * sizeof(TS) * ((np > 0 ? 4.0 + 5.0 * (np - 1) : 0.0) + 4.0 * ns),
                          st, np + ns);
                TS *const pool[4] = {ycur, yother, Yc, Yd};   // y1 is Ya or Yb
                ycur = cheb_pairs<TS>(cheb_code - kPairCode, g, nf, cf32, (float)gamma, sigma_d,
                                      m_it, pool, R, st);
            } else if (m_it > 1 && resident) {
                TS *yf = cheb_final_buffer(ycur, yother, m_it);
                CGK_LAUNCH(sizeof(TS) == 2 ? "cheb_resident_bf16" : "cheb_resident_fp32",
                           (double)n * nf * sizeof(TS) * (3.0 + 4.0 * (m_it - 2)), st,
                           CGK_CUDA(launch_resident<TS>(g, rp, cf32, (float)gamma, sigma_d, m_it,
                                                        ycur, R, yf, rws, rbudget, st)));
                ycur = yf;
            } else {
                double om = 1.0;
                for (int k = 1; k < m_it; ++k) {
                    if (sigma_d > 0.0)
                        om = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma_d * sigma_d))
                                      : 1.0 / (1.0 - om / (4.0 * sigma_d * sigma_d));
                    TS *ynext = yprev ? yprev : yother;
                    if (!persistent)
                        CGK_LAUNCH(sizeof(TS) == 2 ? "cheb_bf16" : "cheb_fp32",
                                   (double)n * nf * sizeof(TS) * (yprev ? 4 : 3), st,
                                   launch_cheb<TS>(cheb_code, g, nf, cf32, (float)gamma, (float)om,
                                                   ycur, yprev, R, ynext, st));
                    yprev = ycur;
                    ycur = ynext;
                }
                CGK_CUDA(cudaGetLastError());
            }
            applications += m_it - 1;
            // x += d and the new FP64 residual; y1 goes to the buffer d is not in
            XT *xnext = (xcur == F1) ? F2 : F1;
            y1buf = (ycur == Ya) ? Yb : Ya;
            if constexpr (kDF)
                CGK_LAUNCH("refine_df", (double)n * nf * (24 + 3 * sizeof(TS)), st,
                           (launch_refine_df<TS, 1>(g, sw, nf, cfdf, p->scheme, (const DF *)xcur,
                                                    (const TS *)ycur, (const DF *)bptr,
                                                    (DF *)xnext, (DF *)nullptr, R, y1buf,
                                                    (float)gamma, partials, sc, sc, st)));
            else
                CGK_LAUNCH("refine64", (double)n * nf * (24 + 3 * sizeof(TS)), st,
                           (k_refine<TS, false><<<sw.grid, blk, 0, st>>>(
                               g, sw.zlen, sw.nzc, c, cf64, p->scheme, xcur, ycur, bptr, xnext,
                               nullptr, R, y1buf, (float)gamma, partials, sc)));
            CGK_CUDA(cudaGetLastError());
            applications += 1;
            ++rounds;
            xcur = xnext;
            if (rounds >= sched) {
                CGK_CUDA(cudaMemcpyAsync(hsc, sc, nf * sizeof(RefScal), cudaMemcpyDeviceToHost, st));
                if (persistent)
                    CGK_CUDA(cudaMemcpyAsync(hgb, gbar, sizeof(GridBar), cudaMemcpyDeviceToHost, st));
                if (resident)   // the resident error word, in the barrier's err slot
                    CGK_CUDA(cudaMemcpyAsync(&hgb->err, rws + (size_t)rp.nblocks * 4, 4,
                                             cudaMemcpyDeviceToHost, st));
                CGK_CUDA(cudaStreamSynchronize(st));
                if ((persistent || resident) && hgb->err) {
                    timed_out = true;
                    break;
                }
                converged = true;
                for (int f = 0; f < nf; ++f) converged = converged && (hsc[f].rr <= tol2 * hsc[f].bb);
                if (converged) break;
            }
        }
        rounds_total += rounds;
        for (int f = 0; f < nf; ++f) {
            double rel = hsc[f].bb > 0 ? std::sqrt(hsc[f].rr / hsc[f].bb) : 0.0;
            if (rel > worst) worst = rel;
        }
        if (timed_out) break;
        sched = rounds > 1 ? rounds : 1;
        // u^{n+1} = xcur; the other two buffers become the spares
        XT *old_u = ubuf;
        XT *other = (xcur == F1) ? F2 : F1;
        ubuf = xcur;
        F1 = old_u;
        F2 = other;
        if (!converged) break;
    }
    if (kDF)
        CGK_LAUNCH("from_double_float", (double)n * nf * 16, st,
                   launch_from_df(g, (size_t)n * nf, (const DF *)ubuf, cells, st));
    else if ((double *)ubuf != cells)
        CGK_CUDA(cudaMemcpyAsync(cells, ubuf, (size_t)n * nf * 8, cudaMemcpyDeviceToDevice, st));
    CGK_CUDA(cudaStreamSynchronize(st));
    if (rep) {
        rep->iters = applications * nf;
        rep->refine_rounds = rounds_total;
        rep->cell_updates = applications * nf * (long long)n;
        rep->final_rel_residual = worst;
        rep->inner_iters_per_round = m_it;
        rep->sweep_shape_used = persistent ? 0 : shape_used;
    }
    if (timed_out)
        return fail(CG_ETIMEOUT, "cg_diffuse: a %s of the inner solve gave up (step %d)",
                    resident ? "neighbour wait" : "grid barrier", s);
    if (!persistent && !resident && cheb_code >= kTmaCode && tma_wait_failed(st))
        return fail(CG_ETIMEOUT, "cg_diffuse: a wait of the TMA-staged sweep gave up");
    if (!converged)
        return fail(CG_ENOCONV, "cg_diffuse: refinement did not reach tol in step %d", s);
    return CG_OK;
}

cg_status diffuse_structured_run(cg_mesh *m, int nf, double *cells, const cg_params *p,
                                 cg_report *rep, cudaStream_t st) {
    double T = p->bandwidth > 0.0 ? p->bandwidth * p->bandwidth / 4.0 : p->T;
    if (p->scheme == CG_SCHEME_EXPLICIT_EULER) return diffuse_explicit(m, nf, cells, p, T, rep, st);
    if (p->precision == CG_PREC_FP64) return diffuse_fp64(m, nf, cells, p, T, rep, st);
    switch (p->precision) {
        case CG_PREC_FP32_REFINE: return diffuse_mixed<float, double>(m, nf, cells, p, T, rep, st);
        case CG_PREC_BF16_REFINE: return diffuse_mixed<__nv_bfloat16, double>(m, nf, cells, p, T, rep, st);
        case CG_PREC_FP32_DF_REFINE: return diffuse_mixed<float, DF>(m, nf, cells, p, T, rep, st);
        default: return diffuse_mixed<__nv_bfloat16, DF>(m, nf, cells, p, T, rep, st);
    }
}


// ============================================================================ batched host
// Host-side plan of a batched call for one z-chunk length: per-snapshot descriptors,
// Chebyshev weights, and the work items of the refinement and Chebyshev phases.
template <class TS>
struct BatchPlan {
    std::vector<SnapDesc<TS>> descs;
    std::vector<float> omegas;
    std::vector<size_t> omega_off;
    std::vector<BItem> ritems, citems;
    std::vector<BItem> pitems;     // the shared expansion's sweeps (one field)
    std::vector<float> pcoef;
    std::vector<size_t> pc_off;
    std::vector<size_t> opt_off;   // the expansions' vectors in one optional buffer
    size_t opt_bytes = 0;
    bool pred = false;
    int Kmax = 0;
    std::vector<int> first_item;   // per (snapshot, field), into ritems
    int mmax = 2;
    long long cells_total = 0;
};

template <class TS>
static cg_status batch_plan(int nsnap, cg_mesh *const *meshes, int nf, double *const *cells,
                            const cg_params *p, const double *bandwidths, int zlen,
                            bool want_pred, int R, BatchPlan<TS> &P) {
    const bool cn = p->scheme == CG_SCHEME_CRANK_NICOLSON;
    const double eps_inner = sizeof(TS) == 2 ? 2e-3 : 1e-6;
    P = BatchPlan<TS>();
    P.descs.resize((size_t)nsnap);
    P.omega_off.resize((size_t)nsnap);
    P.pc_off.resize((size_t)nsnap);
    P.opt_off.resize((size_t)nsnap);
    // the shared expansion serves the batch where it pays for every snapshot: FP32 inner
    // storage, one run of steps, rows the flat-plane engine takes
    P.pred = sizeof(TS) == 4 && want_pred && p->nsteps <= kPredMaxSteps;
    for (int s = 0; s < nsnap; ++s) {
        cg_mesh *m = meshes[s];
        SnapDesc<TS> &d = P.descs[s];
        const int n = (int)m->ncells;
        d.g = Geo{m->nx, m->ny, m->nz, m->nx * m->ny, n};
        const double b = bandwidths ? bandwidths[s] : p->bandwidth;
        const double T = b > 0.0 ? b * b / 4.0 : p->T;
        const double c = (T / p->nsteps) / (m->dx * m->dx);
        const double ce = cn ? 0.5 * c : c;
        const int dims[3] = {m->nx, m->ny, m->nz};
        double lmax = 1.0;
        for (int a = 0; a < 3; ++a) {
            double sv = std::sin(M_PI * (dims[a] - 1) / (2.0 * dims[a]));
            lmax += 4.0 * ce * sv * sv;
        }
        const double theta = 0.5 * (lmax + 1.0), delta = 0.5 * (lmax - 1.0);
        int mi = cheb_iters(lmax, eps_inner);
        if (mi < 2) mi = 2;
        const PredPlan *pl = P.pred ? &pred_plan(m, p->scheme, p->nsteps, mi, c, lmax) : nullptr;
        if (pl && (!pl->use || m->nx > kFlatMaxNx)) P.pred = false;
        if (!P.pred) pl = nullptr;
        if (want_pred && sizeof(TS) == 4 && !P.pred && s > 0 && P.Kmax > 0)   // start over without it
            return batch_plan<TS>(nsnap, meshes, nf, cells, p, bandwidths, zlen, false, R, P);
        // (with two iterations fewer, 14 instead of 16 at b = 3 dx, 64 snapshots of five fields take
        // 79.8 instead of 86.5 ms, but the error against 64 bits, 2.1e-14 with own rounds, is 2.5e-14
        // instead of 1.1e-14)
        if (pl) mi = R > 2 ? pred_round_m(pl->maxm, R) : std::max(mi, pl->maxm);
        if (mi & 1) ++mi;
        d.m = mi;
        P.mmax = std::max(P.mmax, mi);
        d.gamma = (float)(1.0 / theta);
        d.cf32 = coef32(ce);
        d.cfdf = coefdf(c, ce);
        d.scheme = p->scheme;
        P.omega_off[s] = P.omegas.size();
        double sigma = delta > 0.0 ? theta / delta : 0.0, om = 1.0;
        P.omegas.push_back(1.0f);
        for (int k = 1; k < mi; ++k) {
            if (sigma > 0.0)
                om = (k == 1) ? 1.0 / (1.0 - 1.0 / (2.0 * sigma * sigma))
                              : 1.0 / (1.0 - om / (4.0 * sigma * sigma));
            P.omegas.push_back((float)om);
        }
        d.gx = (m->nx + TX - 1) / TX;
        d.gy = (m->ny + TY - 1) / TY;
        d.zlen = std::min(zlen, m->nz);
        d.nzc = (m->nz + d.zlen - 1) / d.zlen;
        d.v4 = (m->nx % 4 == 0) ? 1 : 0;
        d.flat = m->nx <= kFlatMaxNx ? 1 : 0;
        d.nch = (m->nx * m->ny + kFlatCpt * kThreads - 1) / (kFlatCpt * kThreads);
        d.nchr = (m->nx * m->ny + kFlatCptDF * kThreads - 1) / (kFlatCptDF * kThreads);
        d.gx4 = (m->nx + 4 * TX - 1) / (4 * TX);
        d.zlen4 = d.zlen;
        d.nzc4 = d.nzc;
        d.pts = d.flat ? (m->nx * m->ny + 3) / 4 * 4 : m->nx * m->ny;
        d.vcu = (m->dx * m->dx) * m->dx;
        // per-snapshot solver vectors, owned by the snapshot's mesh
        const size_t v64 = align_up((size_t)n * nf * 8);
        const size_t vts = align_up((size_t)m->nz * d.pts * nf * sizeof(TS));
        const size_t t1 = align_up((size_t)m->nz * d.pts * 4);
        if (pl) {
            P.opt_off[s] = P.opt_bytes;
            P.opt_bytes += p->nsteps * vts + (pl->maxK + 1) * t1;
            d.K = pl->K[0];
            d.w = (float)(2.0 * ce / (lmax - 1.0));
            P.Kmax = std::max(P.Kmax, d.K);
            P.pc_off[s] = P.pcoef.size();
            P.pcoef.insert(P.pcoef.end(), pl->coef[0].begin(), pl->coef[0].end());
            for (int zc = 0; zc < d.nzc; ++zc)
                for (int ch = 0; ch < d.nch; ++ch) P.pitems.push_back(BItem{s, ch, 0, zc});
        }
        CGK_TRY(m->ws_diffuse.ensure(4 * v64 + 3 * vts));
        char *wb = m->ws_diffuse.as<char>();
        d.U = (DF *)wb;
        d.X1 = (DF *)(wb + v64);
        d.X2 = (DF *)(wb + 2 * v64);
        d.B = (DF *)(wb + 3 * v64);
        d.R = (TS *)(wb + 4 * v64);
        d.Ya = (TS *)(wb + 4 * v64 + vts);
        d.Yb = (TS *)(wb + 4 * v64 + 2 * vts);
        d.cells = cells[s];
        for (int f = 0; f < nf; ++f) {
            P.first_item.push_back((int)P.ritems.size());
            if (d.flat) {   // plane chunks x z-chunks
                for (int zc = 0; zc < d.nzc; ++zc) {
                    for (int ch = 0; ch < d.nchr; ++ch) P.ritems.push_back(BItem{s, ch, 0, f * d.nzc + zc});
                    for (int ch = 0; ch < d.nch; ++ch) P.citems.push_back(BItem{s, ch, 0, f * d.nzc + zc});
                }
                continue;
            }
            for (int zc = 0; zc < d.nzc; ++zc)
                for (int by = 0; by < d.gy; ++by)
                    for (int bx = 0; bx < d.gx; ++bx) P.ritems.push_back(BItem{s, bx, by, f * d.nzc + zc});
            const int cx = d.v4 ? d.gx4 : d.gx;
            for (int zc = 0; zc < d.nzc4; ++zc)
                for (int by = 0; by < d.gy; ++by)
                    for (int bx = 0; bx < cx; ++bx) P.citems.push_back(BItem{s, bx, by, f * d.nzc4 + zc});
        }
        P.cells_total += (long long)n;
    }
    P.first_item.push_back((int)P.ritems.size());
    return CG_OK;
}

// The batch arena on the first mesh: descriptors | items | partials | hist | barrier | failure
// count | output pointers | masses | expansion items | Chebyshev weights | expansion
// coefficients.  The last two differ in length between calls of one shape (they follow the
// bandwidths) and are reached through the descriptors alone, so they come behind everything
// whose address a captured launch holds.
struct BatchArena {
    char *ab = nullptr;
    size_t o_desc = 0, o_om = 0, o_ri = 0, o_ci = 0, o_fi = 0, o_prr = 0, o_pbb = 0, o_hist = 0,
           o_gb = 0, o_bad = 0, o_out = 0, o_mass = 0, o_pi = 0, o_pc = 0, total = 0;
    size_t nh = 0;
    // every offset that a captured launch holds
    std::vector<size_t> offsets() const {
        return {o_desc, o_ri, o_ci, o_fi, o_prr, o_pbb, o_hist, o_gb, o_bad, o_out, o_mass, o_pi};
    }
};

template <class TS>
static BatchArena batch_layout(const BatchPlan<TS> &P, int nsnap, int nf, int nsteps) {
    BatchArena A;
    const size_t nr = P.ritems.size();
    A.o_desc = 0;
    A.o_ri = align_up(A.o_desc + P.descs.size() * sizeof(SnapDesc<TS>));
    A.o_ci = align_up(A.o_ri + P.ritems.size() * sizeof(BItem));
    A.o_fi = align_up(A.o_ci + P.citems.size() * sizeof(BItem));
    A.o_prr = align_up(A.o_fi + P.first_item.size() * sizeof(int));
    A.o_pbb = align_up(A.o_prr + (size_t)nsteps * nr * 8);
    A.o_hist = align_up(A.o_pbb + (size_t)nsteps * nr * 8);
    A.nh = (size_t)nsteps * nsnap * nf;
    A.o_gb = align_up(A.o_hist + A.nh * sizeof(double2));
    A.o_bad = align_up(A.o_gb + sizeof(GridBar));
    A.o_out = align_up(A.o_bad + sizeof(unsigned int));
    A.o_mass = align_up(A.o_out + (size_t)nsnap * sizeof(double *));
    A.o_pi = align_up(A.o_mass + 2 * (size_t)nsnap * nf * 8);
    A.o_om = align_up(A.o_pi + P.pitems.size() * sizeof(BItem));
    A.o_pc = align_up(A.o_om + P.omegas.size() * sizeof(float));
    A.total = align_up(A.o_pc + P.pcoef.size() * sizeof(float));
    return A;
}

// Uploads the plan into the arena (ensured large enough by the caller).  The host
// vectors are read by the copies, so the stream is synchronised before returning.
template <class TS>
static cg_status batch_upload(BatchPlan<TS> &P, BatchArena &A, char *ab, int nsnap,
                              double *const *cells, cudaStream_t st) {
    A.ab = ab;
    for (int s = 0; s < nsnap; ++s) {
        P.descs[s].omega = (const float *)(ab + A.o_om) + P.omega_off[s];
        P.descs[s].pc = (const float *)(ab + A.o_pc) + P.pc_off[s];
    }
    if (P.pred) {
        CGK_CUDA(cudaMemcpyAsync(ab + A.o_pi, P.pitems.data(), P.pitems.size() * sizeof(BItem),
                                 cudaMemcpyHostToDevice, st));
        CGK_CUDA(cudaMemcpyAsync(ab + A.o_pc, P.pcoef.data(), P.pcoef.size() * sizeof(float),
                                 cudaMemcpyHostToDevice, st));
    }
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_desc, P.descs.data(), P.descs.size() * sizeof(SnapDesc<TS>),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_om, P.omegas.data(), P.omegas.size() * sizeof(float),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_ri, P.ritems.data(), P.ritems.size() * sizeof(BItem),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_ci, P.citems.data(), P.citems.size() * sizeof(BItem),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_fi, P.first_item.data(), P.first_item.size() * sizeof(int),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaMemcpyAsync(ab + A.o_out, cells, (size_t)nsnap * sizeof(double *),
                             cudaMemcpyHostToDevice, st));
    CGK_CUDA(cudaStreamSynchronize(st));
    return CG_OK;
}

// One inner solve per step: the steps of a batch with the expansion end in merged passes,
// whose last iterate is in X2 after an odd number of steps.
static bool batch_mid(bool pred, int R) { return pred && R == 2; }
static int batch_in_x2(bool pred, int R, int nsteps) { return batch_mid(pred, R) && nsteps % 2 ? 1 : 0; }

// The launches of the shared expansion (before either schedule): u^0 -> double-float, then
// per field the recurrence and the combination.
template <class TS>
static cg_status batch_issue_pred(const BatchPlan<TS> &P, const BatchArena &A, int nf, int nsteps,
                                  cudaStream_t st) {
    const SnapDesc<TS> *dsd = (const SnapDesc<TS> *)(A.ab + A.o_desc);
    const BItem *items = (const BItem *)(A.ab + A.o_pi);
    const int nsnap = (int)P.descs.size();
    const double cells = (double)P.cells_total;
    CGK_LAUNCH("bconvert", cells * nf * 16.0, st,
               launch_chain(k_bconvert<TS>, dim3(num_sms() * 2, nsnap), dim3(TX, TY), st, dsd, nf));
    for (int f = 0; f < nf; ++f) {
        CGK_LAUNCH("bpred_start", cells * 12.0, st,
                   launch_chain(k_bpred_start<TS>, dim3(num_sms(), nsnap), dim3(kThreads), st, dsd, f));
        for (int k = 0; k < P.Kmax; ++k)
            CGK_LAUNCH("bpred", cells * 12.0, st,
                       launch_chain(k_bpred<TS>, dim3((unsigned)P.pitems.size()), dim3(TX, TY), st, dsd, items, k));
        const dim3 grid(num_sms(), nsnap);
        CGK_LAUNCH("bpred_combine", cells * 4.0 * (P.Kmax + 1 + nsteps), st, {
            if (nsteps <= 5) launch_chain(k_bpred_combine<TS, 5>, grid, dim3(kThreads), st, dsd, nf, f, nsteps);
            else if (nsteps <= 10) launch_chain(k_bpred_combine<TS, 10>, grid, dim3(kThreads), st, dsd, nf, f, nsteps);
            else launch_chain(k_bpred_combine<TS, kPredMaxSteps>, grid, dim3(kThreads), st, dsd, nf, f, nsteps);
        });
    }
    CGK_CUDA(cudaGetLastError());
    return CG_OK;
}

// The phased schedule's launches on stream st (one per phase, in k_batched's order),
// each with its algorithmic bytes: a Chebyshev iteration reads y_k, y_{k-1} and r and
// writes y_{k+1} of every snapshot that runs it; a refinement pass reads the double-float
// iterate and right-hand side and the correction and writes the iterate, the residual
// and the first Chebyshev iterate.
template <class TS>
static cg_status batch_issue_phased(const BatchPlan<TS> &P, const BatchArena &A, int nf,
                                    int nsteps, int R, bool pred, cudaStream_t st) {
    char *ab = A.ab;
    const SnapDesc<TS> *dsd = (const SnapDesc<TS> *)(ab + A.o_desc);
    const BItem *dri = (const BItem *)(ab + A.o_ri), *dci = (const BItem *)(ab + A.o_ci);
    double *prr = (double *)(ab + A.o_prr), *pbb = (double *)(ab + A.o_pbb);
    const int nr = (int)P.ritems.size(), nc = (int)P.citems.size();
    const int nsnap = (int)P.descs.size();
    const double cells_f = (double)P.cells_total * nf;
    const char *cname = sizeof(TS) == 2 ? "bcheb_bf16" : "bcheb_fp32";
    const char *rname = sizeof(TS) == 2 ? "brefine_bf16" : "brefine_fp32";
    std::vector<double> cheb_bytes((size_t)P.mmax, 0.0);
    for (const auto &d : P.descs)
        for (int k = 1; k < std::min(d.m, P.mmax); ++k) cheb_bytes[(size_t)k] += (double)d.g.n * nf * 4.0 * sizeof(TS);
    const double ref_bytes = cells_f * (24.0 + 3.0 * sizeof(TS));
    const bool cn = P.descs[0].scheme == CG_SCHEME_CRANK_NICOLSON, mid = batch_mid(pred, R);
    if (!pred)
        CGK_LAUNCH("bconvert", cells_f * 16.0, st,
                   launch_chain(k_bconvert<TS>, dim3(num_sms() * 2, nsnap), dim3(TX, TY), st, dsd, nf));
    for (int step = 0; step < nsteps; ++step) {
        if (step == 0 && (!pred || cn))
            CGK_LAUNCH(rname, cells_f * (8.0 + 2.0 * sizeof(TS)), st,
                       launch_chain(k_brefine<TS>, dim3(nr), dim3(TX, TY), st, dsd, nf, dri, 1, 0, R, pbb,
                                    (double *)nullptr, -1, (double *)nullptr));
        for (int round = 1; round <= R; ++round) {
            const bool shared = pred && round == 1;
            if (shared && mid && step > 0) continue;
            for (int k = 1; k < (shared ? 1 : P.mmax); ++k)
                CGK_LAUNCH(cname, cheb_bytes[(size_t)k], st,
                           launch_chain(k_bcheb<TS>, dim3(nc), dim3(TX, TY), st, dsd, dci, k));
            if constexpr (sizeof(TS) == 4)
                if (mid && round == R) {
                    const int end = step + 1 == nsteps ? 1 : 0;
                    CGK_LAUNCH("bmid_fp32", cells_f * (end ? 24.0 : 36.0), st,
                               launch_chain(k_bmid<TS>, dim3(nr), dim3(TX, TY), st, dsd, nf, dri, step, end,
                                            prr + (size_t)step * nr, pbb + (size_t)(end ? step : step + 1) * nr));
                    continue;
                }
            double *part = round == R ? prr + (size_t)step * nr : nullptr;
            double *next = round == R && step + 1 < nsteps && (!pred || cn) ? pbb + (size_t)(step + 1) * nr : nullptr;
            double *partb = shared && !cn ? pbb + (size_t)step * nr : nullptr;
            CGK_LAUNCH(rname, ref_bytes, st,
                       launch_chain(k_brefine<TS>, dim3(nr), dim3(TX, TY), st, dsd, nf, dri, 0, round, R,
                                    part, next, shared ? step : -1, partb));
        }
    }
    CGK_CUDA(cudaGetLastError());
    return CG_OK;
}

// One batched schedule on stream st: reset the barrier and the failure count, the
// persistent launch (G > 0: nsteps pseudo-steps of R rounds) or the phased launches
// (G == 0), the residual history and, if `final`, the write-back (skipped on the device
// when a step missed the tolerance).
template <class TS>
static cg_status batch_issue(const BatchPlan<TS> &P, const BatchArena &A, int nsnap, int nf,
                             int nsteps, int R, int G, long long budget, double tol2, bool pred,
                             bool final, cudaStream_t st) {
    char *ab = A.ab;
    const SnapDesc<TS> *dsd = (const SnapDesc<TS> *)(ab + A.o_desc);
    const BItem *dri = (const BItem *)(ab + A.o_ri), *dci = (const BItem *)(ab + A.o_ci);
    double *prr = (double *)(ab + A.o_prr), *pbb = (double *)(ab + A.o_pbb);
    double2 *hist = (double2 *)(ab + A.o_hist);
    GridBar *gb = (GridBar *)(ab + A.o_gb);
    unsigned int *bad = (unsigned int *)(ab + A.o_bad);
    const int nr = (int)P.ritems.size(), nc = (int)P.citems.size();
    CGK_CUDA(cudaMemsetAsync(gb, 0, sizeof(GridBar), st));
    CGK_CUDA(cudaMemsetAsync(bad, 0, sizeof(unsigned int), st));
    int a_ns = nsnap, a_nf = nf, a_nr = nr, a_nc = nc, a_steps = nsteps, a_R = R, a_mm = P.mmax;
    int a_pred = pred ? 1 : 0, a_cn = P.descs[0].scheme == CG_SCHEME_CRANK_NICOLSON ? 1 : 0;
    int a_mid = batch_mid(pred, R) ? 1 : 0;
    long long a_budget = budget;
    if (pred) CGK_TRY(batch_issue_pred(P, A, nf, nsteps, st));
    void *args[] = {&dsd, &a_ns, &a_nf, &dri, &a_nr, &dci, &a_nc, &a_steps, &a_R, &a_mm, &a_pred, &a_cn, &a_mid,
                    &prr, &pbb, &gb, &a_budget};
    double bytes = 0.0;
    for (const auto &d : P.descs)
        bytes += (double)d.g.n * nf *
                 (16.0 + nsteps * ((8 + 2 * sizeof(TS)) +
                                   R * ((24 + 3 * sizeof(TS)) + (d.m - 1) * 4.0 * sizeof(TS))));
    if (G > 0) {
        CGK_LAUNCH(sizeof(TS) == 2 ? "batched_bf16" : "batched_fp32", bytes, st,
                   CGK_CUDA(cudaLaunchCooperativeKernel((const void *)k_batched<TS>, dim3(G),
                                                        dim3(TX, TY), args, 0, st)));
    } else {
        CGK_TRY(batch_issue_phased(P, A, nf, nsteps, R, pred, st));
    }
    CGK_LAUNCH("batched_hist", 16.0 * nsteps * nr, st,
               k_batched_hist<<<(unsigned)A.nh, kThreads, 0, st>>>(
                   (const int *)(ab + A.o_fi), nsnap, nf, nr, prr, pbb, hist, tol2, bad));
    CGK_CUDA(cudaGetLastError());
    if (final) {
        CGK_LAUNCH("batched_final", 16.0 * P.cells_total * nf, st,
                   k_batched_final<TS><<<dim3(num_sms() * 2, nsnap), kThreads, 0, st>>>(
                       dsd, nf, (double *const *)(ab + A.o_out), bad, batch_in_x2(pred, R, nsteps)));
        CGK_CUDA(cudaGetLastError());
    }
    return CG_OK;
}

// Autotuner of the batched schedule: the z-chunk length and, unless the caller asked
// for the persistent launch (G_only), persistent (G) against phased (one launch per
// phase); one pseudo-step of two rounds per candidate (the caller's arrays are not
// written), timed with events; the fastest is kept per batch shape (the snapshots'
// dimensions, the field count, the inner type and G_only) as a code: z for the
// persistent launch, kPhasedCode + z for the phased one.
constexpr int kPhasedCode = 500;

template <class TS>
static cg_status batch_tune(int nsnap, cg_mesh *const *meshes, int nf, double *const *cells,
                            const cg_params *p, const double *bandwidths, int G, bool G_only,
                            long long budget, cudaStream_t st, int *zbest) {
    std::vector<int> key;
    key.reserve((size_t)nsnap * 3 + 3);
    key.push_back(nf);
    key.push_back((int)sizeof(TS));
    key.push_back(G_only ? 1 : 0);
    for (int s = 0; s < nsnap; ++s) {
        key.push_back(meshes[s]->nx);
        key.push_back(meshes[s]->ny);
        key.push_back(meshes[s]->nz);
    }
    cg_mesh *m0 = meshes[0];
    for (const auto &e : m0->btuned)
        if (e.first == key) {
            *zbest = e.second;
            return CG_OK;
        }
    std::vector<int> cand = {4, 8, 16};
    if (!G_only)
        for (int z : {4, 8, 16}) cand.push_back(kPhasedCode + z);
    float best = 0.f;
    *zbest = G_only ? 8 : kPhasedCode + 8;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    CGK_CUDA(cudaEventCreate(&e0));
    CGK_CUDA(cudaEventCreate(&e1));
    cg_status rc = CG_OK;
    for (int code : cand) {
        const int z = code % kPhasedCode;
        const int g = code >= kPhasedCode ? 0 : G;
        BatchPlan<TS> P;
        rc = batch_plan<TS>(nsnap, meshes, nf, cells, p, bandwidths, z, true, 2, P);
        if (rc != CG_OK) break;
        // with the expansion a step has one inner solve: half the iterations in each of the two
        // rounds, so that sweeps and passes are weighed about as the call runs them
        if (P.pred) P.mmax = (P.mmax + 1) / 2;
        BatchArena A = batch_layout(P, nsnap, nf, 1);
        rc = m0->ws_batch.ensure(A.total);
        if (rc != CG_OK) break;
        rc = batch_upload(P, A, m0->ws_batch.as<char>(), nsnap, cells, st);
        if (rc != CG_OK) break;
        float ms = 0.f;
        for (int rep = 0; rep < 2 && rc == CG_OK; ++rep) {   // the first run warms up
            if (cudaEventRecord(e0, st) != cudaSuccess) rc = fail(CG_ECUDA, "event");
            if (rc == CG_OK) rc = batch_issue(P, A, nsnap, nf, 1, 2, g, budget, 0.0, false, false, st);
            if (rc == CG_OK && cudaEventRecord(e1, st) != cudaSuccess) rc = fail(CG_ECUDA, "event");
            if (rc == CG_OK && cudaEventSynchronize(e1) != cudaSuccess) rc = fail(CG_ECUDA, "sync");
            if (rc == CG_OK) cudaEventElapsedTime(&ms, e0, e1);
        }
        if (rc != CG_OK) break;
        GridBar hgb;
        if (cudaMemcpy(&hgb, A.ab + A.o_gb, sizeof(GridBar), cudaMemcpyDeviceToHost) != cudaSuccess) {
            rc = fail(CG_ECUDA, "readback");
            break;
        }
        if (hgb.err) {
            rc = fail(CG_ETIMEOUT, "cg_diffuse_batched: a grid barrier of the persistent kernel gave up");
            break;
        }
        if (best == 0.f || ms < best) {
            best = ms;
            *zbest = code;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc != CG_OK) return rc;
    m0->btuned.push_back({key, *zbest});
    return CG_OK;
}

template <class TS>
static cg_status diffuse_batched_df(int nsnap, cg_mesh *const *meshes, int nf,
                                    double *const *cells, const cg_params *p,
                                    const double *bandwidths, cg_report *rep, cudaStream_t st) {
    const double tol2 = p->tol * p->tol;
    cg_mesh *m0 = meshes[0];
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batched<TS>, kThreads, 0) != cudaSuccess)
        per_sm = 1;
    cudaGetLastError();
    per_sm = std::max(1, std::min(per_sm, 4));
    const int G = per_sm * num_sms();
    const long long budget = p->barrier_budget > 0 ? p->barrier_budget : 2000000000LL;
    const int max_r = p->max_rounds > 0 ? p->max_rounds : 12;
    // schedule code: z = persistent launch with z planes per work item, kPhasedCode + z =
    // one launch per phase; barrier_budget > 0 asks for the persistent launch
    const bool G_only = p->barrier_budget > 0;
    int code = p->sweep_shape > 0 ? p->sweep_shape : 0;
    if (code >= kPhasedCode && G_only)
        return fail(CG_EINVAL, "cg_diffuse_batched: barrier_budget > 0 needs the persistent schedule "
                               "(sweep_shape below %d)", kPhasedCode);
    if (code == 0)
        CGK_TRY(batch_tune<TS>(nsnap, meshes, nf, cells, p, bandwidths, G, G_only, budget, st, &code));
    const int zlen = code % kPhasedCode;
    const int Gx = code >= kPhasedCode ? 0 : G;
    if (zlen < 1) return fail(CG_EINVAL, "cg_diffuse_batched: bad sweep_shape %d", code);
    // rounds learned by an earlier call with the same signature
    std::vector<double> sig = {(double)nf, (double)p->precision, (double)p->scheme,
                               (double)p->nsteps, p->tol, p->T};
    for (int s = 0; s < nsnap; ++s) {
        sig.push_back(meshes[s]->nx);
        sig.push_back(meshes[s]->ny);
        sig.push_back(meshes[s]->nz);
        sig.push_back(meshes[s]->dx);
        sig.push_back(bandwidths ? bandwidths[s] : p->bandwidth);
    }
    int R = sizeof(TS) == 2 ? 5 : 2;
    int *learned = nullptr;
    for (auto &e : m0->brounds)
        if (e.first == sig) learned = &e.second;
    if (learned) R = std::max(R, *learned);
    // the plan's needed memory first, then the expansions' vectors, in one buffer of the first mesh
    // (an allocation per snapshot would cost a first call of 64 snapshots 25 ms); where those are
    // refused, the plan without them
    auto place = [&](BatchPlan<TS> &Q) {
        for (int s = 0; s < nsnap && Q.pred; ++s) {
            SnapDesc<TS> &d = Q.descs[s];
            d.D = (float *)(m0->ws_opt.as<char>() + Q.opt_off[s]);
            d.T = d.D + (size_t)d.g.nz * d.pts * nf * p->nsteps;
        }
    };
    BatchPlan<TS> P;
    BatchArena A;
    OptUse opt;
    const size_t nh = (size_t)p->nsteps * nsnap * nf;
    const size_t nm = (size_t)nsnap * nf;   // masses per snapshot-field, before and after
    CGK_TRY(m0->h_small.ensure(4096 + nh * sizeof(double2) + 64 + 2 * nm * 8));
    for (bool want = p->max_rounds <= 0 || p->max_rounds >= 2;; want = false) {
        CGK_TRY(batch_plan<TS>(nsnap, meshes, nf, cells, p, bandwidths, zlen, want, R, P));
        if (P.pred && m0->ws_opt.known_refused(P.opt_bytes)) continue;
        A = batch_layout(P, nsnap, nf, p->nsteps);
        const cg_status s = m0->ws_batch.ensure(A.total);
        if (!P.pred) CGK_TRY(s);
        if (!P.pred || (s == CG_OK && opt.take(m0->ws_opt, P.opt_bytes))) break;
    }
    place(P);
    CGK_TRY(batch_upload(P, A, m0->ws_batch.as<char>(), nsnap, cells, st));
    double2 *hh = (double2 *)(m0->h_small.as<char>() + 4096);
    GridBar *hgb = (GridBar *)(hh + nh);
    double *hmass = (double *)(m0->h_small.as<char>() + 4096 + nh * sizeof(double2) + 64);
    const SnapDesc<TS> *dsd = (const SnapDesc<TS> *)(A.ab + A.o_desc);
    double *dmass = (double *)(A.ab + A.o_mass);
    // report: the fields' masses before the smoothing (and after it, below), one block per
    // snapshot-field, read back with the residual history
    if (rep)
        CGK_LAUNCH("mass", 8.0 * P.cells_total * nf, st,
                   k_mass_batched<TS><<<(unsigned)nm, kThreads, 0, st>>>(dsd, nf, dmass));
    auto report_mass = [&]() {
        const int nrep = nf < CG_REPORT_MAX_FIELDS ? nf : CG_REPORT_MAX_FIELDS;
        for (int f = 0; f < nrep; ++f) {
            double a = 0.0, b = 0.0;
            for (int q = 0; q < nsnap; ++q) {
                a += hmass[(size_t)q * nf + f];
                b += hmass[nm + (size_t)q * nf + f];
            }
            rep->mass_in[f] = a;
            rep->mass_out[f] = b;
        }
    };
    const int R0 = R;
    for (; R <= max_r; ++R) {
        if (P.pred && R == 3 && R0 < 3) {   // a second inner solve per step: other counts, the same arena
            BatchPlan<TS> Q;
            CGK_TRY(batch_plan<TS>(nsnap, meshes, nf, cells, p, bandwidths, zlen, true, R, Q));
            place(Q);
            P = std::move(Q);
            A = batch_layout(P, nsnap, nf, p->nsteps);   // (no longer: fewer weights)
            CGK_TRY(batch_upload(P, A, m0->ws_batch.as<char>(), nsnap, cells, st));
        }
        // the schedule is replayed from a CUDA graph captured once per shape
        BatchKey key;
        key.arena = A.ab;
        key.gen = m0->ws_batch.gen;
        key.nsnap = nsnap;
        key.nf = nf;
        key.nsteps = p->nsteps;
        key.R = R;
        key.mmax = P.mmax;
        key.nr = (int)P.ritems.size();
        key.nc = (int)P.citems.size();
        key.grid = Gx;
        key.zlen = zlen;
        key.phased = Gx == 0 ? 1 : 0;
        key.pred = P.pred ? P.Kmax : 0;
        key.np = (int)P.pitems.size();
        key.layout = A.offsets();
        key.tsize = (int)sizeof(TS);
        key.scheme = p->scheme;
        key.budget = budget;
        key.tol2 = tol2;
        const bool prof = prof_on();
        GraphEntry *ge = nullptr;
        for (auto it = m0->graphs.begin(); it != m0->graphs.end();) {
            if (it->batched && it->bkey.arena == A.ab && it->bkey.gen != m0->ws_batch.gen) {
                graph_release(*it);
                it = m0->graphs.erase(it);
                continue;
            }
            if (it->batched && it->bkey == key && it->profiled == prof) ge = &*it;
            ++it;
        }
        if (!ge) {
            if (!m0->capture_stream)
                CGK_CUDA(cudaStreamCreateWithFlags(&m0->capture_stream, cudaStreamNonBlocking));
            cudaStream_t cs = m0->capture_stream;
            GraphEntry e;
            e.batched = true;
            e.bkey = key;
            e.profiled = prof;
            prof_capture_begin(&e.records, &e.kernels);
            cudaError_t ce = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            cg_status is = CG_OK;
            if (ce == cudaSuccess) {
                is = batch_issue(P, A, nsnap, nf, p->nsteps, R, Gx, budget, tol2, P.pred, true, cs);
                cudaGraph_t graph = nullptr;
                ce = cudaStreamEndCapture(cs, &graph);
                if (ce == cudaSuccess && is == CG_OK) ce = cudaGraphInstantiate(&e.exec, graph, 0);
                if (graph) cudaGraphDestroy(graph);
            }
            prof_capture_end();
            if (is != CG_OK || ce != cudaSuccess || !e.exec) {
                graph_release(e);
                cudaGetLastError();
                if (is != CG_OK) return is;
                return cuda_fail(ce == cudaSuccess ? cudaErrorUnknown : ce, "batched graph capture",
                                 __FILE__, __LINE__);
            }
            m0->graphs.push_back(e);
            ge = &m0->graphs.back();
        }
        CGK_CUDA(cudaGraphLaunch(ge->exec, st));
        if (rep)
            CGK_LAUNCH("mass", 8.0 * P.cells_total * nf, st,
                       k_mass_batched<TS><<<(unsigned)nm, kThreads, 0, st>>>(dsd, nf, dmass + nm));
        CGK_CUDA(cudaMemcpyAsync(hh, A.ab + A.o_hist, nh * sizeof(double2), cudaMemcpyDeviceToHost, st));
        CGK_CUDA(cudaMemcpyAsync(hgb, A.ab + A.o_gb, sizeof(GridBar), cudaMemcpyDeviceToHost, st));
        if (rep) CGK_CUDA(cudaMemcpyAsync(hmass, dmass, 2 * nm * 8, cudaMemcpyDeviceToHost, st));
        CGK_CUDA(cudaStreamSynchronize(st));
        prof_account_replay(*ge);
        if (hgb->err)
            return fail(CG_ETIMEOUT, "cg_diffuse_batched: a grid barrier of the persistent kernel gave up");
        bool ok = true;
        double worst = 0.0;
        for (size_t i = 0; i < nh; ++i) {
            ok = ok && (hh[i].x <= tol2 * hh[i].y);
            worst = std::max(worst, hh[i].y > 0 ? std::sqrt(hh[i].x / hh[i].y) : 0.0);
        }
        if (ok) {
            if (learned)
                *learned = R;
            else
                m0->brounds.push_back({sig, R});
            if (rep) {
                long long apps = 0, upd = 0;
                for (const auto &d : P.descs) {
                    // the first pass of the first step, then R rounds of m applications
                    // per step (a step's last pass also starts the next one)
                    long long a = 1 + (long long)p->nsteps * R * d.m;
                    if (P.pred)   // the expansion, then per step one pass and R - 1 rounds
                        a = (p->scheme == CG_SCHEME_CRANK_NICOLSON ? 1 : 0) + d.K +
                            (long long)p->nsteps * (1 + (long long)(R - 1) * d.m);
                    apps += a;
                    upd += a * d.g.n;
                }
                rep->iters = apps * nf;
                rep->refine_rounds = (long long)p->nsteps * R * nsnap;
                rep->cell_updates = upd * nf;
                rep->final_rel_residual = worst;
                rep->inner_iters_per_round = P.mmax;
                rep->sweep_shape_used = code;
                report_mass();
            }
            return CG_OK;
        }
        if (R == max_r) {   // the last iterate is left in place
            unsigned int *bad = (unsigned int *)(A.ab + A.o_bad);
            CGK_CUDA(cudaMemsetAsync(bad, 0, sizeof(unsigned int), st));
            CGK_LAUNCH("batched_final", 16.0 * P.cells_total * nf, st,
                       k_batched_final<TS><<<dim3(num_sms() * 2, nsnap), kThreads, 0, st>>>(
                           (const SnapDesc<TS> *)(A.ab + A.o_desc), nf,
                           (double *const *)(A.ab + A.o_out), bad, batch_in_x2(P.pred, R, p->nsteps)));
            CGK_CUDA(cudaGetLastError());
            if (rep) {
                CGK_LAUNCH("mass", 8.0 * P.cells_total * nf, st,
                           k_mass_batched<TS><<<(unsigned)nm, kThreads, 0, st>>>(dsd, nf, dmass + nm));
                CGK_CUDA(cudaMemcpyAsync(hmass, dmass, 2 * nm * 8, cudaMemcpyDeviceToHost, st));
            }
            CGK_CUDA(cudaStreamSynchronize(st));
            if (rep) {
                rep->final_rel_residual = worst;
                report_mass();
            }
            break;
        }
    }
    return fail(CG_ENOCONV, "cg_diffuse_batched: refinement did not reach tol");
}

cg_status diffuse_batched_run(int nsnap, cg_mesh *const *meshes, int nf, double *const *cells,
                              const cg_params *p, const double *bandwidths, cg_report *rep,
                              cudaStream_t st) {
    if (p->precision == CG_PREC_FP32_DF_REFINE)
        return diffuse_batched_df<float>(nsnap, meshes, nf, cells, p, bandwidths, rep, st);
    return diffuse_batched_df<__nv_bfloat16>(nsnap, meshes, nf, cells, p, bandwidths, rep, st);
}

}  // namespace cgk
