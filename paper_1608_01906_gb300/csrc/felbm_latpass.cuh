// Structured-lattice step in FP64: four launches over the nodes (streamed h
// and rho; grad rho; lap rho, mu and K; grad mu, g and the collision), each
// the per-node arithmetic of the tile step (felbm_lattice.cuh) on global
// fields.
//
// The FP64 pipe bounds it: this part issues an FP64 instruction of a warp
// every 19 cycles per SM, 75 times fewer than in FP32, so nothing is computed
// twice.  The tile step redoes the density on its halo 2.08 times, the
// gradient 1.7 and mu 1.3 times, and puts a 64 x 64 lattice on 16 of 152 SMs;
// here a node is a thread and small meshes spread over all SMs.  The extra
// passes over memory (236 B per node, mostly L2) cost less than a tenth of
// what they save: us a step 64 x 64 65.6 -> 24.3, 357 x 203 176 -> 82, 256 x
// 1024 423 -> 271.  Row kinds are decided per node: a node whose row is no wall
// row takes the integer-weight operators, so results depend neither on tiles
// nor on how a lattice is cut into slabs.
#pragma once

#include "felbm_internal.h"
#include "felbm_kernels.cuh"
#include "felbm_lattice.cuh"

namespace felbm {

// Largest number of threads per block of the passes.
constexpr int kPassBlock = 128;

// Rows of storage that a pass covers: d rows more on both sides of a slab's
// own rows than its last pass (values that only feed rows outside the slab
// are never read); all rows of a whole lattice.
FELBM_HD inline void pass_rows(int32_t ny, int32_t gny, int32_t ylo, int32_t yhi, int d, int32_t &lo, int32_t &hi) {
    const bool whole = gny == ny;
    lo = whole ? 0 : (ylo - d > 0 ? ylo - d : 0);
    hi = whole ? ny : (yhi + d < ny ? yhi + d : ny);
}

// One node and its neighbours' columns and rows.
struct LatNode {
    bool valid;
    int32_t x, xl, xr, y, yd, yu;
    int k;  // row kind
    template <typename T>
    __device__ __forceinline__ void set(const LatArgs<T> &A, int d, int64_t idx) {
        int32_t lo, hi;
        pass_rows(A.ny, A.gny, A.ylo, A.yhi, d, lo, hi);
        valid = idx < (int64_t)(hi - lo) * A.nx;
        if (!valid) return;
        const int32_t r = (int32_t)(idx / A.nx);
        x = (int32_t)(idx - (int64_t)r * A.nx);
        y = lo + r;
        xl = x == 0 ? A.nx - 1 : x - 1;
        xr = x == A.nx - 1 ? 0 : x + 1;
        const int32_t gy = y + A.row0;
        k = lat_kind(A.walls, gy, A.gny);
        // (past a walled lattice's first and last row the row itself stands in:
        // those coefficients are zero)
        yd = k == 1 ? y : (y == 0 ? A.ny - 1 : y - 1);
        yu = k == 2 ? y : (y == A.ny - 1 ? 0 : y + 1);
        if (A.walls && (gy < 0 || gy >= A.gny)) valid = false;  // a slab's rows outside the lattice
    }
    // f of the node, then of the neighbours o = (1,0), (1,1), (0,1), (-1,0),
    // (-1,-1), (0,-1), from an array with rows of `pitch`
    template <typename E>
    __device__ __forceinline__ void gather(const E *f, int32_t pitch, E &s, E *n) const {
        const E *r0 = f + (size_t)pitch * y, *ru = f + (size_t)pitch * yu, *rd = f + (size_t)pitch * yd;
        s = r0[x];
        n[0] = r0[xr];
        n[1] = ru[xr];
        n[2] = ru[x];
        n[3] = r0[xl];
        n[4] = rd[xl];
        n[5] = rd[x];
    }
};

// The four streamed, bounced-back pairs of a node (pairs: pair 0's array,
// pair q np further each).
template <typename T>
__device__ __forceinline__ void pass_stream(const LatArgs<T> &A, const LatNode &v, const V2<T> *pairs, size_t np,
                                            V2<T> *out) {
    auto one = [&](auto qc) {
        constexpr int q = decltype(qc)::value;
        V2<T> s, n[6];
        v.gather(pairs + q * np, A.pitch, s, n);
        if (A.uni && v.k == 0) {
            out[q] = stream_uni_v<T, q>(s, n[0], n[1], n[2], n[3], n[4], n[5], A.su);
        } else {
            V2<T> acc = vset(T(0), T(0));
#pragma unroll
            for (int o = 0; o < 6; ++o) acc = vfma(A.c.s[v.k][o][q], vsub<T>(n[o], s), acc);
            out[q] = bounce_pair<T>(v.k, q, vfma(vset(-A.P.dt, -A.P.dt), acc, s));
        }
    };
    one(IntC<0>{});
    one(IntC<1>{});
    one(IntC<2>{});
    one(IntC<3>{});
}

// Recovered gradient from a field's value and neighbours.
template <typename T>
__device__ __forceinline__ void pass_grad(const LatArgs<T> &A, int k, T s, const T *n, T &gx, T &gy) {
    if (A.uni && k == 0) {
        rec_uni<T>(n[0], n[1], n[2], n[3], n[4], n[5], gx, gy);
        gx *= A.al;
        gy *= A.al;
    } else {
        gx = gy = T(0);
#pragma unroll
        for (int o = 0; o < 6; ++o) grad_edge<T>(A.c.r[k][o][0], A.c.r[k][o][1], n[o] - s, gx, gy);
    }
}

// Scratch fields of a state on a lattice of n nodes: rho, grad rho (pairs),
// mu, K (pairs).
template <typename T>
struct PassFields {
    T *rho, *mu;
    V2<T> *grd, *K;
    __device__ __forceinline__ PassFields(T *s, size_t n) {
        grd = reinterpret_cast<V2<T> *>(s);
        K = grd + n;
        rho = s + 4 * n;
        mu = rho + n;
    }
};

// Pass S of node idx of the pass.  h* is kept in the h part of fout until
// the last pass replaces it.
template <typename T, int S>
__device__ __forceinline__ void lat_pass(const LatArgs<T> &A, int64_t idx) {
    LatNode v;
    v.set(A, 3 - S, idx);
    if (!v.valid) return;
    const size_t n = (size_t)A.nx * A.ny, np = pad4((size_t)A.pitch * A.ny);
    const size_t i = (size_t)A.nx * v.y + v.x, ip = (size_t)A.pitch * v.y + v.x;
    if (!chk_idx((long long)ip, (long long)A.pitch * A.ny, 1u)) return;
    const PassFields<T> F(A.rho, n);
    if constexpr (S == 0) {
        V2<T> h[4];
        pass_stream<T>(A, v, reinterpret_cast<const V2<T> *>(A.fin + np), np, h);
        const T h0 = A.fin[ip];
        V2<T> *ho = reinterpret_cast<V2<T> *>(A.fout + np);
#pragma unroll
        for (int q = 0; q < 4; ++q) ho[q * np + ip] = h[q];
        F.rho[i] = h0 + ((h[0].x + h[0].y) + (h[1].x + h[1].y)) + ((h[2].x + h[2].y) + (h[3].x + h[3].y));
    } else if constexpr (S == 1) {
        T s, nb[6], gx, gy;
        v.gather(F.rho, A.nx, s, nb);
        pass_grad<T>(A, v.k, s, nb, gx, gy);
        F.grd[i] = vset(gx, gy);
    } else if constexpr (S == 2) {
        const Phys<T> &P = A.P;
        V2<T> s, nb[6];
        v.gather(F.grd, A.nx, s, nb);
        T lap, kx = T(0), ky = T(0);
        if (A.uni && v.k == 0) {
            const V2<T> E0 = vsub<T>(nb[0], nb[3]), E1 = vsub<T>(nb[1], nb[4]), E2 = vsub<T>(nb[2], nb[5]);
            lap = A.al * (fma(T(2), E0.x, E1.x - E2.x) + fma(T(2), E2.y, E1.y - E0.y));
            stress_uni<T>(E0, E1, E2, nb, P.kappa * A.al, kx, ky);
        } else {
            lap = T(0);
#pragma unroll
            for (int o = 0; o < 6; ++o) {
                const T ax = A.c.r[v.k][o][0], ay = A.c.r[v.k][o][1];
                lap_edge<T>(ax, ay, s.x, s.y, nb[o].x, nb[o].y, lap);
                stress_edge<T>(ax, ay, s.x, s.y, nb[o].x, nb[o].y, kx, ky);
            }
            kx *= P.kappa;
            ky *= P.kappa;
        }
        F.mu[i] = mu_bulk<T>(P, F.rho[i]) - P.kappa * lap;
        F.K[i] = vset(kx, ky);
    } else {
        V2<T> g[4], h[4];
        pass_stream<T>(A, v, reinterpret_cast<const V2<T> *>(A.fin + 10 * np), np, g);
        const V2<T> *hs = reinterpret_cast<const V2<T> *>(A.fout + np);
#pragma unroll
        for (int q = 0; q < 4; ++q) h[q] = hs[q * np + ip];
        const T h0 = A.fin[ip], g0 = A.fin[9 * np + ip], r = F.rho[i];
        T s, nb[6], dmx, dmy, sg, mx, my;
        v.gather(F.mu, A.nx, s, nb);
        pass_grad<T>(A, v.k, s, nb, dmx, dmy);
        g_moments<T>(g0, g, sg, mx, my);
        const V2<T> dr = F.grd[i], K = F.K[i];
        const CollidePrep<T> c = collide_prep<T>(A.P, sg, mx, my, r, dr.x, dr.y, dmx, dmy, K.x, K.y);
        collide_store<T>(c, h, g, h0, g0, np, reinterpret_cast<V2<T> *>(A.fout + np) + ip,
                         reinterpret_cast<V2<T> *>(A.fout + 10 * np) + ip, A.fout + ip, A.fout + 9 * np + ip);
        if (!(finite_val(r) && finite_val(c.ux) && finite_val(c.uy) && finite_val(c.p))) atomicOr(A.flag, 1);
        if (A.mom) {
            A.mom[i] = r;
            A.mom[n + i] = c.ux;
            A.mom[2 * n + i] = c.uy;
            A.mom[3 * n + i] = c.p;
        }
    }
}

template <typename T, int S>
__global__ void __launch_bounds__(kPassBlock) k_lat_pass(const __grid_constant__ LatArgs<T> A) {
    pdl_wait();
    lat_pass<T, S>(A, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

}  // namespace felbm
