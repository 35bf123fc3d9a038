// Device kernels of one FE-LBM time step on tetrahedral meshes (D3Q19, the
// paper's own setting), on two topologies: general rows (DevELL3) and the
// Kuhn-split cube lattice (DevLattice3).  Four dependent passes, as in the
// two-dimensional general path (felbm_kernels.cuh):
//   rho       Taylor-Galerkin streaming of the 19 h populations (Sec.
//             2.2.1, lumped mass), wall bounce-back, rho = sum_a h_a; the
//             streamed h* is kept for the collision;
//   grad      recovered grad rho (Sec. 2.3);
//   mu        Laplacian of rho, the stress force
//             K_i = kappa [d_i |grad rho|^2 - d_j (d_i rho d_j rho)] and
//             mu = mu_phi(rho) - kappa lap rho (Sec. 2.1);
//   collide   recovered grad mu, streaming of the 19 g populations,
//             bounce-back, moments (Eqs. velocity, pressure) and the
//             post- and next pre-streaming collision (Sec. 2.2).
// Each pass has a form that splits a node over three threads (k_*3_split or
// k_*3_rows: general meshes, small lattices) and one for lattices with a
// thread per node (k_*3_node) or per column of nodes (k_*3_col).
// D3Q19 directions are ordered so that 2q+1 and 2q+2 are opposite (q =
// 0..8); the populations are stored as the rest value plus 9 interleaved
// opposite pairs (pop layout of felbm_internal.h with 19 per distribution).
#pragma once

#include <type_traits>

#include "felbm_internal.h"
#include "felbm_kernels.cuh"

namespace felbm {

// D3Q19: rest, +-x, +-y, +-z, then the 12 edge directions in opposite pairs.
__host__ __device__ constexpr int e3x(int a) {
    return (a == 1 || a == 7 || a == 9 || a == 11 || a == 13) ? 1
           : (a == 2 || a == 8 || a == 10 || a == 12 || a == 14) ? -1 : 0;
}
__host__ __device__ constexpr int e3y(int a) {
    return (a == 3 || a == 7 || a == 10 || a == 15 || a == 17) ? 1
           : (a == 4 || a == 8 || a == 9 || a == 16 || a == 18) ? -1 : 0;
}
__host__ __device__ constexpr int e3z(int a) {
    return (a == 5 || a == 11 || a == 14 || a == 15 || a == 18) ? 1
           : (a == 6 || a == 12 || a == 13 || a == 16 || a == 17) ? -1 : 0;
}
template <typename T>
__host__ __device__ constexpr T w3(int a) {
    return a == 0 ? T(1) / T(3) : (a <= 6 ? T(1) / T(18) : T(1) / T(36));
}

// 3 w_a of D3Q19 in the working precision with the moment identities exact
// in T (see kW3): sum_a 3 w_a = 3 (w3_0 + 6 w3_1 + 12 w3_7) and
// sum_a 3 w_a e_ax^2 = 1 (2 w3_1 + 8 w3_7), from e ~ 1/12 (kTwelfth):
// w3_7 = e, w3_1 = (1 - 8 e)/2, w3_0 = 12 e.
template <typename T>
__host__ __device__ constexpr T w3x3(int a) {
    return a == 0 ? T(12) * kTwelfth<T>() : (a <= 6 ? (T(1) - T(8) * kTwelfth<T>()) / T(2) : kTwelfth<T>());
}

// Model constants of one state (Sec. 2.1) with three-component gravity.
template <typename T>
struct Phys3 {
    T rho_l, rho_v, beta, kappa, inv_tau_l, inv_tau_v, dt, g[3];
    T inv_drho;  // 1 / (rho_l - rho_v)
};

template <typename T>
__device__ __forceinline__ T mu_bulk3(const Phys3<T> &P, T r) {
    return T(4) * P.beta * (r - P.rho_v) * (r - P.rho_l) * (r - T(0.5) * (P.rho_v + P.rho_l));
}

// Both topologies give, for node i, the neighbours j with their
// coefficients: for_each<K>(i, fn(j, a)) with a = (a_x, a_y, a_z) at least,
// for_each_pair<K>(i, dt/2, fn(j, c)) with c[q] = (e.a + dt/2 e.b.e) for the
// pair q = (2q+1, 2q+2) as (first, second) = (even + odd, even - odd) parts.
// K >= 0 promises that node i is of z-layer kind K (lattice only; -1 = any).
//
constexpr int kSplitGroups = 3;  // threads of a node in the split passes

// General tetrahedral mesh, reverse Cuthill-McKee order: rows in slices of
// 32 nodes (see DevELL), per entry {a_x, a_y, a_z, neighbour}, {b_xx, b_xy,
// b_xz, b_yy} and {b_yz, b_zz}.
template <typename T>
struct DevELL3 {
    static constexpr bool kLattice = false;
    int32_t n;
    const int32_t *sbase;
    const Ell4<T> *a, *b;
    const Ell2<T> *c;
    const uint8_t *tag;  // nullptr if no walls
#ifdef __CUDACC__
    template <int K, typename Fn>
    __device__ __forceinline__ void for_each(int32_t i, Fn &&fn) const {
        const int32_t r0 = __ldg(sbase + (i >> 5)), r1 = __ldg(sbase + (i >> 5) + 1);
        const size_t p = (size_t)r0 * 32 + (i & 31);
        const Ell4<T> *pa = a + p, *pb = b + p;
        const Ell2<T> *pc = c + p;
#pragma unroll 4
        for (int32_t k = 0; k < r1 - r0; ++k) {
            const Ell4<T> v = ell_load(pa + 32 * k), w = ell_load(pb + 32 * k);
            const Ell2<T> z = ell_load(pc + 32 * k);
            const int32_t j = ell_get(v.w);
            if (!chk_idx(j, n, 1u)) continue;
            const T cf[9] = {v.x, v.y, v.z, w.x, w.y, w.z, w.w, z.x, z.y};
            fn(j, cf);
        }
    }
    template <int K, typename Fn>
    __device__ __forceinline__ void for_each_pair(int32_t i, T hdt, Fn &&fn) const {
        for_each<K>(i, [&](int32_t j, const T *cf) {
            V2<T> c[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const int a = 2 * q + 1;
                const T ex = T(e3x(a)), ey = T(e3y(a)), ez = T(e3z(a));
                const T odd = ex * cf[0] + ey * cf[1] + ez * cf[2];
                const T even = hdt * ((ex * ex * cf[3] + ey * ey * cf[6] + ez * ez * cf[8]) +
                                      T(2) * (ex * ey * cf[4] + ex * ez * cf[5] + ey * ez * cf[7]));
                c[q] = vset(even + odd, even - odd);
            }
            fn(j, c);
        });
    }
    // Entries g, g + kSplitGroups, ... of the row of node i: the first kPart of them are
    // read by part_row (no kernel writes them), with the recovery
    // coefficients only.  4 in FP32, 2 in FP64 (jittered tetrahedra 12^3, 28^3,
    // 40^3, 56^3 FP32 16.1, 19.4, 38.4, 122 us a step, with 6 15.8, 19.0, 37.8,
    // 121, with 2 17.0, 20.3, 36.8, 120; FP64 40^3 581, with 4 601, with 1 570).
    static constexpr int kPart = sizeof(T) == 4 ? 4 : 2, kGroups = kSplitGroups;
    struct PartRow {
        size_t p;
        int32_t rows, g;
        Ell4<T> v[kPart];
    };
    __device__ __forceinline__ PartRow part_row(int32_t i, int g) const {
        PartRow r;
        const int32_t r0 = __ldg(sbase + (i >> 5));
        r.rows = __ldg(sbase + (i >> 5) + 1) - r0;
        r.p = (size_t)r0 * 32 + (i & 31);
        r.g = g;
        part_load(r, g, r.v, i);
        return r;
    }
    __device__ __forceinline__ void part_load(const PartRow &r, int32_t k0, Ell4<T> *v, int32_t i) const {
#pragma unroll
        for (int k = 0; k < kPart; ++k) {
            v[k] = {T(0), T(0), T(0), ell_id<T>(i)};
            if (k0 + kGroups * k < r.rows) v[k] = ell_load(a + r.p + 32 * (size_t)(k0 + kGroups * k));
        }
    }
    template <typename Fn>
    __device__ __forceinline__ void each_part(const PartRow &r, int32_t i, Fn &&fn) const {
        part_run(r.v, fn);
        for (int32_t k = r.g + kGroups * kPart; k < r.rows; k += kGroups * kPart) {
            Ell4<T> v[kPart];
            part_load(r, k, v, i);
            part_run(v, fn);
        }
    }
    template <typename Fn>
    __device__ __forceinline__ void part_run(const Ell4<T> *v, Fn &&fn) const {
#pragma unroll
        for (int k = 0; k < kPart; ++k) {
            const int32_t j = ell_get(v[k].w);
            const T cf[3] = {v[k].x, v[k].y, v[k].z};
            if (chk_idx(j, n, 1u)) fn(j, cf);
        }
    }
    __device__ __forceinline__ int kind_of(int32_t) const { return -1; }
    __device__ __forceinline__ int tag_of(int32_t i) const { return tag ? (int)tag[i] : 0; }
#endif
};

// Coefficients of the Kuhn lattice per z-layer kind (0 interior, 1 bottom
// wall layer, 2 top wall layer) and neighbour offset o (lat3_d*(o)), passed
// as kernel parameters: the pair form of the streaming coefficients with
// dt/2 folded in, and the recovery coefficients a_ij.
template <typename T>
struct Lat3Coef {
    V2<T> pc[3][14][9];
    T a[3][14][3];
    T s12;  // 1 / (12 h): a = kuhn_w s12 in the interior of a uniform lattice
};

// Kuhn-split cube lattice in natural order (i = x + nx (y + ny z)): the 14
// neighbour ids follow from the node's position; a walled z direction has
// tags 5 (bottom layer, inward normal +z) and 6 (top layer).
template <typename T>
struct DevLattice3 {
    static constexpr bool kLattice = true;
    int32_t n, nx, ny, nz;
    int32_t walls;
    int32_t tables;  // layers whose recovery weights are not the integers kuhn_w times k.s12: 0 none, 1 the wall
                     // layers, 2 all (see kuhn_uniform)
    Lat3Coef<T> k;
#ifdef __CUDACC__
    __device__ __forceinline__ int kind_of(int32_t i) const {
        if (!walls) return 0;
        const int32_t z = i / (nx * ny);
        return z == 0 ? 1 : (z == nz - 1 ? 2 : 0);
    }
    __device__ __forceinline__ int tag_of(int32_t i) const {
        const int kd = kind_of(i);
        return kd == 0 ? 0 : 4 + kd;
    }
    // Where an offset leaves a walled domain its coefficients are zero and
    // the id is an in-range stand-in (the wrapped x-y neighbour in-layer).
    __device__ __forceinline__ void nbrs(int32_t i, int32_t *j) const {
        const int32_t L = nx * ny;
        const int32_t z = i / L, r = i - z * L, y = r / nx, x = r - y * nx;
        const int32_t xp = x == nx - 1 ? 1 - nx : 1, xm = x == 0 ? nx - 1 : -1;
        const int32_t yp = (y == ny - 1 ? 1 - ny : 1) * nx, ym = (y == 0 ? ny - 1 : -1) * nx;
        int32_t zp, zm;
        if (walls) {
            zp = z == nz - 1 ? 0 : L;
            zm = z == 0 ? 0 : -L;
        } else {
            zp = (z == nz - 1 ? 1 - nz : 1) * L;
            zm = (z == 0 ? nz - 1 : -1) * L;
        }
#pragma unroll
        for (int o = 0; o < 14; ++o)
            j[o] = i + (lat3_dx(o) > 0 ? xp : (lat3_dx(o) < 0 ? xm : 0)) +
                   (lat3_dy(o) > 0 ? yp : (lat3_dy(o) < 0 ? ym : 0)) +
                   (lat3_dz(o) > 0 ? zp : (lat3_dz(o) < 0 ? zm : 0));
    }
    template <int K, typename Fn>
    __device__ __forceinline__ void for_each(int32_t i, Fn &&fn) const {
        int32_t j[14];
        nbrs(i, j);
        const int kd = K >= 0 ? K : kind_of(i);
#pragma unroll
        for (int o = 0; o < 14; ++o)
            if (chk_idx(j[o], n, 1u)) fn(j[o], k.a[kd][o]);
    }
    template <int K, typename Fn>
    __device__ __forceinline__ void for_each_pair(int32_t i, T, Fn &&fn) const {
        int32_t j[14];
        nbrs(i, j);
        const int kd = K >= 0 ? K : kind_of(i);
#pragma unroll
        for (int o = 0; o < 14; ++o)
            if (chk_idx(j[o], n, 1u)) fn(j[o], k.pc[kd][o]);
    }
#endif
};

#ifdef __CUDACC__
// Runs fn(integral_constant<K>) with K = 0 for interior lattice nodes (the
// coefficients are then compile-time parameter offsets) and K = -1 otherwise.
template <typename Topo, typename Fn>
__device__ __forceinline__ void by_kind(const Topo &m, int32_t i, Fn &&fn) {
    if constexpr (Topo::kLattice) {
        if (m.kind_of(i) == 0) {
            fn(std::integral_constant<int, 0>());
            return;
        }
    }
    fn(std::integral_constant<int, -1>());
}
#endif

// Fields of one time level: rho, mu, K (N each); grad rho interleaved as
// (x, y, z, unused) per node (4 N, 16-byte aligned), so that one gather
// reads a neighbour's gradient; and the streamed, bounced-back h* of k_rho3
// (19 values per node, population layout: rest at [0, Np), pair q at
// Np + 2 Np q).
template <typename T>
struct Fields3 {
    T *rho, *dr4, *mu, *k[3];
    T *hs;
};

#ifdef __CUDACC__
template <typename T>
__device__ __forceinline__ void load_grad3(const T *dr4, int32_t j, T *g) {
    if constexpr (sizeof(T) == 4) {
        const float4 v = ldp(reinterpret_cast<const float4 *>(dr4) + j);
        g[0] = v.x;
        g[1] = v.y;
        g[2] = v.z;
    } else {
        const double2 *p = reinterpret_cast<const double2 *>(dr4) + 2 * (size_t)j;
        const double2 a = ldp(p), b = ldp(p + 1);
        g[0] = a.x;
        g[1] = a.y;
        g[2] = b.x;
    }
}

template <typename T>
__device__ __forceinline__ void store_grad3(T *dr4, int32_t i, const T *g) {
    if constexpr (sizeof(T) == 4) {
        reinterpret_cast<float4 *>(dr4)[i] = make_float4(g[0], g[1], g[2], 0.0f);
    } else {
        double2 *p = reinterpret_cast<double2 *>(dr4) + 2 * (size_t)i;
        p[0] = make_double2(g[0], g[1]);
        p[1] = make_double2(g[2], 0.0);
    }
}
#endif

// Streamed values of pairs Q0 .. Q0+NQ-1 of one distribution of node i
// (base: its rest values; pair q at base + Np + 2 Np q):
// psi* = psi - dt sum_j (e.a_ij + dt/2 e.b_ij.e) (psi_j - psi_i).
template <typename T, int Q0, int NQ, int K, typename Topo>
__device__ __forceinline__ void stream_range3(const Topo &m, const T *base, size_t np, int32_t i,
                                              T dt, V2<T> *out) {
    const V2<T> *pb = reinterpret_cast<const V2<T> *>(base + np);
    const V2<T> m1 = vset(T(-1), T(-1));
    V2<T> own[NQ], acc[NQ];
#pragma unroll
    for (int r = 0; r < NQ; ++r) {
        own[r] = ldp(pb + (Q0 + r) * np + i);
        acc[r] = vset(T(0), T(0));
    }
    m.template for_each_pair<K>(i, T(0.5) * dt, [&](int32_t j, const V2<T> *c) {
#pragma unroll
        for (int r = 0; r < NQ; ++r)
            acc[r] = vfma(c[Q0 + r], vfma(own[r], m1, ldp(pb + (Q0 + r) * np + j)), acc[r]);
    });
    const V2<T> mdt = vset(-dt, -dt);
#pragma unroll
    for (int r = 0; r < NQ; ++r) out[r] = vfma(mdt, acc[r], own[r]);
}

// The 9 streamed pairs in two passes over the neighbours (5 + 4 pairs):
// fewer live registers per thread, more threads per SM.
template <typename T, int K, typename Topo>
__device__ __forceinline__ void stream_all3(const Topo &m, const T *base, size_t np, int32_t i, T dt, V2<T> *out) {
    stream_range3<T, 0, 5, K>(m, base, np, i, dt, out);
    stream_range3<T, 5, 4, K>(m, base, np, i, dt, out + 5);
}

// Bounce-back of pair q = (a, a+1), a = 2q+1, at a wall node with inward
// normal e_k: the member with e . e_k > 0 takes the value of the other.
template <typename T>
__device__ __forceinline__ void bounce_pair3(int k, int q, V2<T> &p) {
    const int a = 2 * q + 1;
    const int d = e3x(a) * e3x(k) + e3y(a) * e3y(k) + e3z(a) * e3z(k);
    if (d > 0)
        p.x = p.y;
    else if (d < 0)
        p.y = p.x;
}

// ---- a thread per node: large lattices ---------------------------------------
// Bound by the latency of the gathers at 32 (h) and 20 (g) warps an SM and, from
// 10^6 nodes on, by HBM with the h* round trip (128^3 FP32: 111 and 169 us for
// 327 and 713 MB).  All pairs of a neighbour at once is the order that hides
// most: pair by pair over columns of 1, 2 or 4 nodes, which loads 11 or 9
// values a node and pair instead of 15, took 142, 132 and 183 us for h.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 1)
    k_rho3_node(const __grid_constant__ DevLattice3<T> m, const T *f, T dt, T *rho, T *hs) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const size_t np = pad4((size_t)m.n);
    pdl_wait();
    f = pdl_ptr(f);
    V2<T> h[9];
    by_kind(m, i, [&](auto K) { stream_all3<T, decltype(K)::value>(m, f, np, i, dt, h); });
    const T h0 = ldp(f + i);
    const int k = m.tag_of(i);
    T r = h0;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        if (k) bounce_pair3<T>(k, q, h[q]);
        r += h[q].x;
        r += h[q].y;
    }
    rho[i] = r;
    V2<T> *hb = reinterpret_cast<V2<T> *>(hs + np);
#pragma unroll
    for (int q = 0; q < 9; ++q) hb[q * np + i] = h[q];
    hs[i] = h0;
}

// ---- a node split over three threads -----------------------------------------
// A block has 64 nodes; the warps 2 g and 2 g + 1 of it take the pairs 3 g ..
// 3 g + 2.  The groups of a node read its row one after the other, from L1.
// What bounds the passes below some 10^5 nodes is the latency of the gathers
// (14 neighbours x 9 pairs, two accesses deep on general rows); a thread per
// node has 13 warps per SM on a 40^3 mesh, three have 40 and each waits for a
// third of the gathers.  Jittered tetrahedra, FP32, us a step: 40^3 52 -> 37.8,
// 16^3 15.3; four threads (3, 2, 2, 2 pairs) 39.2 and 15.4, with more loads of
// the rows.
constexpr int kSplitNodes = 64;
constexpr int kSplitBlock = kSplitNodes * kSplitGroups;
constexpr int split_first(int g) { return 3 * g; }
constexpr int split_count(int) { return 3; }

// Runs fn(integral_constant<g>) with the group of the thread (warp-uniform).
template <typename Fn>
__device__ __forceinline__ void by_group(int g, Fn &&fn) {
    if (g == 0)
        fn(std::integral_constant<int, 0>());
    else if (g == 1)
        fn(std::integral_constant<int, 1>());
    else
        fn(std::integral_constant<int, 2>());
}

// The sum of the groups' values of a node.
template <typename T>
__device__ __forceinline__ T group_sum(const T (&v)[kSplitGroups][kSplitNodes], int l) {
    T s = v[0][l];
#pragma unroll
    for (int g = 1; g < kSplitGroups; ++g) s += v[g][l];
    return s;
}

template <typename T, typename Topo>
__global__ void __launch_bounds__(kSplitBlock, sizeof(T) == 4 ? 4 : 2)
    k_rho3_split(const __grid_constant__ Topo m, const T *f, T dt, T *rho, T *hs) {
    __shared__ T part[kSplitGroups][kSplitNodes];
    const int l = threadIdx.x % kSplitNodes, grp = threadIdx.x / kSplitNodes;
    const int32_t i = blockIdx.x * kSplitNodes + l;
    const bool in = i < m.n;
    const size_t np = pad4((size_t)m.n);
    const int k = in ? m.tag_of(i) : 0;
    pdl_wait();
    f = pdl_ptr(f);
    T h0 = T(0);
    if (in) {
        by_group(grp, [&](auto G) {
            constexpr int Q0 = split_first(decltype(G)::value), NQ = split_count(decltype(G)::value);
            V2<T> h[NQ];
            by_kind(m, i, [&](auto K) { stream_range3<T, Q0, NQ, decltype(K)::value>(m, f, np, i, dt, h); });
            V2<T> *hb = reinterpret_cast<V2<T> *>(hs + np);
            T r = T(0);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                if (k) bounce_pair3<T>(k, Q0 + q, h[q]);
                r += h[q].x;
                r += h[q].y;
                hb[(Q0 + q) * np + i] = h[q];
            }
            part[grp][l] = r;
        });
        if (grp == 0) {
            h0 = ldp(f + i);
            hs[i] = h0;
        }
    }
    __syncthreads();
    if (grp == 0 && in) rho[i] = h0 + group_sum(part, l);
}

// ---- columns of the lattice --------------------------------------------------
// A thread has LZ nodes one above the other.  The 14 neighbours of a node lie
// at 7 places of its plane, 4 above and 4 below, and a column shares them: 11
// loads a node for LZ = 2 against 15.  The scalar passes (grad rho; mu and K)
// with the integer weights, us on 128^3 FP32: 21.0 and 47.0 with the tables,
// 19 and 36 with LZ = 1, 14.2 and 30.8 with LZ = 2; LZ = 4 no faster (14.4, 32).
// A block takes columns of one layer of columns, whose plane offsets are then
// the block's; PACK: columns in order, so that small planes share a block (3 x
// 3 x 40000 FP32 122 us a step without, 67 with; 64^3 43.2 and 43.6, 12^3 FP64
// 53 and 58, 3 x 3 x 1000 12.3 and 11.0).
template <int LZ, bool PACK>
struct Col3 {
    int32_t r[7];        // in the plane: own, +x, -x, +y, -y, +x+y, -x-y
    int32_t pl[LZ + 2];  // first nodes of the planes z0 - 1 .. z0 + LZ (wrapped)
    int32_t z0, n;
    int count;           // nodes of the column in the lattice
    bool table;          // its nodes take the tables: some are of a layer of m.tables
    // false: no column of the lattice
    template <typename T>
    __device__ __forceinline__ bool set(const DevLattice3<T> &m) {
        const int32_t L = m.nx * m.ny;
        int32_t zb, p;
        if (PACK) {
            const uint32_t k = blockIdx.x * blockDim.x + threadIdx.x;  // below 2^31 + 256
            zb = k / L;
            p = k - (uint32_t)zb * L;
            if (zb >= (m.nz + LZ - 1) / LZ) return false;
        } else {
            const int32_t planes = (L + blockDim.x - 1) / blockDim.x;  // blocks of LZ planes
            zb = blockIdx.x / planes;
            p = (blockIdx.x - zb * planes) * blockDim.x + threadIdx.x;
            if (p >= L) return false;
        }
        const int32_t y = p / m.nx, x = p - y * m.nx;
        const int32_t xp = x == m.nx - 1 ? 1 - m.nx : 1, xm = x == 0 ? m.nx - 1 : -1;
        const int32_t yp = (y == m.ny - 1 ? 1 - m.ny : 1) * m.nx, ym = (y == 0 ? m.ny - 1 : -1) * m.nx;
        n = m.n;
        r[0] = p;
        r[1] = p + xp;
        r[2] = p + xm;
        r[3] = p + yp;
        r[4] = p + ym;
        r[5] = p + xp + yp;
        r[6] = p + xm + ym;
        z0 = zb * LZ;
        int32_t z = z0 == 0 ? m.nz - 1 : z0 - 1;
#pragma unroll
        for (int k = 0; k < LZ + 2; ++k) {
            pl[k] = z * L;
            z = z + 1 == m.nz ? 0 : z + 1;
        }
        count = m.nz - z0 < LZ ? m.nz - z0 : LZ;
        table = m.tables && (m.tables == 2 || z0 == 0 || z0 + LZ >= m.nz);
        return true;
    }
    // node l of the column
    __device__ __forceinline__ int32_t id(int l) const { return pl[l + 1] + r[0]; }
    // v[k][s]: what ld gives for place s of plane k, where a node of the
    // column has a neighbour there
    template <typename V, typename Ld>
    __device__ __forceinline__ void load(V (&v)[LZ + 2][7], Ld &&ld) const {
#pragma unroll
        for (int k = 0; k < LZ + 2; ++k)
#pragma unroll
            for (int s = 0; s < 7; ++s) {
                const bool plus = s == 0 || s == 1 || s == 3 || s == 5, minus = s == 0 || s == 2 || s == 4 || s == 6;
                if ((k >= 1 && k <= LZ) || (k == 0 && minus) || (k == LZ + 1 && plus)) {
                    const int32_t j = pl[k] + r[s];
                    if (chk_idx(j, n, 1u)) v[k][s] = ld(j);
                }
            }
    }
};
// place in its plane of neighbour offset o
__host__ __device__ constexpr int col3_place(int o) {
    return o < 4 ? o + 1 : (o < 6 ? 0 : (o < 8 ? o - 1 : o - 7));
}


// Recovered gradient of a scalar field (3 components).
template <typename T, int K, typename Topo>
__device__ __forceinline__ void recover3(const Topo &m, const T *f, int32_t i, T *g) {
    const T fi = ldp(f + i);
    T s0 = T(0), s1 = T(0), s2 = T(0);
    m.template for_each<K>(i, [&](int32_t j, const T *cf) {
        const T d = ldp(f + j) - fi;
        s0 += cf[0] * d;
        s1 += cf[1] * d;
        s2 += cf[2] * d;
    });
    g[0] = s0;
    g[1] = s1;
    g[2] = s2;
}

// lap rho = sum_c R_c(d_c rho);
// K_i = kappa [sum_{k != i} R_i((d_k rho)^2) - sum_{j != i} R_j(d_i rho d_j rho)]
// (the printed form with the identical (d_i rho)^2 contributions cancelled);
// differences of the products in product form.
template <typename T>
__device__ __forceinline__ void mu_edge3(const T *cf, const T *gi, const T *gj, T &lap, T *K3) {
    T d[3], sq[3];  // sq: differences of (d_c rho)^2
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d[c] = gj[c] - gi[c];
        lap += cf[c] * d[c];
        sq[c] = d[c] * (gj[c] + gi[c]);
    }
    // differences of d_a rho d_b rho (a < b), each formed once
    const T pxy = gj[0] * d[1] + gi[1] * d[0];
    const T pxz = gj[0] * d[2] + gi[2] * d[0];
    const T pyz = gj[1] * d[2] + gi[2] * d[1];
    K3[0] += cf[0] * (sq[1] + sq[2]) - (cf[1] * pxy + cf[2] * pxz);
    K3[1] += cf[1] * (sq[0] + sq[2]) - (cf[0] * pxy + cf[2] * pyz);
    K3[2] += cf[2] * (sq[0] + sq[1]) - (cf[0] * pxz + cf[1] * pyz);
}

// ---- grad rho, mu and K -------------------------------------------------------
// General rows, three threads a node: thread group g of a block (as in the
// split passes) takes the entries g, g + 3, ... of the rows of its nodes, all
// of them in flight at once, and the sums meet in shared memory.
template <typename T, int NV>
__device__ __forceinline__ void split_sum(T (&part)[NV][kSplitGroups][kSplitNodes], int grp, int l, T *v) {
#pragma unroll
    for (int c = 0; c < NV; ++c) part[c][grp][l] = v[c];
    __syncthreads();
    if (grp) return;
#pragma unroll
    for (int c = 0; c < NV; ++c) v[c] = group_sum(part[c], l);
}

template <typename T>
__global__ void __launch_bounds__(kSplitBlock) k_grad3_rows(const __grid_constant__ DevELL3<T> m, Fields3<T> F) {
    __shared__ T part[3][kSplitGroups][kSplitNodes];
    const int l = threadIdx.x % kSplitNodes, grp = threadIdx.x / kSplitNodes;
    const int32_t i = blockIdx.x * kSplitNodes + l;
    const bool in = i < m.n;
    const auto row = m.part_row(in ? i : 0, grp);
    pdl_wait();
    T g[3] = {T(0), T(0), T(0)};
    if (in) {
        const T *rho = pdl_ptr(F.rho);
        const T fi = ldp(rho + i);
        m.each_part(row, i, [&](int32_t j, const T *cf) {
            const T d = ldp(rho + j) - fi;
            g[0] += cf[0] * d;
            g[1] += cf[1] * d;
            g[2] += cf[2] * d;
        });
    }
    split_sum<T, 3>(part, grp, l, g);
    if (in && grp == 0) store_grad3<T>(F.dr4, i, g);
}

template <typename T>
__global__ void __launch_bounds__(kSplitBlock) k_mu3_rows(const __grid_constant__ DevELL3<T> m, Fields3<T> F,
                                                          Phys3<T> P) {
    __shared__ T part[4][kSplitGroups][kSplitNodes];
    const int l = threadIdx.x % kSplitNodes, grp = threadIdx.x / kSplitNodes;
    const int32_t i = blockIdx.x * kSplitNodes + l;
    const bool in = i < m.n;
    const auto row = m.part_row(in ? i : 0, grp);
    pdl_wait();
    T s[4] = {T(0), T(0), T(0), T(0)};  // K, lap rho
    if (in) {
        const T *dr4 = pdl_ptr(F.dr4);
        T gi[3];
        load_grad3<T>(dr4, i, gi);
        m.each_part(row, i, [&](int32_t j, const T *cf) {
            T gj[3];
            load_grad3<T>(dr4, j, gj);
            mu_edge3<T>(cf, gi, gj, s[3], s);
        });
    }
    split_sum<T, 4>(part, grp, l, s);
    if (in && grp == 0) {
        F.mu[i] = mu_bulk3<T>(P, F.rho[i]) - P.kappa * s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) F.k[c][i] = P.kappa * s[c];
    }
}

// Interior nodes of a uniform lattice: 12 h a_ij are small integers, opposite at opposite
// offsets, so that R f = (1/(12 h)) sum over the seven offset pairs p of
// kuhn_w(p) (f_{+o} - f_{-o}), o = lat3_d*(2p).  Half the differences and
// products of the table form, and weights without rounding.  The host checks
// the assembled weights against them (kuhn_uniform): elements that leave gaps
// or cover the box unevenly, but alike around every node, are a lattice of
// the same offsets with other weights, and take the tables.
__host__ __device__ constexpr int kuhn_w(int p, int c) {
    return p < 3 ? (p == c ? 3 : -1) : (p < 6 ? (c == 5 - p ? -1 : 1) : 1);
}

// 12 h R f from the differences D of the seven offset pairs (the sum with
// the weights' common part taken out: 19 operations, not 21 and 7).
template <typename T>
__device__ __forceinline__ void kuhn_recover(const T *D, T *g) {
    const T S = ((D[3] + D[4]) + (D[5] + D[6])) - ((D[0] + D[1]) + D[2]);
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] = fma(T(4), D[c], fma(T(-2), D[5 - c], S));
}

// Recovered gradient of a scalar at an interior node.
template <typename T>
__device__ __forceinline__ void kuhn_recover_node(const DevLattice3<T> &m, const T *f, int32_t i, T *g) {
    int32_t j[14];
    m.nbrs(i, j);
    T D[7];
#pragma unroll
    for (int p = 0; p < 7; ++p) D[p] = chk_idx(j[2 * p], m.n, 1u) && chk_idx(j[2 * p + 1], m.n, 1u)
                                           ? ldp(f + j[2 * p]) - ldp(f + j[2 * p + 1]) : T(0);
    kuhn_recover<T>(D, g);
#pragma unroll
    for (int c = 0; c < 3; ++c) g[c] *= m.k.s12;
}

// Recovered gradients of a scalar at the nodes of an interior column.
template <typename T, int LZ, bool PACK>
__device__ __forceinline__ void recover_col3(const DevLattice3<T> &m, const Col3<LZ, PACK> &c, const T *f, T (&g)[LZ][3]) {
    T v[LZ + 2][7];
    c.load(v, [&](int32_t j) { return ldp(f + j); });
#pragma unroll
    for (int l = 0; l < LZ; ++l) {
        T D[7];
#pragma unroll
        for (int p = 0; p < 7; ++p)
            D[p] = v[l + 1 + lat3_dz(2 * p)][col3_place(2 * p)] - v[l + 1 - lat3_dz(2 * p)][col3_place(2 * p + 1)];
        kuhn_recover<T>(D, g[l]);
#pragma unroll
        for (int k = 0; k < 3; ++k) g[l][k] *= m.k.s12;
    }
}

template <typename T, int LZ, bool PACK>
__global__ void __launch_bounds__(256) k_grad3_col(const __grid_constant__ DevLattice3<T> m, Fields3<T> F) {
    Col3<LZ, PACK> c;
    if (!c.set(m)) return;
    pdl_wait();
    const T *rho = pdl_ptr(F.rho);
    if (c.table) {
        for (int l = 0; l < c.count; ++l) {
            const int32_t i = c.r[0] + (c.z0 + l) * m.nx * m.ny;
            T g[3];
            recover3<T, -1>(m, rho, i, g);
            store_grad3<T>(F.dr4, i, g);
        }
        return;
    }
    T g[LZ][3];
    recover_col3<T>(m, c, rho, g);
#pragma unroll
    for (int l = 0; l < LZ; ++l)
        if (l < c.count) store_grad3<T>(F.dr4, c.id(l), g[l]);
}

template <typename T>
struct Vec3 {
    T v[3];
};

template <typename T, int LZ, bool PACK>
__global__ void __launch_bounds__(256) k_mu3_col(const __grid_constant__ DevLattice3<T> m, Fields3<T> F, Phys3<T> P) {
    Col3<LZ, PACK> c;
    if (!c.set(m)) return;
    pdl_wait();
    const T *dr4 = pdl_ptr(F.dr4), *rho = pdl_ptr(F.rho);
    if (c.table) {
        for (int l = 0; l < c.count; ++l) {
            const int32_t i = c.r[0] + (c.z0 + l) * m.nx * m.ny;
            T gi[3], lap = T(0), K[3] = {T(0), T(0), T(0)};
            load_grad3<T>(dr4, i, gi);
            m.template for_each<-1>(i, [&](int32_t j, const T *cf) {
                T gj[3];
                load_grad3<T>(dr4, j, gj);
                mu_edge3<T>(cf, gi, gj, lap, K);
            });
            F.mu[i] = mu_bulk3<T>(P, ldp(rho + i)) - P.kappa * lap;
#pragma unroll
            for (int k = 0; k < 3; ++k) F.k[k][i] = P.kappa * K[k];
        }
        return;
    }
    Vec3<T> v[LZ + 2][7];
    c.load(v, [&](int32_t j) {
        Vec3<T> g;
        load_grad3<T>(dr4, j, g.v);
        return g;
    });
    const T f = P.kappa * m.k.s12;
#pragma unroll
    for (int l = 0; l < LZ; ++l) {
        T lap = T(0), K[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int p = 0; p < 7; ++p) {
            const T *gp = v[l + 1 + lat3_dz(2 * p)][col3_place(2 * p)].v;
            const T *gm = v[l + 1 - lat3_dz(2 * p)][col3_place(2 * p + 1)].v;
            T d[3], s[3], sq[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                d[k] = gp[k] - gm[k];
                s[k] = gp[k] + gm[k];
                sq[k] = d[k] * s[k];  // difference of (d_k rho)^2
                lap = fma(T(kuhn_w(p, k)), d[k], lap);
            }
            // twice the differences of d_a rho d_b rho
            const T pxy = fma(d[0], s[1], s[0] * d[1]);
            const T pxz = fma(d[0], s[2], s[0] * d[2]);
            const T pyz = fma(d[1], s[2], s[1] * d[2]);
            const T wx = T(kuhn_w(p, 0)), wy = T(kuhn_w(p, 1)), wz = T(kuhn_w(p, 2)), mh = T(-0.5);
            K[0] = fma(mh * wz, pxz, fma(mh * wy, pxy, fma(wx, sq[1] + sq[2], K[0])));
            K[1] = fma(mh * wz, pyz, fma(mh * wx, pxy, fma(wy, sq[0] + sq[2], K[1])));
            K[2] = fma(mh * wy, pyz, fma(mh * wx, pxz, fma(wz, sq[0] + sq[1], K[2])));
        }
        if (l < c.count) {
            const int32_t i = c.id(l);
            F.mu[i] = mu_bulk3<T>(P, ldp(rho + i)) - f * lap;
#pragma unroll
            for (int k = 0; k < 3; ++k) F.k[k][i] = f * K[k];
        }
    }
}

// Per-node scalars of the collision (3-D form of CollidePrep).
template <typename T>
struct Prep3 {
    T r, u[3], p;
    T nr, np, nomw, nhuu;
    T X[3], hA, hZ, V[3], gA, B[3], gZ, G[3], du[3];
};
template <>
struct Prep3<float> {
    float r, u[3], p, omw, opw, hdt, X[3], dr[3], K[3], du[3], uX, uD, uK, uu, udu;
};

// The scalars for given moments and relaxation factors omw = 1 - w, opw = 1 + w.
template <typename T>
__device__ __forceinline__ void prep3_terms(const Phys3<T> &P, Prep3<T> &c, T omw, T opw, const T *dr, const T *dm,
                                            const T *K) {
    constexpr T cs2 = T(1) / T(3);
    const T r = c.r, f = opw * (T(0.5) * P.dt), m = omw * r, hr = T(0.5) * opw * r;
    T uX = T(0), uV = T(0), uK = T(0), uu = T(0), uG = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c.X[k] = f * (cs2 * dr[k] - r * dm[k]);
        const T Kk = f * K[k];
        c.V[k] = fma(T(3), Kk, f * dr[k]);
        c.du[k] = P.g[k] * P.dt;
        c.G[k] = hr * c.du[k];
        c.B[k] = Kk + c.G[k];
        uX += c.u[k] * c.X[k];
        uV += c.u[k] * c.V[k];
        uK += c.u[k] * Kk;
        uu += c.u[k] * c.u[k];
        uG += c.G[k] * (c.u[k] + T(0.5) * c.du[k]);
    }
    c.nr = -r;
    c.np = -c.p;
    c.nomw = -omw;
    c.nhuu = T(-0.5) * uu;
    c.hZ = -uX;
    c.hA = fma(T(-3), uX, m);
    c.gA = m - uV;
    c.gZ = -uK - uG;
}
__device__ __forceinline__ void prep3_terms(const Phys3<float> &P, Prep3<float> &c, float omw, float opw,
                                            const float *dr, const float *dm, const float *K) {
    constexpr float cs2 = 1.0f / 3.0f;
    c.omw = omw;
    c.opw = opw;
    c.hdt = 0.5f * P.dt;
    c.uX = c.uD = c.uK = c.uu = c.udu = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c.X[k] = cs2 * dr[k] - c.r * dm[k];
        c.dr[k] = dr[k];
        c.K[k] = K[k];
        c.du[k] = P.g[k] * P.dt;
        c.uX += c.u[k] * c.X[k];
        c.uD += c.u[k] * dr[k];
        c.uK += c.u[k] * K[k];
        c.uu += c.u[k] * c.u[k];
        c.udu += c.du[k] * (2.0f * c.u[k] + c.du[k]);
    }
}

template <typename T>
__device__ __forceinline__ Prep3<T> prep3(const Phys3<T> &P, T sg, const T *mg, T r, const T *dr,
                                          const T *dm, const T *K) {
    Prep3<T> c;
    const T hdt = T(0.5) * P.dt;
    c.r = r;
    const T inv_r = recip_rn(r);
    T ud = T(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        c.u[k] = (mg[k] + hdt * K[k] + hdt * r * P.g[k]) * inv_r;
        ud += c.u[k] * dr[k];
    }
    c.p = div3(sg + hdt * ud);  // correctly rounded: a rounded 1/3 is a gain on p (see kW3)
    T C = (r - P.rho_v) * P.inv_drho;
    C = C < T(0) ? T(0) : (C > T(1) ? T(1) : C);
    const T s = C * P.inv_tau_l + (T(1) - C) * P.inv_tau_v;  // 1/tau
    const T d = recip_rn(T(2) + s);
    prep3_terms(P, c, T(2) * s * d, T(4) * d, dr, dm, K);
    return c;
}

// e.v for pair q's first direction, by sums and differences of components
template <typename T>
__device__ __forceinline__ T dir_dot3(int q, const T *v) {
    const int a = 2 * q + 1;
    T s = T(0);
    bool any = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int e = k == 0 ? e3x(a) : (k == 1 ? e3y(a) : e3z(a));
        if (e != 0) {
            const T t = e > 0 ? v[k] : -v[k];
            s = any ? s + t : t;
            any = true;
        }
    }
    return s;
}

// Collision of the opposite pair q = (a, a+1), a = 2q+1 (collide_pair's
// arithmetic in three dimensions).
template <typename T>
__device__ __forceinline__ void collide_pair3(const Prep3<T> &c, int q, V2<T> hs, V2<T> gs, V2<T> &ho, V2<T> &go,
                                              V2<T> &ds) {
    const int a = 2 * q + 1;
    const T wa = w3<T>(a), w3a = w3x3<T>(a);
    const T eu = dir_dot3<T>(q, c.u), eX = dir_dot3<T>(q, c.X), eV = dir_dot3<T>(q, c.V), eB = dir_dot3<T>(q, c.B);
    const T eG = dir_dot3<T>(q, c.G), ed = dir_dot3<T>(q, c.du);
    const T qe = fma(T(1.5) * eu, eu, c.nhuu), eA = T(3) * eX;
    const T ge = fma(eG, fma(T(1.5), ed, T(3) * eu), c.gZ);
    const V2<T> qv = vset(qe + eu, qe - eu);
    const V2<T> hz = vfma(qv, vset(c.hA + eA, c.hA - eA), vset(c.hZ + eX, c.hZ - eX));
    const V2<T> gz = vfma(qv, vset(c.gA + eV, c.gA - eV), vset(ge + eB, ge - eB));
    const V2<T> w32 = vset(w3a, w3a), nomw = vset(c.nomw, c.nomw);
    ho = vadd(hs, vfma(nomw, vfma(vset(c.nr, c.nr), vset(wa, wa), hs), vmul(w32, hz)));
    go = vadd(gs, vfma(nomw, vfma(vset(c.np, c.np), w32, gs), vmul(w32, gz)));
    ds = vadd(ds, vfma(hs, vset(T(-1), T(-1)), ho));
}

__device__ __forceinline__ PairTerms rest_terms3(const Prep3<float> &c) {
    return {0.f, 0.f, 0.f, 0.f, 0.f, c.uX, c.uD, c.uK, c.uu, c.udu, c.r, c.p, c.omw, c.opw, c.hdt};
}
__device__ __forceinline__ void collide_pair3(const Prep3<float> &c, int q, float2 hs, float2 gs, float2 &ho,
                                              float2 &go, float2 &ds) {
    const int a = 2 * q + 1;
    PairTerms t = rest_terms3(c);
    t.eu = dir_dot3<float>(q, c.u);
    t.eX = dir_dot3<float>(q, c.X);
    t.eD = dir_dot3<float>(q, c.dr);
    t.eK = dir_dot3<float>(q, c.K);
    t.ed = dir_dot3<float>(q, c.du);
    collide_terms_pair(t, w3<float>(a), w3x3<float>(a), hs, gs, ho, go);
    ds = vadd(ds, vfma(hs, vset(-1.0f, -1.0f), ho));
}

// The rest population without the mass fix.
template <typename T>
__device__ __forceinline__ void collide_rest_terms3(const Prep3<T> &c, T hs, T gs, T &h, T &go) {
    const T wa = w3<T>(0), w3a = w3x3<T>(0);
    if constexpr (sizeof(T) == 4) {
        collide_terms_rest(rest_terms3(c), wa, w3a, hs, gs, h, go);
    } else {
        h = hs + fma(c.nomw, fma(c.nr, wa, hs), w3a * fma(c.nhuu, c.hA, c.hZ));
        go = gs + fma(c.nomw, fma(c.np, w3a, gs), w3a * fma(c.nhuu, c.gA, c.gZ));
    }
}
// Its h takes the sum of the node's h increments (see collide_rest).
template <typename T>
__device__ __forceinline__ void collide_rest3(const Prep3<T> &c, T hs, T gs, V2<T> ds, T &ho, T &go) {
    T h;
    collide_rest_terms3<T>(c, hs, gs, h, go);
    ho = h - ((ds.x + ds.y) + (h - hs));
}

template <typename T, typename Topo>
struct Collide3Args {
    Topo m;
    const T *fin;
    T *fout;
    Fields3<T> F;
    Phys3<T> P;
    T *mom;  // 5N (rho, ux, uy, uz, p) or nullptr
    int *flag;
};

// The rest of a node's update from grad mu dm, the sum sg and first moments
// mg of its streamed g and the scalars of the collision.
template <typename T, typename Topo>
__device__ __forceinline__ Prep3<T> prep3_node(const Collide3Args<T, Topo> &A, int32_t i, T sg, const T *mg,
                                               const T *dm) {
    T dr[3], K[3];
    load_grad3<T>(pdl_ptr(A.F.dr4), i, dr);
#pragma unroll
    for (int c = 0; c < 3; ++c) K[c] = ldp(pdl_ptr(A.F.k[c]) + i);
    return prep3<T>(A.P, sg, mg, ldp(pdl_ptr(A.F.rho) + i), dr, dm, K);
}

// Finite check and, on the last step of a call, the moments.
template <typename T, typename Topo>
__device__ __forceinline__ void moments_out3(const Collide3Args<T, Topo> &A, int32_t i, const Prep3<T> &c) {
    if (!(finite_val(c.r) && finite_val(c.u[0]) && finite_val(c.u[1]) && finite_val(c.u[2]) && finite_val(c.p)))
        atomicOr(A.flag, 1);
    if (A.mom) {
        const size_t n = (size_t)A.m.n;
        A.mom[i] = c.r;
        A.mom[n + i] = c.u[0];
        A.mom[2 * n + i] = c.u[1];
        A.mom[3 * n + i] = c.u[2];
        A.mom[4 * n + i] = c.p;
    }
}

// Adds pair q's part of the moments of g: first moments from the differences
// of opposite pairs.
template <typename T>
__device__ __forceinline__ void add_moments3(int q, V2<T> g, T &sg, T *mg) {
    const int a = 2 * q + 1;
    const T d = g.x - g.y;
    sg += g.x + g.y;
    mg[0] += T(e3x(a)) * d;
    mg[1] += T(e3y(a)) * d;
    mg[2] += T(e3z(a)) * d;
}

template <typename T, typename Topo>
__global__ void __launch_bounds__(kSplitBlock, sizeof(T) == 4 ? 4 : 2)
    k_collide3_split(const __grid_constant__ Collide3Args<T, Topo> A) {
    // moments of g by group; grad mu in [4 ..][0]; the groups' h increments in [5 ..][1 ..]
    __shared__ T part[7][kSplitGroups][kSplitNodes];
    // FP64: one group forms the scalars of a node for all three (its pipe
    // bounds the pass; in FP32 each group forms them, a barrier less)
    constexpr bool kShare = sizeof(T) == 8;
    const int l = threadIdx.x % kSplitNodes, grp = threadIdx.x / kSplitNodes;
    const int32_t i = blockIdx.x * kSplitNodes + l;
    const Topo &m = A.m;
    const bool in = i < m.n;
    const size_t np = pad4((size_t)m.n);
    const int k = in ? m.tag_of(i) : 0;
    pdl_wait();
    const T *g = pdl_ptr(A.fin) + 19 * np;
    const T *hs = pdl_ptr(A.F.hs), *mu = pdl_ptr(A.F.mu);
    V2<T> gp[3], hp[3];
    T g0 = T(0), h0 = T(0);
    if (in) {
        by_group(grp, [&](auto G) {
            constexpr int Q0 = split_first(decltype(G)::value), NQ = split_count(decltype(G)::value);
            by_kind(m, i, [&](auto K) {
                stream_range3<T, Q0, NQ, decltype(K)::value>(m, g, np, i, A.P.dt, gp);
                if (decltype(G)::value == kSplitGroups - 1) {
                    T dm[3];
                    recover3<T, decltype(K)::value>(m, mu, i, dm);
#pragma unroll
                    for (int c = 0; c < 3; ++c) part[4 + c][0][l] = dm[c];
                }
            });
            // h: streamed and bounced back by the rho pass
            const V2<T> *hb = reinterpret_cast<const V2<T> *>(hs + np);
            T sg = T(0), mg[3] = {T(0), T(0), T(0)};
            if (decltype(G)::value == 0) {
                g0 = sg = ldp(g + i);
                h0 = ldp(hs + i);
            }
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                hp[q] = ldp(hb + (Q0 + q) * np + i);
                if (k) bounce_pair3<T>(k, Q0 + q, gp[q]);
                add_moments3<T>(Q0 + q, gp[q], sg, mg);
            }
            part[0][grp][l] = sg;
#pragma unroll
            for (int c = 0; c < 3; ++c) part[1 + c][grp][l] = mg[c];
        });
    }
    __syncthreads();
    V2<T> ds = vset(T(0), T(0));
    Prep3<T> c;
    if (in && (!kShare || grp == 0)) {
        T s[4], dm[3];
#pragma unroll
        for (int v = 0; v < 4; ++v) s[v] = group_sum(part[v], l);
#pragma unroll
        for (int v = 0; v < 3; ++v) dm[v] = part[4 + v][0][l];
        c = prep3_node(A, i, s[0], s + 1, dm);
    }
    if constexpr (kShare) {
        constexpr int NV = sizeof(Prep3<T>) / sizeof(T);
        __shared__ T sc[NV][kSplitNodes];
        T *cv = reinterpret_cast<T *>(&c);
        if (grp == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) sc[v][l] = cv[v];
        }
        __syncthreads();
#pragma unroll
        for (int v = 0; v < NV; ++v) cv[v] = sc[v][l];
    }
    if (in) {
        V2<T> *ho = reinterpret_cast<V2<T> *>(A.fout + np);
        V2<T> *go = reinterpret_cast<V2<T> *>(A.fout + 20 * np);
        by_group(grp, [&](auto G) {
            constexpr int Q0 = split_first(decltype(G)::value), NQ = split_count(decltype(G)::value);
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                V2<T> h, gg;
                collide_pair3(c, Q0 + q, hp[q], gp[q], h, gg, ds);
                ho[(Q0 + q) * np + i] = h;
                go[(Q0 + q) * np + i] = gg;
            }
        });
        if (grp > 0) {  // (entries that grad mu leaves free)
            part[5][grp][l] = ds.x;
            part[6][grp][l] = ds.y;
        }
    }
    __syncthreads();
    if (grp == 0 && in) {
#pragma unroll
        for (int v = 1; v < kSplitGroups; ++v) {
            ds.x += part[5][v][l];
            ds.y += part[6][v][l];
        }
        collide_rest3<T>(c, h0, g0, ds, A.fout[i], A.fout[19 * np + i]);
        moments_out3(A, i, c);
    }
}

// (all loads before the first store: interleaved with them the pass took
// 232 us, not 172, on a 128^3 lattice in FP32)
// UNI: the interior takes the integer weights (read here instead it cost 1 % of a step).
template <typename T, bool UNI>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 1)
    k_collide3_node(const __grid_constant__ Collide3Args<T, DevLattice3<T>> A) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const DevLattice3<T> &m = A.m;
    if (i >= m.n) return;
    const size_t np = pad4((size_t)m.n);
    pdl_wait();
    const T *g = pdl_ptr(A.fin) + 19 * np;
    const T *hs = pdl_ptr(A.F.hs), *mu = pdl_ptr(A.F.mu);
    T dm[3];
    V2<T> hp[9], gp[9];
    by_kind(m, i, [&](auto K) {
        if (decltype(K)::value == 0 && UNI)
            kuhn_recover_node<T>(m, mu, i, dm);
        else
            recover3<T, decltype(K)::value>(m, mu, i, dm);
        stream_all3<T, decltype(K)::value>(m, g, np, i, A.P.dt, gp);
    });
    const T g0 = ldp(g + i), h0 = ldp(hs + i);
    // h: streamed and bounced back by the rho pass
    const V2<T> *hb = reinterpret_cast<const V2<T> *>(hs + np);
#pragma unroll
    for (int q = 0; q < 9; ++q) hp[q] = ldp(hb + q * np + i);
    const int k = m.tag_of(i);
    T sg = g0, mg[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        if (k) bounce_pair3<T>(k, q, gp[q]);
        add_moments3<T>(q, gp[q], sg, mg);
    }
    const Prep3<T> c = prep3_node(A, i, sg, mg, dm);
    V2<T> *ho = reinterpret_cast<V2<T> *>(A.fout + np);
    V2<T> *go = reinterpret_cast<V2<T> *>(A.fout + 20 * np);
    V2<T> ds = vset(T(0), T(0));
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        V2<T> h, gg;
        collide_pair3(c, q, hp[q], gp[q], h, gg, ds);
        ho[q * np + i] = h;
        go[q * np + i] = gg;
    }
    collide_rest3<T>(c, h0, g0, ds, A.fout[i], A.fout[19 * np + i]);
    moments_out3(A, i, c);
}

// Initial pre-collided state psibar = eq + S of (rho, u, p) in mom.
template <typename T, typename Topo>
__global__ void __launch_bounds__(128) k_init3(const __grid_constant__ Topo m, T *__restrict__ fout,
                                               Fields3<T> F, Phys3<T> P, const T *__restrict__ mom) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const size_t n = (size_t)m.n, np = pad4(n);
    T dm[3], dr[3], K[3];
    by_kind(m, i, [&](auto KD) { recover3<T, decltype(KD)::value>(m, F.mu, i, dm); });
    load_grad3<T>(F.dr4, i, dr);
#pragma unroll
    for (int c = 0; c < 3; ++c) K[c] = F.k[c][i];
    const T r = mom[i];
    Prep3<T> c;
    c.r = r;
    c.p = mom[4 * n + i];
#pragma unroll
    for (int k = 0; k < 3; ++k) c.u[k] = mom[(1 + k) * n + i];
    // eq + S: the collision's increment with 1 - w = 1 and 1 + w = 1 from
    // psi* = 0
    prep3_terms(P, c, T(1), T(1), dr, dm, K);
    V2<T> *hb = reinterpret_cast<V2<T> *>(fout + np);
    V2<T> *gb = reinterpret_cast<V2<T> *>(fout + 20 * np);
    const V2<T> zero = vset(T(0), T(0));
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        V2<T> h, g, ds = zero;
        collide_pair3(c, q, zero, zero, h, g, ds);
        hb[q * np + i] = h;
        gb[q * np + i] = g;
    }
    collide_rest_terms3<T>(c, T(0), T(0), fout[i], fout[19 * np + i]);
}

// Moments in caller order, FP64: out[0..N) rho, [N..2N) C, [2N..5N) u
// interleaved (ux, uy, uz), [5N..6N) p.
template <typename T>
__global__ void k_gather_moments3(int32_t n, const T *__restrict__ mom, const int32_t *__restrict__ iperm,
                                  double rho_l, double rho_v, double *__restrict__ out) {
    const int32_t c = blockIdx.x * blockDim.x + threadIdx.x;  // caller id
    if (c >= n) return;
    const int32_t i = iperm[c];
    const size_t N = (size_t)n;
    const double r = (double)mom[i];
    out[c] = r;
    out[N + c] = (r - rho_v) / (rho_l - rho_v);
    for (int k = 0; k < 3; ++k) out[2 * N + 3 * (size_t)c + k] = (double)mom[(1 + k) * N + i];
    out[5 * N + c] = (double)mom[4 * N + i];
}

// FP64 totals: per-block partials of sum m rho and sum m rho u (4 values,
// [4][blocks]), then one warp reduces them in a fixed order.
template <typename T>
__global__ void __launch_bounds__(256) k_totals3_partial(int32_t n, const T *__restrict__ mom,
                                                         const double *__restrict__ mass,
                                                         double *__restrict__ part) {
    __shared__ double s[4][256];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const size_t N = (size_t)n;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double mr = mass[i] * (double)mom[i];
        acc[0] += mr;
        for (int k = 0; k < 3; ++k) acc[1 + k] += mr * (double)mom[(1 + k) * N + i];
    }
    for (int k = 0; k < 4; ++k) s[k][threadIdx.x] = acc[k];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int k = 0; k < 4; ++k) s[k][threadIdx.x] += s[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) part[(size_t)k * gridDim.x + blockIdx.x] = s[k][0];
}

__global__ void k_totals3_final(int nparts, const double *__restrict__ part, double *__restrict__ out) {
    const int l = threadIdx.x;
    for (int k = 0; k < 4; ++k) {
        double v = 0.0;
        for (int b = l; b < nparts; b += 32) v += part[(size_t)k * nparts + b];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (l == 0) out[k] = v;
    }
}

}  // namespace felbm
