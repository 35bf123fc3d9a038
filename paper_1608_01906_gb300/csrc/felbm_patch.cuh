// Step of a general triangle mesh in two launches: k_rho (streamed h, rho),
// then k_patch_step, one block per patch of kPatch nodes (a compact piece of
// the mesh along a Hilbert curve, internal order patch-major).  A node's
// collision depends on rho up to 3 edges away (rho -> grad rho -> lap rho and
// mu -> grad mu, Sec. 2.1 and Sec. 2.3), so the block
//   0. gathers rho on its region (own nodes and rings 1..3) into shared
//      memory, and streams the g pairs of its own nodes, which need no rho;
//   1. recovers grad rho on rings <= 2, then
//   2. lap rho and mu on rings <= 1 (and the stress force at its own nodes);
//   3. at its own node: grad mu, the moments and the collision, and one
//      write of the 18 populations.
// The rows of rings <= 2 (recovery coefficients and 16-bit region indices,
// sliced as DevELL's) are copied to shared memory by cp.async before the
// block waits for k_rho, so that a stage waits for shared memory only.
// Every stage is the four-launch path's per-node arithmetic in the same
// order (k_grad, k_mu, k_collide), so both give the same results bit for bit.
//
// What bounds it: latency below about 10^5 nodes (one wave of blocks; three
// dependent gathers and four barriers), bytes above (about 450 of rows a node
// in the two launches, 190 in k_rho, 260 here, beside 220 of populations, h*
// and rho).  Streaming h on rings
// <= 3 here too, in one launch, redid the costliest pass 1.9 times and waited
// for its rows' coefficients in each stage: 24.5 us a step against 10.7 on a
// 256 x 256 jittered Delaunay mesh (FP32), 270 against 159 on 1024 x 1024.
#pragma once

#include "felbm_internal.h"
#include "felbm_kernels.cuh"

namespace felbm {

template <typename T>
struct PatchArgs {
    CollideArgs<T, DevELL<T>> c;
    const int32_t *nbase;   // region list offsets, one per patch + 1
    const int32_t *count;   // per patch: nodes of rings <= 0, 1, 2, 3
    const int32_t *node;    // region nodes (internal ids), own first
    const int32_t *pslice;  // first slice of each patch in psbase
    const int32_t *psbase;  // first row of 32 entries of each slice, their end, the patch's end
    const int32_t *pstail;  // of each slice: -1, or its table of further entries (LONG)
    const int2 *ptail;      // first of them (from the patch's first entry) and count, 32 a table
    const uint16_t *pcol;   // region index of each entry
    const V2<T> *pa;        // recovery coefficients of each entry (a_x, a_y)
    const V2<double> *pa64; // the same in FP64 (LAP64 only)
    int32_t r1max, r2max, r3max, pemax, psmax;
    double kappa64;
};

// Shared-memory bytes of one block (layout of k_patch_step).
template <typename T>
inline size_t patch_smem(int32_t r1max, int32_t r2max, int32_t r3max, int32_t pemax, int32_t psmax) {
    return (size_t)pemax * 32 * (sizeof(V2<T>) + sizeof(uint16_t)) + (size_t)r2max * sizeof(V2<T>) +
           (size_t)(r3max + r1max) * sizeof(T) + (size_t)(psmax + 1) * sizeof(int32_t);
}

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(smem)),
                 "l"(gmem)
                 : "memory");
}

// LAP64: the kappa lap rho term of mu in FP64, as k_mu_lap64 forms it.  Its
// FP64 coefficients are read from global memory where they are used; staged in
// place of the FP32 ones, they made every stage convert (the conversions take
// the FP64 pipe).
// ONE: all blocks are resident at once with two per SM, whose registers then
// hold more gathers in flight (jittered Delaunay meshes, FP32, both launches:
// 256 x 256 10.7 us a step with two blocks per SM, 13.2 with three; 300 x 300,
// 352 blocks, 17.6 and 13.9; 1024 x 1024 182 and 159).
// LONG: some rows have entries behind the slices (HostCSR::ptail).
template <typename T, bool LAP64, bool ONE, bool LONG>
__global__ void __launch_bounds__(kPatch, sizeof(T) == 4 ? (ONE ? 2 : 3) : 1) k_patch_step(const __grid_constant__ PatchArgs<T> A) {
    using CT = typename std::conditional<LAP64, double, T>::type;  // of lap rho
    extern __shared__ __align__(16) unsigned char psm[];
    const DevELL<T> &m = A.c.m;
    const int p = blockIdx.x, tid = threadIdx.x;
    const int32_t n = m.n;
    // (the two cp.async destinations first: whole 32-entry rows keep both, and
    // what follows, 16-byte aligned)
    V2<T> *pa = reinterpret_cast<V2<T> *>(psm);                               // [pemax * 32]
    uint16_t *pc = reinterpret_cast<uint16_t *>(pa + (size_t)A.pemax * 32);   // [pemax * 32]
    V2<T> *grd = reinterpret_cast<V2<T> *>(pc + (size_t)A.pemax * 32);        // [r2max]
    T *rho = reinterpret_cast<T *>(grd + A.r2max);                            // [r3max]
    T *mu = rho + A.r3max;                                                    // [r1max]
    int32_t *sb = reinterpret_cast<int32_t *>(mu + A.r1max);                  // [psmax + 1]
    // 0. static data: rows, region ids, the own node's row
    const int32_t base = __ldg(A.nbase + p);
    const int4 cnt = __ldg(reinterpret_cast<const int4 *>(A.count) + p);
    const int32_t n0 = cnt.x, n1 = cnt.y, n2 = cnt.z, n3 = cnt.w;
    const int32_t s0 = __ldg(A.pslice + p), e0 = __ldg(A.psbase + s0);
    {
        const int32_t ns = (n2 + 31) / 32, rows = __ldg(A.psbase + s0 + ns + 1) - e0;
        for (int s = tid; s <= ns; s += kPatch) sb[s] = (__ldg(A.psbase + s0 + s) - e0) * 32;
        const char *ga = reinterpret_cast<const char *>(A.pa + (size_t)e0 * 32);
        const char *gc = reinterpret_cast<const char *>(A.pcol + (size_t)e0 * 32);
        const int ba = rows * 32 * (int)sizeof(V2<T>), bc = rows * 64;
        for (int b = tid * 16; b < ba; b += kPatch * 16) cp_async16(reinterpret_cast<char *>(pa) + b, ga + b);
        for (int b = tid * 16; b < bc; b += kPatch * 16) cp_async16(reinterpret_cast<char *>(pc) + b, gc + b);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    const bool own = tid < n0;
    const int32_t g = own ? p * kPatch + tid : p * kPatch;
    const int32_t g1 = tid + kPatch < n3 ? __ldg(A.node + base + tid + kPatch) : g;
    const auto row = m.template row<false>(g);
    const int tag = m.tag_of(g);
    pdl_wait();
    if (ONE) pdl_trigger();
    // rho of the region, in flight while g is streamed (the own rows' a from
    // shared memory, the rest of their entries from the mesh's rows)
    const T *grho = A.c.F.rho;
    const T rho_own = grho[g], rho1 = chk_idx(g1, n, 1u) ? grho[g1] : T(0);
    const size_t np = pad4(m.slots());
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    V2<T> gs[4];
    // the entries of region row r behind the slices
    auto further = [&](int32_t r) {
        int32_t t = -1;
        if (LONG) t = __ldg(A.pstail + s0 + (r >> 5));
        return t < 0 ? make_int2(0, 0) : __ldg(A.ptail + 32 * (size_t)t + (r & 31));
    };
    {
        const int o0 = own ? sb[tid >> 5] + (tid & 31) : 0;
        const int2 q0 = further(own ? tid : 0);
        stream_pairs<T>(m, A.c.fin + 9 * np, np, g, A.c.P.dt, gs, [&](auto &&fn) {
            m.template each_get<false>(row, fn, [&](int k, Ell2<T>) {
                Ell2<T> v{T(0), T(0)};
                if (k < row.deg && (!LONG || k < kPatchRow + q0.y)) {
                    const V2<T> a = pa[!LONG || k < kPatchRow ? o0 + 32 * k : q0.x + (k - kPatchRow)];
                    v = {a.x, a.y};
                }
                return v;
            });
        });
        if (tag) bounce_pairs<T>(tag, gs);
    }
    const T g0 = A.c.fin[9 * np + g];
    if (tid < n3) rho[tid] = own ? rho_own : grho[__ldg(A.node + base + tid)];
    if (tid + kPatch < n3) rho[tid + kPatch] = rho1;
    for (int32_t r = tid + 2 * kPatch; r < n3; r += kPatch) {
        const int32_t j = __ldg(A.node + base + r);
        rho[r] = chk_idx(j, n, 1u) ? grho[j] : T(0);
    }
    __syncthreads();
    // fn(j, a, e) for the entries e of region row r (lim: rows in the next ring)
    auto each = [&](int32_t r, int32_t lim, auto &&fn) {
        const int32_t e1 = sb[(r >> 5) + 1];
#pragma unroll 4
        for (int32_t e = sb[r >> 5] + (r & 31); e < e1; e += 32) {
            const int j = pc[e];
            if (chk_idx(j, lim, 2u)) fn(j, pa[e], e);
        }
        if (LONG) {
            const int2 q = further(r);
#pragma unroll 4
            for (int32_t e = q.x; e < q.x + q.y; ++e) {
                const int j = pc[e];
                if (chk_idx(j, lim, 2u)) fn(j, pa[e], e);
            }
        }
    };
    // 1. recovered grad rho on rings <= 2 (k_grad)
    for (int32_t r = tid; r < n2; r += kPatch) {
        const T fi = rho[r];
        T gx = T(0), gy = T(0);
        each(r, n3, [&](int j, V2<T> a, int) { grad_edge<T>(a.x, a.y, rho[j] - fi, gx, gy); });
        grd[r] = vset(gx, gy);
    }
    __syncthreads();
    // 2. lap rho and mu on rings <= 1, the stress force at the own node (k_mu)
    T kx_own = T(0), ky_own = T(0);
    auto lap_of = [&](V2<T> a, int e, V2<T> gi, V2<T> gj, CT &lap) {
        if constexpr (LAP64) {
            const double2 c = __ldg(reinterpret_cast<const double2 *>(A.pa64) + (size_t)e0 * 32 + e);
            lap_edge<CT>(c.x, c.y, gi.x, gi.y, gj.x, gj.y, lap);
        } else {
            lap_edge<T>(a.x, a.y, gi.x, gi.y, gj.x, gj.y, lap);
        }
    };
    for (int32_t r = tid; r < n1; r += kPatch) {
        const V2<T> gi = grd[r];
        T kx = T(0), ky = T(0);
        CT lap = CT(0);
        if (r < n0) {
            each(r, n2, [&](int j, V2<T> a, int e) {
                const V2<T> gj = grd[j];
                lap_of(a, e, gi, gj, lap);
                stress_edge<T>(a.x, a.y, gi.x, gi.y, gj.x, gj.y, kx, ky);
            });
            kx_own = A.c.P.kappa * kx;
            ky_own = A.c.P.kappa * ky;
        } else {
            each(r, n2, [&](int j, V2<T> a, int e) {
                const V2<T> gj = grd[j];
                lap_of(a, e, gi, gj, lap);
            });
        }
        if (LAP64)
            mu[r] = (T)((double)mu_bulk<T>(A.c.P, rho[r]) - A.kappa64 * (double)lap);
        else
            mu[r] = mu_bulk<T>(A.c.P, rho[r]) - A.c.P.kappa * (T)lap;
    }
    __syncthreads();
    // 3. own node: grad mu and the collision (k_collide)
    if (!own) return;
    T dmx = T(0), dmy = T(0);
    {
        const T fi = mu[tid];
        each(tid, n1, [&](int j, V2<T> a, int) { grad_edge<T>(a.x, a.y, mu[j] - fi, dmx, dmy); });
    }
    const V2<T> gr = grd[tid];
    collide_write<T>(A.c, g, np, g0, gs, rho_own, gr.x, gr.y, dmx, dmy, kx_own, ky_own);
}

}  // namespace felbm
