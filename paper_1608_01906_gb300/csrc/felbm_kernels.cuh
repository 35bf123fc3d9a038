// Device kernels of one FE-LBM time step, general (unstructured CSR) path.
//
// One step = four dependent neighbour passes, each a gather over the
// assembled per-node operators (HostCSR in felbm_internal.h):
//   k_rho      Taylor-Galerkin streaming of the 9 h populations (Sec. 2.2.1,
//              Eq. galerkin_lbm with the lumped mass), wall bounce-back,
//              rho = sum_a h_a.
//   k_grad     recovered grad rho (Sec. 2.3).
//   k_mu       Laplacian of rho (recovery of the recovered gradient), the
//              stress force K = kappa [d_i |grad rho|^2 - d_j (d_i rho d_j rho)]
//              and mu = mu_phi(rho) - kappa lap rho (Sec. 2.1).
//   k_collide  recovered grad mu; streaming of all 18 populations; bounce-back;
//              moments (Eqs. velocity, pressure); post-streaming collision and
//              the next pre-streaming collision (Sec. 2.2) in one update.
// Operators use the difference form sum_{j != i} c_ij (f_j - f_i), exact for
// constant fields in any precision.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "felbm_internal.h"

namespace felbm {

// D2Q9 velocity components, weights, opposite directions.
__host__ __device__ constexpr int kEx(int a) { return a == 1 || a == 5 || a == 8 ? 1 : (a == 3 || a == 6 || a == 7 ? -1 : 0); }
__host__ __device__ constexpr int kEy(int a) { return a == 2 || a == 5 || a == 6 ? 1 : (a == 4 || a == 7 || a == 8 ? -1 : 0); }
__host__ __device__ constexpr int kOpp(int a) { return a == 0 ? 0 : (a <= 4 ? ((a + 1) % 4) + 1 : ((a - 5 + 2) % 4) + 5); }
template <typename T>
__host__ __device__ constexpr T kW(int a) { return a == 0 ? T(4) / T(9) : (a <= 4 ? T(1) / T(9) : T(1) / T(36)); }

// 1/12 rounded to a multiple of 2^-25 (FP32) or 2^-54 (FP64): the base of the
// 3 w_a constants below, chosen so that they are exact in T.
template <typename T>
__host__ __device__ constexpr T kTwelfth() {
    return sizeof(T) == 4 ? T(2796203.0 / 33554432.0) : T(1501199875790165.0 / 18014398509481984.0);
}

// 3 w_a in the working precision, with the moment identities of the
// equilibria exact in T: sum_a 3 w_a = 3 (w3_0 + 4 w3_1 + 4 w3_5) and
// sum_a 3 w_a e_ax^2 = 1 (2 w3_1 + 4 w3_5), from e ~ 1/12: w3_5 = e,
// w3_1 = (1 - 4 e)/2, w3_0 = 1 + 4 e.  The nearest values to 4/3, 1/3, 1/12
// miss both identities by about one rounding; through the pressure and the
// momentum of g that bias is a gain on p and u applied every step, which a
// near-steady FP32 run accumulates (1.3e-5 in u after 1000 steps of a
// droplet, against 1.3e-6 with these constants).
template <typename T>
__host__ __device__ constexpr T kW3(int a) {
    return a == 0 ? T(1) + T(4) * kTwelfth<T>() : (a <= 4 ? (T(1) - T(4) * kTwelfth<T>()) / T(2) : kTwelfth<T>());
}

template <typename T>
__device__ __forceinline__ bool finite_val(T v) { return isfinite(v); }

// ---- packed two-wide arithmetic on a pair of opposite populations ----

template <typename T>
struct V2T;
template <>
struct V2T<float> {
    using type = float2;
};
template <>
struct V2T<double> {
    using type = double2;
};
template <typename T>
using V2 = typename V2T<T>::type;

// packed two-wide arithmetic (one instruction per operation in FP32)
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
    return make_double2(fma(a.x, b.x, c.x), fma(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 vset(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 vset(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }


// Streaming coefficient of direction a from the assembled tensors:
//   c = e.a_ij + (dt/2) e.b_ij.e
template <typename T, int A>
__device__ __forceinline__ T stream_coef(T ax, T ay, T hbxx, T hbxy, T hbyy) {
    constexpr int ex = kEx(A), ey = kEy(A);
    T c = T(0);
    if (ex) c += T(ex) * ax + hbxx;
    if (ey) c += T(ey) * ay + hbyy;
    if (ex && ey) c += T(2 * ex * ey) * hbxy;
    return c;
}

// Streaming coefficients of pair q (directions pair_dir(q, 0), its opposite):
// c = e.a_ij + (dt/2) e.b_ij.e, the odd part e.a flipping sign between the
// two; the slot-0 directions are (1,0), (0,1), (1,1), (-1,1).
template <typename T>
__device__ __forceinline__ V2<T> pair_coef(int q, T ax, T ay, T hbxx, T hbxy, T hbyy) {
    T odd, even;
    if (q == 0) {
        odd = ax;
        even = hbxx;
    } else if (q == 1) {
        odd = ay;
        even = hbyy;
    } else if (q == 2) {
        odd = ax + ay;
        even = (hbxx + hbyy) + T(2) * hbxy;
    } else {
        odd = ay - ax;
        even = (hbxx + hbyy) - T(2) * hbxy;
    }
    return vset(even + odd, even - odd);
}

// Streamed pairs of node i of one distribution (f: its rest values, pair q
// at f + np + 2 np q, np = padded slot count): psi* = psi - dt sum_{j != i}
// c_ij (psi_j - psi_i), one 8-byte load per pair and neighbour.  each(fn)
// calls fn(j, ax, ay, bxx, bxy, byy) for the node's neighbours.
template <typename T, typename Topo, typename Each>
__device__ __forceinline__ void stream_pairs(const Topo &m, const T *f, size_t np, int32_t i, T dt, V2<T> *out,
                                             Each &&each) {
    const V2<T> *pb = reinterpret_cast<const V2<T> *>(f + np);
    const size_t si = m.slot(i);
    const V2<T> m1 = vset(T(-1), T(-1));
    V2<T> own[4], acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        own[q] = pb[q * np + si];
        acc[q] = vset(T(0), T(0));
    }
    const T hdt = T(0.5) * dt;
    each([&](int32_t j, T ax, T ay, T bxx, T bxy, T byy) {
        const size_t sj = m.slot(j);
        const T hbxx = hdt * bxx, hbxy = hdt * bxy, hbyy = hdt * byy;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const V2<T> c = pair_coef<T>(q, ax, ay, hbxx, hbxy, hbyy);
            acc[q] = vfma(c, vfma(own[q], m1, pb[q * np + sj]), acc[q]);
        }
    });
    const V2<T> mdt = vset(-dt, -dt);
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = vfma(mdt, acc[q], own[q]);
}

// Bounce-back at a wall node with inward normal e_k: every population with
// e_a . e_k > 0 takes the value of its opposite.
template <typename T>
__device__ __forceinline__ void bounce_pairs(int k, V2<T> *p) {
    const int nx = kEx(k), ny = kEy(k);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int a = pair_dir(q, 0), d = kEx(a) * nx + kEy(a) * ny;
        if (d > 0) p[q].x = p[q].y;
        if (d < 0) p[q].y = p[q].x;
    }
}

// ONE: the mesh's blocks are all resident at once (see kOneWave); they may
// then have more registers, for more gathers in flight.
template <typename T, typename Topo, bool ONE>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? (ONE ? 4 : 5) : 2)
    k_rho(const __grid_constant__ Topo m, const T *f, T dt, T *rho, T *hs) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const size_t np = pad4(m.slots());
    const auto row = m.row(i);
    const int k = m.tag_of(i);
    pdl_wait();
    if (ONE) pdl_trigger();
    V2<T> hp[4];
    stream_pairs<T>(m, f, np, i, dt, hp, [&](auto &&fn) { m.each(row, fn); });
    const size_t si = m.slot(i);
    const T h0 = f[si];
    if (k) bounce_pairs<T>(k, hp);
    rho[i] = ((h0 + (hp[0].x + hp[0].y)) + (hp[1].x + hp[1].y)) + ((hp[2].x + hp[2].y) + (hp[3].x + hp[3].y));
    V2<T> *hb = reinterpret_cast<V2<T> *>(hs + np);
#pragma unroll
    for (int q = 0; q < 4; ++q) hb[q * np + si] = hp[q];
    hs[si] = h0;
}

// One neighbour's part of a recovered gradient (d: difference of the field).
template <typename T>
__device__ __forceinline__ void grad_edge(T ax, T ay, T d, T &gx, T &gy) {
    gx = fma(ax, d, gx);
    gy = fma(ay, d, gy);
}

// Recovered gradient of a scalar field.
template <typename T, typename Topo>
__device__ __forceinline__ void recover(const Topo &m, const typename Topo::Row &row, const T *f,
                                        int32_t i, T &gx, T &gy) {
    const T fi = f[i];
    gx = gy = T(0);
    m.each(row, [&](int32_t j, T ax, T ay, T, T, T) { grad_edge<T>(ax, ay, f[j] - fi, gx, gy); });
}

template <typename T, typename Topo>
__global__ void __launch_bounds__(256) k_grad(const __grid_constant__ Topo m, Fields<T> F) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const auto row = m.row(i);
    pdl_wait();
    T gx, gy;
    recover(m, row, F.rho, i, gx, gy);
    F.drx[i] = gx;
    F.dry[i] = gy;
}

// mu_phi = 4 beta (rho - rho_v)(rho - rho_l)(rho - (rho_v + rho_l)/2).
template <typename T>
__device__ __forceinline__ T mu_bulk(const Phys<T> &P, T r) {
    return T(4) * P.beta * (r - P.rho_v) * (r - P.rho_l) * (r - T(0.5) * (P.rho_v + P.rho_l));
}

// lap rho = R_x(d_x rho) + R_y(d_y rho);
// K_x = kappa [R_x((d_y rho)^2) - R_y(d_x rho d_y rho)],
// K_y = kappa [R_y((d_x rho)^2) - R_x(d_x rho d_y rho)]
// (the printed form d_i(|grad rho|^2) - d_j(d_i rho d_j rho) with the
// identical (d_i rho)^2 contributions cancelled, R linear);
// mu = 4 beta (rho - rho_v)(rho - rho_l)(rho - (rho_v + rho_l)/2) - kappa lap rho.
// One neighbour's part of K / kappa, with the differences of the gradient
// products in product form (no cancellation between two squares of nearly
// equal size).
template <typename T>
__device__ __forceinline__ void stress_edge(T ax, T ay, T gxi, T gyi, T gxj, T gyj, T &kx, T &ky) {
    const T ddx = gxj - gxi, ddy = gyj - gyi;
    const T dxx = ddx * (gxj + gxi), dxy = fma(gxj, ddy, gyi * ddx), dyy = ddy * (gyj + gyi);
    kx = fma(ax, dyy, fma(-ay, dxy, kx));
    ky = fma(ay, dxx, fma(-ax, dxy, ky));
}
// One neighbour's part of lap rho.
template <typename T>
__device__ __forceinline__ void lap_edge(T ax, T ay, T gxi, T gyi, T gxj, T gyj, T &lap) {
    lap = fma(ax, gxj - gxi, fma(ay, gyj - gyi, lap));
}

template <typename T, typename Topo>
__global__ void __launch_bounds__(256) k_mu(const __grid_constant__ Topo m, Fields<T> F, Phys<T> P) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const auto row = m.row(i);
    pdl_wait();
    const T gxi = F.drx[i], gyi = F.dry[i];
    T lap = T(0), kx = T(0), ky = T(0);
    m.each(row, [&](int32_t j, T ax, T ay, T, T, T) {
        const T gxj = F.drx[j], gyj = F.dry[j];
        lap_edge<T>(ax, ay, gxi, gyi, gxj, gyj, lap);
        stress_edge<T>(ax, ay, gxi, gyi, gxj, gyj, kx, ky);
    });
    F.mu[i] = mu_bulk<T>(P, F.rho[i]) - P.kappa * lap;
    F.kx[i] = P.kappa * kx;
    F.ky[i] = P.kappa * ky;
}

// k_mu for FP32 fields with the kappa lap rho term of mu in FP64
// (FELBM_PARAM_LAP_FP64): Topo64 carries the mesh's FP64 coefficients; the
// Laplacian of the FP32 gradient and its product with kappa are formed in
// FP64 and subtracted from the bulk term in FP64, rounded once.  K is formed
// as in k_mu, from the same coefficients rounded to FP32.
template <typename Topo64>
__global__ void __launch_bounds__(256) k_mu_lap64(const __grid_constant__ Topo64 m, Fields<float> F, Phys<float> P,
                                                  double kappa) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const auto row = m.row(i);
    pdl_wait();
    const float gxi = F.drx[i], gyi = F.dry[i];
    double lap = 0.0;
    float kx = 0.f, ky = 0.f;
    m.each(row, [&](int32_t j, double ax, double ay, double, double, double) {
        const float gxj = F.drx[j], gyj = F.dry[j];
        lap_edge<double>(ax, ay, gxi, gyi, gxj, gyj, lap);
        stress_edge<float>((float)ax, (float)ay, gxi, gyi, gxj, gyj, kx, ky);
    });
    F.mu[i] = (float)((double)mu_bulk<float>(P, F.rho[i]) - kappa * lap);
    F.kx[i] = P.kappa * kx;
    F.ky[i] = P.kappa * ky;
}

// Local collision of one node (Sec. 2.2), split in two so that callers can
// keep the streamed populations outside registers:
//   collide_prep  moments (Eqs. velocity, pressure), tau, and the per-node
//                 scalars of the equilibria and sources;
//   collide_pair  the update of a pair of opposite directions.
// With eq and source S of the node, the post-streaming collision
//   psi = psi* + 2tau/(2tau+1) (-(psi* - eq)/(2tau) + S)
// followed by the pre-streaming collision of the next step
//   psibar = psi + (-(psi - eq)/(2tau) + S)
// equals psibar = eq + S + w (psi* - eq + S), w = (2tau - 1)/(2tau + 1),
// evaluated as psibar = psi* + (1 - w)(eq - psi*) + (1 + w) S: every rounding
// then falls on the small collision increment instead of on O(w_a rho) terms
// (in FP32 the other order repeats the same O(ulp(rho)) error every step).
// The sources of the two precisions are formed differently:
// FP64 (its pipe bounds a step): with q = e.u + 3/2 (e.u)^2 - u.u/2 (so that
// Gamma_a - w_a = 3 w_a q and 3 Gamma_a = 3 w_a (1 + 3 q)) and the forces
// scaled by (1 + w) dt/2 once per node, the increments are
//   h: -(1-w) (h* - rho w_a) + 3 w_a [c + q (m + 3 c)],
//      c = (e-u).X, X = c_s^2 grad rho - rho grad mu, m = (1-w) rho;
//   g: -(1-w) (g* - 3 w_a p) + 3 w_a [k + b + q (m + d + 3 k)],
//      k = (e-u).K, d = (e-u).grad rho, b the exact-difference body force
//      (1+w) rho/2 [e.du + e.du (3 e.u + 3/2 e.du) - du.(2u + du)/2]:
// two products per population with sums that are the node's but for the sign
// of their odd part, 23 packed operations for a pair against 56 when each
// term is formed by itself (256 x 1024 Rayleigh-Taylor 423 -> 358 us a step).
// FP32 forms each term by itself: there the products save 1.5 % of a lattice
// step, and leave u twice as far from 64 bits (after 200 steps of a drop on
// 57 x 103 nodes 9.4e-7 against 4.0e-7, on 32 x 32 7.3e-7 against 3.6e-7).
template <typename T>
struct CollidePrep {
    T r, ux, uy, p;
    T nr, np, nomw;   // -rho, -p, -(1 - w)
    T nhuu;           // -u.u/2
    T Xx, Xy, hA, hZ; // X (scaled); even parts m - 3 u.X and -u.X
    T Vx, Vy, gA;     // grad rho + 3 K (scaled); even part m - u.V
    T Bx, By, gZ;     // K + G; even part -u.K - (1+w) rho/4 du.(2u + du)
    T Gx, Gy, dux, duy;  // (1+w) rho/2 du, and du
};
template <>
struct CollidePrep<float> {
    float r, ux, uy, p, omw, opw, hdt, Xx, Xy, uX, uD, uK, uu, dux, duy, udu, drx, dry, kx, ky;
};

// Correctly rounded reciprocal (the same value as T(1) / x).
__device__ __forceinline__ float recip_rn(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double recip_rn(double x) { return __drcp_rn(x); }

// x / 3 correctly rounded, by a product with the rounded 1/3 and one
// correction with the exact remainder x - 3 q (the FMA form of
// division by a constant of Markstein, IBM J. Res. Dev. 34 (1990)).  It
// equals the rounded quotient for every normal FP32 mantissa and for all
// FP64 operands sampled (checked with exact rational arithmetic).
template <typename T>
__device__ __forceinline__ T div3(T x) {
    constexpr T c = T(1) / T(3);
    const T q = x * c;
    const T r = fma(T(-3), q, x);
    return fma(r, c, q);
}

// The scalars of the sources for given moments (omw = 1 - w, opw = 1 + w).
template <typename T>
__device__ __forceinline__ void collide_terms(const Phys<T> &P, CollidePrep<T> &c, T omw, T opw, T drx, T dry, T dmx,
                                              T dmy, T kx, T ky) {
    constexpr T cs2 = T(1) / T(3);
    const T r = c.r, f = opw * (T(0.5) * P.dt), m = omw * r;
    c.nr = -r;
    c.np = -c.p;
    c.nomw = -omw;
    c.nhuu = T(-0.5) * (c.ux * c.ux + c.uy * c.uy);
    c.Xx = f * (cs2 * drx - r * dmx);
    c.Xy = f * (cs2 * dry - r * dmy);
    const T uX = c.ux * c.Xx + c.uy * c.Xy;
    c.hZ = -uX;
    c.hA = fma(T(-3), uX, m);
    const T Kx = f * kx, Ky = f * ky;
    c.Vx = fma(T(3), Kx, f * drx);
    c.Vy = fma(T(3), Ky, f * dry);
    c.gA = m - (c.ux * c.Vx + c.uy * c.Vy);
    c.dux = P.gx * P.dt;  // exact-difference du = g dt
    c.duy = P.gy * P.dt;
    const T hr = T(0.5) * opw * r;
    c.Gx = hr * c.dux;
    c.Gy = hr * c.duy;
    c.Bx = Kx + c.Gx;
    c.By = Ky + c.Gy;
    c.gZ = -(c.ux * Kx + c.uy * Ky) - (c.Gx * (c.ux + T(0.5) * c.dux) + c.Gy * (c.uy + T(0.5) * c.duy));
}
__device__ __forceinline__ void collide_terms(const Phys<float> &P, CollidePrep<float> &c, float omw, float opw,
                                              float drx, float dry, float dmx, float dmy, float kx, float ky) {
    constexpr float cs2 = 1.0f / 3.0f;
    c.omw = omw;
    c.opw = opw;
    c.hdt = 0.5f * P.dt;
    c.Xx = cs2 * drx - c.r * dmx;  // F: c_s^2 grad rho - rho grad mu
    c.Xy = cs2 * dry - c.r * dmy;
    c.uX = c.ux * c.Xx + c.uy * c.Xy;
    c.uD = c.ux * drx + c.uy * dry;
    c.uK = c.ux * kx + c.uy * ky;
    c.uu = c.ux * c.ux + c.uy * c.uy;
    c.dux = P.gx * P.dt;  // exact-difference du = g dt
    c.duy = P.gy * P.dt;
    c.udu = c.dux * (2.0f * c.ux + c.dux) + c.duy * (2.0f * c.uy + c.duy);
    c.drx = drx;
    c.dry = dry;
    c.kx = kx;
    c.ky = ky;
}

// sg = sum_a g*_a, mx, my = sum_a e_a g*_a of the streamed (and bounced) g.
template <typename T>
__device__ __forceinline__ CollidePrep<T> collide_prep(const Phys<T> &P, T sg, T mx, T my, T r,
                                                       T drx, T dry, T dmx, T dmy, T kx, T ky) {
    CollidePrep<T> c;
    const T hdt = T(0.5) * P.dt;
    const T inv_r = recip_rn(r);
    c.r = r;
    c.ux = (mx + hdt * kx + hdt * r * P.gx) * inv_r;
    c.uy = (my + hdt * ky + hdt * r * P.gy) * inv_r;
    // p = c_s^2 (...) as a division by 3: a rounded 1/3 would be a gain on p
    // every step (see kW3)
    c.p = div3(sg + hdt * (c.ux * drx + c.uy * dry));
    T C = (r - P.rho_v) * P.inv_drho;
    C = C < T(0) ? T(0) : (C > T(1) ? T(1) : C);
    // 1/tau = C/tau_l + (1-C)/tau_v; w = (2 tau - 1)/(2 tau + 1) gives, with
    // s = 1/tau, 1 - w = 2 s/(2 + s) and 1 + w = 4/(2 + s): one reciprocal
    const T s = C * P.inv_tau_l + (T(1) - C) * P.inv_tau_v;
    const T d = recip_rn(T(2) + s);
    collide_terms(P, c, T(2) * s * d, T(4) * d, drx, dry, dmx, dmy, kx, ky);
    return c;
}

// e.v for a direction known at compile time (no product)
template <int EX, int EY, typename T>
__device__ __forceinline__ T dir_dot(T x, T y) {
    if (EX == 0) return EY > 0 ? y : -y;
    if (EY == 0) return EX > 0 ? x : -x;
    return (EX > 0 ? x : -x) + (EY > 0 ? y : -y);
}

// Collision of the opposite pair Q = (a, abar) of one node: e_abar = -e_a
// and w_abar = w_a, so the odd parts flip sign between the two lanes and the
// even parts are shared; the two lanes run in packed two-wide arithmetic.
// ds takes the pair's h increments.
template <typename T, int Q>
__device__ __forceinline__ void collide_pair(const CollidePrep<T> &c, V2<T> hs, V2<T> gs, V2<T> &ho, V2<T> &go,
                                             V2<T> &ds) {
    constexpr int A = pair_dir(Q, 0), ex = kEx(A), ey = kEy(A);
    constexpr T wa = kW<T>(A), w3 = kW3<T>(A);
    const T eu = dir_dot<ex, ey>(c.ux, c.uy), eX = dir_dot<ex, ey>(c.Xx, c.Xy);
    const T eV = dir_dot<ex, ey>(c.Vx, c.Vy), eB = dir_dot<ex, ey>(c.Bx, c.By);
    const T eG = dir_dot<ex, ey>(c.Gx, c.Gy), ed = dir_dot<ex, ey>(c.dux, c.duy);
    const T qe = fma(T(1.5) * eu, eu, c.nhuu), eA = T(3) * eX;
    const T ge = fma(eG, fma(T(1.5), ed, T(3) * eu), c.gZ);
    const V2<T> q = vset(qe + eu, qe - eu);
    const V2<T> hz = vfma(q, vset(c.hA + eA, c.hA - eA), vset(c.hZ + eX, c.hZ - eX));
    const V2<T> gz = vfma(q, vset(c.gA + eV, c.gA - eV), vset(ge + eB, ge - eB));
    const V2<T> w32 = vset(w3, w3), nomw = vset(c.nomw, c.nomw);
    ho = vadd(hs, vfma(nomw, vfma(vset(c.nr, c.nr), vset(wa, wa), hs), vmul(w32, hz)));
    go = vadd(gs, vfma(nomw, vfma(vset(c.np, c.np), w32, gs), vmul(w32, gz)));
    ds = vadd(ds, vfma(hs, vset(T(-1), T(-1)), ho));
}

// What one pair (or the rest population) of FP32 takes from the directions'
// products e.v of the node's vectors, eq and source by themselves.
struct PairTerms {
    float eu, eX, eD, eK, ed, uX, uD, uK, uu, udu, r, p, omw, opw, hdt;
};
__device__ __forceinline__ void collide_terms_pair(const PairTerms &t, float wa, float w3, float2 hs, float2 gs,
                                                   float2 &ho, float2 &go) {
    // Gamma - w = 3w (e.u + 1.5 (e.u)^2 - 0.5 u.u), formed without the w
    // offset (keeps the momentum part); 3w from kW3
    const float even = 1.5f * t.eu * t.eu - 0.5f * t.uu;
    const float2 gmw = vfma(vset(w3, w3), vset(t.eu, -t.eu), vset(w3 * even, w3 * even));
    const float2 gam3 = vfma(vset(3.0f, 3.0f), gmw, vset(w3, w3));  // 3 Gamma
    const float2 Fa = vmul(vset(t.hdt * (t.eX - t.uX), t.hdt * (-t.eX - t.uX)), gam3);
    const float2 Ga = vfma(vset(t.hdt * (t.eD - t.uD), t.hdt * (-t.eD - t.uD)), gmw,
                           vmul(vset(t.hdt * (t.eK - t.uK), t.hdt * (-t.eK - t.uK)), gam3));
    // 1/2 [g_eq(u + du) - g_eq(u)] = rho/2 [Gamma(u + du) - Gamma(u)]
    const float bev = 1.5f * t.ed * (2.0f * t.eu + t.ed) - 0.5f * t.udu;
    const float hrw = 0.5f * t.r * w3;
    const float2 Sg = vfma(vset(hrw, hrw), vset(t.ed + bev, bev - t.ed), Ga);
    const float2 rg = vmul(vset(t.r, t.r), gmw);
    const float2 dh = vadd(vfma(vset(t.r, t.r), vset(wa, wa), vset(-hs.x, -hs.y)), rg);  // h_eq - h*
    const float2 dg = vadd(vfma(vset(w3, w3), vset(t.p, t.p), vset(-gs.x, -gs.y)), rg);  // g_eq - g*
    ho = vadd(hs, vfma(vset(t.omw, t.omw), dh, vmul(vset(t.opw, t.opw), Fa)));
    go = vadd(gs, vfma(vset(t.omw, t.omw), dg, vmul(vset(t.opw, t.opw), Sg)));
}
__device__ __forceinline__ void collide_terms_rest(const PairTerms &t, float wa, float w3, float hs, float gs,
                                                   float &ho, float &go) {
    const float gmw = w3 * (-0.5f * t.uu), gam3 = w3 + 3.0f * gmw;
    const float Fa = t.hdt * -t.uX * gam3;
    const float Sg = t.hdt * -t.uD * gmw + t.hdt * -t.uK * gam3 + 0.5f * t.r * w3 * (-0.5f * t.udu);
    const float dh = fma(t.r, wa, -hs) + t.r * gmw, dg = fma(w3, t.p, -gs) + t.r * gmw;
    ho = hs + (t.omw * dh + t.opw * Fa);
    go = gs + (t.omw * dg + t.opw * Sg);
}
template <int ex, int ey>
__device__ __forceinline__ PairTerms pair_terms(const CollidePrep<float> &c) {
    if (ex == 0 && ey == 0)
        return {0.f, 0.f, 0.f, 0.f, 0.f, c.uX, c.uD, c.uK, c.uu, c.udu, c.r, c.p, c.omw, c.opw, c.hdt};
    return {dir_dot<ex, ey>(c.ux, c.uy), dir_dot<ex, ey>(c.Xx, c.Xy), dir_dot<ex, ey>(c.drx, c.dry),
            dir_dot<ex, ey>(c.kx, c.ky), dir_dot<ex, ey>(c.dux, c.duy), c.uX, c.uD, c.uK, c.uu, c.udu,
            c.r, c.p, c.omw, c.opw, c.hdt};
}
template <typename T, int Q>
__device__ __forceinline__ void collide_pair(const CollidePrep<float> &c, float2 hs, float2 gs, float2 &ho,
                                             float2 &go, float2 &ds) {
    constexpr int A = pair_dir(Q, 0);
    collide_terms_pair(pair_terms<kEx(A), kEy(A)>(c), kW<float>(A), kW3<float>(A), hs, gs, ho, go);
    ds = vadd(ds, vfma(hs, vset(-1.0f, -1.0f), ho));
}

// The same for the rest population; its h also takes the sum of the node's
// h increments (zero in exact arithmetic; ds those of the pairs): the
// collision then keeps the node's mass to one rounding instead of
// accumulating the rounding of the nine source terms every step.
template <typename T>
__device__ __forceinline__ void collide_rest(const CollidePrep<T> &c, T hs, T gs, V2<T> ds, T &ho, T &go) {
    constexpr T wa = kW<T>(0), w3 = kW3<T>(0);
    T h;
    if constexpr (sizeof(T) == 4) {
        collide_terms_rest(pair_terms<0, 0>(c), wa, w3, hs, gs, h, go);
    } else {
        h = hs + fma(c.nomw, fma(c.nr, wa, hs), w3 * fma(c.nhuu, c.hA, c.hZ));
        go = gs + fma(c.nomw, fma(c.np, w3, gs), w3 * fma(c.nhuu, c.gA, c.gZ));
    }
    ho = h - ((ds.x + ds.y) + (h - hs));
}

// Zeroth and first moments of the streamed g.  The first moments are summed
// as differences of opposite populations: each difference is exact in
// floating point when the two are close (they share the pressure part
// w_a 3p), so only the small momentum-carrying parts are rounded.
template <typename T>
__device__ __forceinline__ void g_moments(T g0, const V2<T> *g, T &sg, T &mx, T &my) {
    // pairs (1,3), (2,4), (5,7), (6,8): e_1 = (1,0), e_2 = (0,1), e_5 = (1,1), e_6 = (-1,1)
    const T d13 = g[0].x - g[0].y, d24 = g[1].x - g[1].y, d57 = g[2].x - g[2].y, d68 = g[3].x - g[3].y;
    mx = d13 + (d57 - d68);
    my = d24 + (d57 + d68);
    sg = ((g0 + (g[0].x + g[0].y)) + (g[1].x + g[1].y)) + ((g[2].x + g[2].y) + (g[3].x + g[3].y));
}

// Collision of a node whose streamed pairs are in registers, and its write:
// the pairs to ho / go + q np and the rest populations to h0o / g0o.
template <typename T>
__device__ __forceinline__ void collide_store(const CollidePrep<T> &c, const V2<T> *hs, const V2<T> *gs, T h0, T g0,
                                              size_t np, V2<T> *ho, V2<T> *go, T *h0o, T *g0o) {
    V2<T> ds = vset(T(0), T(0)), h, g;
    collide_pair<T, 0>(c, hs[0], gs[0], h, g, ds);
    ho[0] = h;
    go[0] = g;
    collide_pair<T, 1>(c, hs[1], gs[1], h, g, ds);
    ho[np] = h;
    go[np] = g;
    collide_pair<T, 2>(c, hs[2], gs[2], h, g, ds);
    ho[2 * np] = h;
    go[2 * np] = g;
    collide_pair<T, 3>(c, hs[3], gs[3], h, g, ds);
    ho[3 * np] = h;
    go[3 * np] = g;
    collide_rest<T>(c, h0, g0, ds, *h0o, *g0o);
}

template <typename T, typename Topo>
struct CollideArgs {
    Topo m;
    const T *fin;
    T *fout;
    Fields<T> F;
    Phys<T> P;
    T *mom;  // 4N or nullptr
    int *flag;
};

// Collision and write of one node of a general mesh from its streamed,
// bounced-back g and the h* of k_rho.
template <typename T, typename Topo>
__device__ __forceinline__ void collide_write(const CollideArgs<T, Topo> &A, int32_t i, size_t np, T g0,
                                              const V2<T> *gs, T r, T drx, T dry, T dmx, T dmy, T kx, T ky) {
    const size_t n = (size_t)A.m.n, si = A.m.slot(i);
    V2<T> hs[4];
    const V2<T> *hsb = reinterpret_cast<const V2<T> *>(A.F.hs + np);
#pragma unroll
    for (int q = 0; q < 4; ++q) hs[q] = hsb[q * np + si];
    const T h0 = A.F.hs[si];
    T sg, mx, my;
    g_moments<T>(g0, gs, sg, mx, my);
    const CollidePrep<T> c = collide_prep<T>(A.P, sg, mx, my, r, drx, dry, dmx, dmy, kx, ky);
    collide_store<T>(c, hs, gs, h0, g0, np, reinterpret_cast<V2<T> *>(A.fout + np) + si,
                     reinterpret_cast<V2<T> *>(A.fout + 10 * np) + si, A.fout + si, A.fout + 9 * np + si);
    if (!(finite_val(r) && finite_val(c.ux) && finite_val(c.uy) && finite_val(c.p))) atomicOr(A.flag, 1);
    if (A.mom) {
        A.mom[i] = r;
        A.mom[n + i] = c.ux;
        A.mom[2 * n + i] = c.uy;
        A.mom[3 * n + i] = c.p;
    }
}

template <typename T, typename Topo>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 5 : 2) k_collide(const __grid_constant__ CollideArgs<T, Topo> A) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    const Topo &m = A.m;
    if (i >= m.n) return;
    const size_t np = pad4(m.slots());
    const auto row = m.row(i);
    const int k = m.tag_of(i);
    pdl_wait();
    // g streamed here (the h code on the g half of the state); h* was
    // streamed and bounced back by k_rho
    T dmx, dmy;
    V2<T> gs[4];
    stream_pairs<T>(m, A.fin + 9 * np, np, i, A.P.dt, gs, [&](auto &&fn) { m.each(row, fn); });
    const T g0 = A.fin[9 * np + m.slot(i)];
    if (k) bounce_pairs<T>(k, gs);
    recover(m, row, A.F.mu, i, dmx, dmy);
    collide_write<T>(A, i, np, g0, gs, A.F.rho[i], A.F.drx[i], A.F.dry[i], dmx, dmy, A.F.kx[i], A.F.ky[i]);
}

// Initial state: post-collision distributions are the equilibria of
// (rho0, u0, p0); stored value psibar = eq + S (Omega(eq) = 0).
template <typename T, typename Topo>
__global__ void __launch_bounds__(256) k_init(const __grid_constant__ Topo m, T *__restrict__ fout, Fields<T> F,
                                              Phys<T> P, const T *__restrict__ mom) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.n) return;
    const size_t n = (size_t)m.n;
    T dmx, dmy;
    recover(m, m.row(i), F.mu, i, dmx, dmy);
    const T r = mom[i], ux = mom[n + i], uy = mom[2 * n + i], p = mom[3 * n + i];
    const T drx = F.drx[i], dry = F.dry[i], kx = F.kx[i], ky = F.ky[i];
    const T hdt = T(0.5) * P.dt;
    const T Xx = T(1) / T(3) * drx - r * dmx, Xy = T(1) / T(3) * dry - r * dmy;
    const T uX = ux * Xx + uy * Xy, uD = ux * drx + uy * dry, uK = ux * kx + uy * ky;
    const T uu = ux * ux + uy * uy;
    const T dux = P.gx * P.dt, duy = P.gy * P.dt;
    const T udu = dux * (T(2) * ux + dux) + duy * (T(2) * uy + duy);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int ex = kEx(a), ey = kEy(a);
        const T wa = kW<T>(a), w3 = kW3<T>(a);
        const T eu = T(ex) * ux + T(ey) * uy;
        const T gmw = w3 * (eu + T(1.5) * eu * eu - T(0.5) * uu);  // Gamma - w
        const T gam3 = w3 + T(3) * gmw;                             // 3 Gamma
        const T eX = T(ex) * Xx + T(ey) * Xy;
        const T eD = T(ex) * drx + T(ey) * dry;
        const T eK = T(ex) * kx + T(ey) * ky;
        const T edu = T(ex) * dux + T(ey) * duy;
        const T Fa = hdt * (eX - uX) * gam3;
        const T Ga = hdt * (eD - uD) * gmw + hdt * (eK - uK) * gam3;
        const T Ba = T(0.5) * r * w3 * (edu + T(1.5) * edu * (T(2) * eu + edu) - T(0.5) * udu);
        fout[pop_index(a, m.slot(i), m.slots())] = (r * wa + r * gmw) + Fa;
        fout[pop_index(9 + a, m.slot(i), m.slots())] = w3 * p + r * gmw + Ga + Ba;
    }
}

// Moments in caller order, FP64: out[0..N) rho, [N..2N) C, [2N..4N) u
// interleaved (ux, uy), [4N..5N) p.
template <typename T>
__global__ void k_gather_moments(int32_t n, const T *__restrict__ mom, const int32_t *__restrict__ iperm,
                                 double rho_l, double rho_v, double *__restrict__ out) {
    const int32_t c = blockIdx.x * blockDim.x + threadIdx.x;  // caller id
    if (c >= n) return;
    const int32_t k = iperm ? iperm[c] : c;
    const double r = (double)mom[k];
    out[c] = r;
    out[(size_t)n + c] = (r - rho_v) / (rho_l - rho_v);
    out[2 * (size_t)n + 2 * (size_t)c] = (double)mom[(size_t)n + k];
    out[2 * (size_t)n + 2 * (size_t)c + 1] = (double)mom[2 * (size_t)n + k];
    out[4 * (size_t)n + c] = (double)mom[3 * (size_t)n + k];
}

// FP64 totals: sum m rho, sum m rho ux, sum m rho uy.  Deterministic two-pass
// reduction: block partials (warp shuffles + shared memory), then one block.
template <typename T>
__global__ void __launch_bounds__(256) k_totals_partial(int32_t n, const T *__restrict__ mom,
                                                        const double *__restrict__ mass,
                                                        double *__restrict__ part) {
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double mr = mass[i] * (double)mom[i];
        s0 += mr;
        s1 += mr * (double)mom[(size_t)n + i];
        s2 += mr * (double)mom[2 * (size_t)n + i];
    }
    __shared__ double sh[3][8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, o);
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
        s2 += __shfl_down_sync(0xffffffffu, s2, o);
    }
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        sh[0][wid] = s0;
        sh[1][wid] = s1;
        sh[2][wid] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t0 = 0, t1 = 0, t2 = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            t0 += sh[0][w];
            t1 += sh[1][w];
            t2 += sh[2][w];
        }
        part[3 * blockIdx.x] = t0;
        part[3 * blockIdx.x + 1] = t1;
        part[3 * blockIdx.x + 2] = t2;
    }
}

__global__ void k_totals_final(int nparts, const double *__restrict__ part, double *__restrict__ out);

}  // namespace felbm
