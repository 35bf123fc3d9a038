// C ABI on tetrahedral meshes (D3Q19; kind 2 general CSR, kind 3 Kuhn
// lattice): mesh creation and the per-state work the common entry points of
// felbm_api.cu hand over here.
#include <algorithm>
#include <cmath>
#include <new>
#include <type_traits>
#include <vector>

#include "felbm_internal.h"
#include "felbm_kernels.cuh"
#include "felbm_kernels3.cuh"

namespace felbm {

static inline unsigned nblocks3(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// Storage index of population a (D3Q19 order) of node i: rest at [0, S),
// pair q = (2q+1, 2q+2) at Np + 2 Np q + 2 i + slot; g from 19 Np.
static size_t pop_index3(int a, size_t i, size_t n) {
    const size_t np = pad4(n);
    const size_t base = a < 19 ? 0 : 19 * np;
    const int d = a % 19;
    if (d == 0) return base + i;
    const int q = (d - 1) / 2, slot = (d - 1) % 2;
    return base + np + 2 * np * (size_t)q + 2 * i + (size_t)slot;
}

template <typename T>
static DevELL3<T> dev_ell3(const felbm_mesh *m) {
    DevELL3<T> d;
    d.n = (int32_t)m->n_nodes;
    d.sbase = m->d_sbase;
    void *const *e = m->d_ell[sizeof(T) == 8];
    d.a = reinterpret_cast<const Ell4<T> *>(e[0]);
    d.b = reinterpret_cast<const Ell4<T> *>(e[1]);
    d.c = reinterpret_cast<const Ell2<T> *>(e[2]);
    d.tag = m->d_tag;
    return d;
}

// The entries of DevELL3<T> from the assembled rows, on the device.
template <typename T>
static cudaError_t hold_ell3(felbm_mesh *m) {
    const HostCSR3 &H = m->host3;
    void **d = m->d_ell[sizeof(T) == 8];
    const std::lock_guard<std::mutex> guard(m->lock);
    if (d[0] && d[1] && d[2]) return cudaSuccess;
    const std::vector<int32_t> sb = ell_slices(H.n, H.rowptr);
    const size_t entries = (size_t)sb.back() * 32, nnz = H.col.size();
    const double *cf = H.coef.data();
    std::vector<Ell4<T>> a(entries), b(entries);
    std::vector<T> c(2 * entries, T(0));
    for (size_t s = 0; s + 1 < sb.size(); ++s)
        for (int32_t k = 0; k < sb[s + 1] - sb[s]; ++k)
            for (int32_t l = 0; l < 32; ++l) {
                const size_t p = ((size_t)sb[s] + k) * 32 + l;
                const int64_t i = std::min<int64_t>(32 * (int64_t)s + l, H.n - 1);
                const int64_t q = (int64_t)H.rowptr[i] + k;
                if (q < H.rowptr[i + 1]) {
                    a[p] = {(T)cf[q], (T)cf[nnz + q], (T)cf[2 * nnz + q], ell_id<T>(H.col[q])};
                    b[p] = {(T)cf[3 * nnz + q], (T)cf[4 * nnz + q], (T)cf[5 * nnz + q], (T)cf[6 * nnz + q]};
                    c[2 * p] = (T)cf[7 * nnz + q];
                    c[2 * p + 1] = (T)cf[8 * nnz + q];
                } else {
                    a[p] = {T(0), T(0), T(0), ell_id<T>((int32_t)i)};
                    b[p] = {T(0), T(0), T(0), T(0)};
                }
            }
    cudaError_t e = mesh_hold(m, &d[0], a.data(), entries * sizeof(Ell4<T>));
    if (e == cudaSuccess) e = mesh_hold(m, &d[1], b.data(), entries * sizeof(Ell4<T>));
    if (e == cudaSuccess) e = mesh_hold(m, &d[2], c.data(), 2 * entries * sizeof(T));
    return e;
}

// Whether the interior recovery weights of a lattice are those of the full
// split that the integer-weight passes assume, to 1e-12 of their size.
static bool kuhn_uniform(const Lattice3Info &L) {
    const double s12 = L.c[0][0][0] / kuhn_w(0, 0);
    for (int o = 0; o < 14; ++o)
        for (int c = 0; c < 3; ++c) {
            const double w = (o % 2 ? -1.0 : 1.0) * kuhn_w(o / 2, c) * s12;
            if (!(std::fabs(L.c[0][o][c] - w) <= 1e-12 * std::fabs(3.0 * s12))) return false;
        }
    return true;
}

template <typename T>
static DevLattice3<T> dev_lat3(const felbm_mesh *m, double dt) {
    const Lattice3Info &L = m->linfo3;
    DevLattice3<T> d;
    d.n = (int32_t)m->n_nodes;
    d.nx = L.nx;
    d.ny = L.ny;
    d.nz = L.nz;
    d.walls = L.walls ? 1 : 0;
    const double hdt = 0.5 * dt;
    for (int k = 0; k < 3; ++k)
        for (int o = 0; o < 14; ++o) {
            const double *cf = L.c[k][o];
            for (int q = 0; q < 9; ++q) {
                const int a = 2 * q + 1;
                const double ex = e3x(a), ey = e3y(a), ez = e3z(a);
                const double odd = ex * cf[0] + ey * cf[1] + ez * cf[2];
                const double even = hdt * ((ex * ex * cf[3] + ey * ey * cf[6] + ez * ez * cf[8]) +
                                           2.0 * (ex * ey * cf[4] + ex * ez * cf[5] + ey * ez * cf[7]));
                d.k.pc[k][o][q].x = (T)(even + odd);
                d.k.pc[k][o][q].y = (T)(even - odd);
            }
            for (int c = 0; c < 3; ++c) d.k.a[k][o][c] = (T)cf[c];
        }
    d.k.s12 = (T)(L.c[0][0][0] / kuhn_w(0, 0));
    d.tables = !kuhn_uniform(L) ? 2 : d.walls;
    return d;
}

template <typename T>
static Phys3<T> phys3_of(const felbm_params &p) {
    const double dd = p.rho_l - p.rho_v;
    Phys3<T> P;
    P.rho_l = (T)p.rho_l;
    P.rho_v = (T)p.rho_v;
    P.beta = (T)(12.0 * p.sigma / (p.xi * dd * dd * dd * dd));
    P.kappa = (T)(1.5 * p.xi * p.sigma / (dd * dd));
    P.inv_tau_l = (T)(1.0 / p.tau_l);
    P.inv_tau_v = (T)(1.0 / p.tau_v);
    P.dt = (T)p.dt;
    for (int k = 0; k < 3; ++k) P.g[k] = (T)p.gravity[k];
    P.inv_drho = (T)(1.0 / dd);
    return P;
}

// Scratch layout (19 Np + 9 N): streamed h*, grad rho (4 N interleaved,
// 16-byte aligned since Np is a multiple of 4), rho, mu, K (3).
template <typename T>
static Fields3<T> fields3_of(felbm_state *s) {
    const size_t n = (size_t)s->mesh->n_nodes;
    Fields3<T> F;
    F.hs = reinterpret_cast<T *>(s->scratch);
    F.dr4 = F.hs + 19 * pad4(n);
    T *b = F.dr4 + 4 * n;
    F.rho = b;
    F.mu = b + n;
    for (int k = 0; k < 3; ++k) F.k[k] = b + (2 + k) * n;
    return F;
}

// Forms of the passes over a lattice (us a launch or step, GB300):
//   streaming of h split over three threads a node up to 2^16 nodes (FP32
//   step of 32^3 12.1 us split, 13.4 with a thread per node; 40^3 17.5 and
//   18.0; 48^3 26.0 and 25.2; FP64 pass 24^3 27 and 47, 36^3 58 and 87, 48^3
//   130 and 127), a thread per node above;
//   the collision likewise in FP64 (14^3 30 and 46, 36^3 117 and 125, 48^3
//   265 and 244); in FP32 always a thread per node (16^3 9.9 us a step
//   against 9.2 split, 24^3 11.0 and 11.6, 64^3 42.9 and 57);
//   the scalar passes with two nodes a column from 2^18 nodes on in FP32
//   (96^3 26.4 us for the two, 30.2 with one; 64^3 equal), else one.
constexpr int64_t kSplitMax = 1 << 16, kColumnMin = 1 << 18;

//   columns packed into blocks where a plane fills at most half a block and
//   there are layers of columns for more than one block an SM (3 x 3 x 1000
//   FP32 12.3 -> 11.0 us, FP64 66 -> 59; 12^3 without).
constexpr int kColBlock = 256, kPackPlane = kColBlock / 2, kPackLayers = 152;

// fn(nodes a column, packed, blocks)
template <typename T, typename Fn>
static void with_columns(const DevLattice3<T> &d, Fn &&fn) {
    auto run = [&](auto Z) {
        const int64_t plane = (int64_t)d.nx * d.ny, layers = nblocks3(d.nz, decltype(Z)::value);
        if (plane <= kPackPlane && layers > kPackLayers)
            fn(Z, std::true_type(), nblocks3(plane * layers, kColBlock));
        else
            fn(Z, std::false_type(), (unsigned)(nblocks3(plane, kColBlock) * layers));
    };
    if constexpr (sizeof(T) == 4) {
        if (d.n >= kColumnMin) return run(std::integral_constant<int, 2>());
    }
    run(std::integral_constant<int, 1>());
}

// grad rho, then lap rho, K and mu, from F.rho.
template <typename T, typename Topo>
static void chain3(felbm_state *s, const Topo &d, const Fields3<T> &F, const Phys3<T> &P) {
    const felbm_mesh *m = s->mesh;
    int sl = prof_begin(s, 1);
    if constexpr (Topo::kLattice) {
        with_columns<T>(d, [&](auto Z, auto Pack, unsigned blocks) {
            launch_pdl(k_grad3_col<T, decltype(Z)::value, decltype(Pack)::value>, blocks, kColBlock, 0, m->stream, d, F);
        });
    } else {
        launch_pdl(k_grad3_rows<T>, nblocks3(m->n_nodes, kSplitNodes), kSplitBlock, 0, m->stream, d, F);
    }
    prof_end(s, sl);
    sl = prof_begin(s, 2);
    if constexpr (Topo::kLattice) {
        with_columns<T>(d, [&](auto Z, auto Pack, unsigned blocks) {
            launch_pdl(k_mu3_col<T, decltype(Z)::value, decltype(Pack)::value>, blocks, kColBlock, 0, m->stream, d, F, P);
        });
    } else {
        launch_pdl(k_mu3_rows<T>, nblocks3(m->n_nodes, kSplitNodes), kSplitBlock, 0, m->stream, d, F, P);
    }
    prof_end(s, sl);
}

// Calls fn(topology) with the device view of the state's mesh.
template <typename T, typename Fn>
static void with_topo(felbm_state *s, Fn &&fn) {
    if (s->mesh->kind == 3)
        fn(dev_lat3<T>(s->mesh, s->params.dt));
    else
        fn(dev_ell3<T>(s->mesh));
}

template <typename T>
static void init3(felbm_state *s) {
    with_topo<T>(s, [&](const auto &d) {
        using Topo = std::decay_t<decltype(d)>;
        const felbm_mesh *m = s->mesh;
        const Fields3<T> F = fields3_of<T>(s);
        const Phys3<T> P = phys3_of<T>(s->params);
        cudaMemcpyAsync(F.rho, s->mom, (size_t)m->n_nodes * sizeof(T), cudaMemcpyDeviceToDevice, m->stream);
        chain3<T>(s, d, F, P);
        k_init3<T, Topo><<<nblocks3(m->n_nodes, 128), 128, 0, m->stream>>>(
            d, reinterpret_cast<T *>(s->f[s->cur]), F, P, reinterpret_cast<const T *>(s->mom));
    });
}

template <typename T, typename Topo>
static void step3(felbm_state *s, const Topo &d, const Fields3<T> &F, const Phys3<T> &P, bool write_mom) {
    const felbm_mesh *m = s->mesh;
    const T *fin = reinterpret_cast<const T *>(s->f[s->cur]);
    T *fout = reinterpret_cast<T *>(s->f[s->cur ^ 1]);
    const bool split = !Topo::kLattice || d.n <= kSplitMax;
    int sl = prof_begin(s, 0);
    if (split)
        launch_pdl(k_rho3_split<T, Topo>, nblocks3(m->n_nodes, kSplitNodes), kSplitBlock, 0, m->stream, d, fin, P.dt,
                   F.rho, F.hs);
    else if constexpr (Topo::kLattice)
        launch_pdl(k_rho3_node<T>, nblocks3(m->n_nodes, 256), 256, 0, m->stream, d, fin, P.dt, F.rho, F.hs);
    prof_end(s, sl);
    chain3<T>(s, d, F, P);
    Collide3Args<T, Topo> A;
    A.m = d;
    A.fin = fin;
    A.fout = fout;
    A.F = F;
    A.P = P;
    A.mom = write_mom ? reinterpret_cast<T *>(s->mom) : nullptr;
    A.flag = s->d_flag;
    sl = prof_begin(s, 3);
    if constexpr (Topo::kLattice) {
        if (sizeof(T) == 4 || !split)
            launch_pdl(d.tables < 2 ? k_collide3_node<T, true> : k_collide3_node<T, false>, nblocks3(m->n_nodes, 128), 128, 0,
                       m->stream, A);
        else if constexpr (sizeof(T) == 8)
            launch_pdl(k_collide3_split<T, Topo>, nblocks3(m->n_nodes, kSplitNodes), kSplitBlock, 0, m->stream, A);
    } else {
        launch_pdl(k_collide3_split<T, Topo>, nblocks3(m->n_nodes, kSplitNodes), kSplitBlock, 0, m->stream, A);
    }
    prof_end(s, sl);
    s->cur ^= 1;
}

template <typename T>
static void steps3_t(felbm_state *s, int64_t n) {
    with_topo<T>(s, [&](const auto &d) {
        const Fields3<T> F = fields3_of<T>(s);
        const Phys3<T> P = phys3_of<T>(s->params);
        for (int64_t k = 0; k < n; ++k) step3<T>(s, d, F, P, k == n - 1);
    });
}

void steps3(felbm_state *s, int64_t n) {
    if (s->esize == 8)
        steps3_t<double>(s, n);
    else
        steps3_t<float>(s, n);
}

int state_init3(const felbm_mesh *mesh, const felbm_params *params, const double *rho0,
                const double *u0, const double *p0, felbm_state **out) {
    if (params->flags & FELBM_PARAM_LAP_FP64) return FELBM_ERR_UNSUPPORTED;
    const size_t N = (size_t)mesh->n_nodes;
    for (size_t i = 0; i < N; ++i)
        if (!(rho0[i] > 0.0) || !std::isfinite(rho0[i])) return FELBM_ERR_INVALID_ARG;
    felbm_state *s = new (std::nothrow) felbm_state();
    if (!s) return FELBM_ERR_OOM;
    s->mesh = mesh;
    s->params = *params;
    s->precision = params->precision;
    s->esize = params->precision == FELBM_FP64 ? 8 : 4;
    const size_t es = s->esize;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(p, bytes);
    };
    alloc(&s->f[0], 38 * pad4(N) * es);
    alloc(&s->f[1], 38 * pad4(N) * es);
    alloc(&s->scratch, (19 * pad4(N) + 9 * N) * es);
    alloc(&s->mom, 5 * N * es);
    alloc((void **)&s->d_out, (6 * N + 4 * (kTotalsBlocks + 1)) * sizeof(double));
    alloc((void **)&s->d_flag, sizeof(int));
    if (e == cudaSuccess && mesh->kind == 2) {
        felbm_mesh *m = const_cast<felbm_mesh *>(mesh);
        try {
            e = es == 8 ? hold_ell3<double>(m) : hold_ell3<float>(m);
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    if (e != cudaSuccess) {
        const int rs = cuda_status(e);
        state_free(s);
        return rs;
    }
    // initial moments (rho, ux, uy, uz, p) in internal order and precision
    std::vector<unsigned char> hm(5 * N * es);
    for (size_t k = 0; k < N; ++k) {
        const size_t c = (size_t)mesh->host3.perm[k];
        const double v[5] = {rho0[c], u0 ? u0[3 * c] : 0.0, u0 ? u0[3 * c + 1] : 0.0,
                             u0 ? u0[3 * c + 2] : 0.0, p0 ? p0[c] : 0.0};
        for (int q = 0; q < 5; ++q) {
            if (!std::isfinite(v[q])) {
                state_free(s);
                return FELBM_ERR_INVALID_ARG;
            }
            if (es == 8)
                reinterpret_cast<double *>(hm.data())[q * N + k] = v[q];
            else
                reinterpret_cast<float *>(hm.data())[q * N + k] = (float)v[q];
        }
    }
    e = cudaMemcpyAsync(s->mom, hm.data(), hm.size(), cudaMemcpyHostToDevice, mesh->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_flag, 0, sizeof(int), mesh->stream);
    for (int c = 0; c < 2 && e == cudaSuccess; ++c)
        e = cudaMemsetAsync(s->f[c], 0, 38 * pad4(N) * es, mesh->stream);
    if (e == cudaSuccess) {
        if (es == 8)
            init3<double>(s);
        else
            init3<float>(s);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(mesh->stream);  // hm is a temporary
    if (e != cudaSuccess) {
        const int rs = cuda_status(e);
        state_free(s);
        return rs;
    }
    s->have_moments = true;
    *out = s;
    return FELBM_OK;
}

template <typename T>
static void launch_moments3(felbm_state *s) {
    const felbm_mesh *m = s->mesh;
    const int32_t n = (int32_t)m->n_nodes;
    k_gather_moments3<T><<<nblocks3(n, 256), 256, 0, m->stream>>>(
        n, reinterpret_cast<const T *>(s->mom), m->d_perm + n, s->params.rho_l, s->params.rho_v, s->d_out);
    double *part = s->d_out + 6 * (size_t)n;
    k_totals3_partial<T><<<kTotalsBlocks, 256, 0, m->stream>>>(n, reinterpret_cast<const T *>(s->mom),
                                                               m->d_mass, part);
    k_totals3_final<<<1, 32, 0, m->stream>>>(kTotalsBlocks, part, part + 4 * kTotalsBlocks);
}

int moments3(felbm_state *s, double *rho, double *C, double *u, double *p, double *totals) {
    const size_t N = (size_t)s->mesh->n_nodes;
    const cudaStream_t st = s->mesh->stream;
    if (s->esize == 8)
        launch_moments3<double>(s);
    else
        launch_moments3<float>(s);
    cudaError_t e = cudaGetLastError();
    const double *o = s->d_out;
    if (e == cudaSuccess && rho) e = cudaMemcpyAsync(rho, o, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && C) e = cudaMemcpyAsync(C, o + N, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && u) e = cudaMemcpyAsync(u, o + 2 * N, 3 * N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && p) e = cudaMemcpyAsync(p, o + 5 * N, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && totals)
        e = cudaMemcpyAsync(totals, o + 6 * N + 4 * kTotalsBlocks, 4 * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return cuda_status(e);
}

int export3(felbm_state *s, double *hbar, double *gbar) {
    const size_t N = (size_t)s->mesh->n_nodes, es = s->esize;
    std::vector<unsigned char> buf(38 * pad4(N) * es);
    cudaError_t e = cudaMemcpyAsync(buf.data(), s->f[s->cur], buf.size(), cudaMemcpyDeviceToHost,
                                    s->mesh->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->mesh->stream);
    if (e != cudaSuccess) return cuda_status(e);
    for (int a = 0; a < 38; ++a)
        for (size_t k = 0; k < N; ++k) {
            const size_t c = (size_t)s->mesh->host3.perm[k];
            const size_t q = pop_index3(a, k, N);
            const double v = es == 8 ? reinterpret_cast<double *>(buf.data())[q]
                                     : (double)reinterpret_cast<float *>(buf.data())[q];
            (a < 19 ? hbar : gbar)[(a % 19) * N + c] = v;
        }
    return FELBM_OK;
}

int import3(felbm_state *s, const double *hbar, const double *gbar) {
    const size_t N = (size_t)s->mesh->n_nodes, es = s->esize;
    std::vector<unsigned char> buf(38 * pad4(N) * es, 0);
    for (int a = 0; a < 38; ++a)
        for (size_t k = 0; k < N; ++k) {
            const size_t c = (size_t)s->mesh->host3.perm[k];
            const double v = (a < 19 ? hbar : gbar)[(a % 19) * N + c];
            if (!std::isfinite(v)) return FELBM_ERR_INVALID_ARG;
            const size_t q = pop_index3(a, k, N);
            if (es == 8)
                reinterpret_cast<double *>(buf.data())[q] = v;
            else
                reinterpret_cast<float *>(buf.data())[q] = (float)v;
        }
    cudaError_t e = cudaMemcpyAsync(s->f[s->cur], buf.data(), buf.size(), cudaMemcpyHostToDevice,
                                    s->mesh->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_flag, 0, sizeof(int), s->mesh->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->mesh->stream);
    if (e != cudaSuccess) return cuda_status(e);
    s->have_moments = false;
    return FELBM_OK;
}

FELBM_CHECK_READER(check_bits_api3)

}  // namespace felbm

using namespace felbm;

extern "C" int felbm_mesh_create_tet(const double *xyz, int64_t n_nodes, const int32_t *tet, int64_t n_tet,
                                     const double box[3], uint32_t flags, const uint8_t *node_tag,
                                     void *stream, felbm_mesh **out) {
    if (!xyz || !tet || !box || !out) return FELBM_ERR_INVALID_ARG;
    if (n_nodes < 4 || n_tet < 1 || n_nodes > 0x7fffffffLL || n_tet > 0x7fffffffLL / 4)
        return FELBM_ERR_INVALID_ARG;
    if (flags & ~(FELBM_PERIODIC_X | FELBM_PERIODIC_Y | FELBM_PERIODIC_Z | FELBM_MESH_GENERAL))
        return FELBM_ERR_INVALID_ARG;
    felbm_mesh *m = new (std::nothrow) felbm_mesh();
    if (!m) return FELBM_ERR_OOM;
    m->n_nodes = n_nodes;
    m->n_tri = n_tet;
    m->flags = flags;
    m->stream = reinterpret_cast<cudaStream_t>(stream);
    m->kind = 2;
    int st = FELBM_OK;
    try {
        st = build_csr3(xyz, n_nodes, tet, n_tet, box, flags, node_tag, m->host3);
    } catch (const std::bad_alloc &) {
        st = FELBM_ERR_OOM;
    }
    if (st != FELBM_OK) {
        delete m;
        return st;
    }
    HostCSR3 &H = m->host3;
    if (!(flags & FELBM_MESH_GENERAL)) detect_lattice3(xyz, n_nodes, box, flags, node_tag, H, m->linfo3);
    if (m->linfo3.ok) {
        // the lattice kernels take neighbours and coefficients from the node
        // position: natural order, no assembled arrays on the device
        m->kind = 3;
        std::vector<double> mass(H.n);
        for (int32_t c = 0; c < H.n; ++c) {
            mass[c] = H.mass[H.iperm[c]];
            H.perm[c] = H.iperm[c] = c;
        }
        H.mass.swap(mass);
        std::vector<int32_t>().swap(H.col);
        std::vector<double>().swap(H.coef);
        std::vector<uint8_t>().swap(H.tag);
    }
    const size_t N = (size_t)n_nodes;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) {
            e = cudaMalloc(p, bytes);
            if (e == cudaSuccess) m->device_bytes += (int64_t)bytes;
        }
    };
    const bool csr = m->kind == 2;
    alloc((void **)&m->d_mass, N * sizeof(double));
    alloc((void **)&m->d_perm, 2 * N * sizeof(int32_t));
    if (csr && !H.tag.empty()) alloc((void **)&m->d_tag, N);
    if (e == cudaSuccess) e = cudaMemcpy(m->d_mass, H.mass.data(), N * sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->d_perm, H.perm.data(), N * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(m->d_perm + N, H.iperm.data(), N * sizeof(int32_t), cudaMemcpyHostToDevice);
    if (csr) {
        try {
            const std::vector<int32_t> sb = ell_slices(H.n, H.rowptr);
            if (e == cudaSuccess)
                e = mesh_upload(m, (void **)&m->d_sbase, sb.data(), sb.size() * sizeof(int32_t));
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    if (e == cudaSuccess && m->d_tag) e = cudaMemcpy(m->d_tag, H.tag.data(), N, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        const int rs = cuda_status(e);
        mesh_free(m);
        return rs;
    }
    *out = m;
    return FELBM_OK;
}
