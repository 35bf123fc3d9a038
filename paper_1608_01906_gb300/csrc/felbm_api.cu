// C ABI of the FE-LBM library: handle management, uploads, launches.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "felbm_internal.h"
#include "felbm_kernels.cuh"
#include "felbm_lattice.cuh"
#include "felbm_latpass.cuh"
#include "felbm_patch.cuh"

using namespace felbm;

namespace felbm {

__global__ void k_totals_final(int nparts, const double *__restrict__ part, double *__restrict__ out) {
    // single warp, fixed order over lanes then shuffle tree: deterministic
    double s0 = 0, s1 = 0, s2 = 0;
    for (int k = threadIdx.x; k < nparts; k += 32) {
        s0 += part[3 * k];
        s1 += part[3 * k + 1];
        s2 += part[3 * k + 2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s0 += __shfl_down_sync(0xffffffffu, s0, o);
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
        s2 += __shfl_down_sync(0xffffffffu, s2, o);
    }
    if (threadIdx.x == 0) {
        out[0] = s0;
        out[1] = s1;
        out[2] = s2;
    }
}

int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return FELBM_OK;
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return FELBM_ERR_OOM;
    }
    return FELBM_ERR_CUDA;
}

#define FELBM_CK(x)                              \
    do {                                         \
        cudaError_t _e = (x);                    \
        if (_e != cudaSuccess) return cuda_status(_e); \
    } while (0)

// with_b false: for kernels that read no b_xx, b_xy (a stands in for them)
template <typename T>
static DevELL<T> dev_ell(const felbm_mesh *m, bool with_b = true) {
    DevELL<T> d;
    d.n = (int32_t)m->n_nodes;
    d.sbase = m->d_sbase;
    void *const *e = m->d_ell[sizeof(T) == 8];
    d.a = reinterpret_cast<const Ell2<T> *>(e[0]);
    d.b = reinterpret_cast<const Ell2<T> *>(e[with_b ? 1 : 0]);
    d.c = reinterpret_cast<const Ell2<T> *>(e[2]);
    d.deg = m->d_deg;
    d.tag = m->d_tag;
    return d;
}

std::vector<int32_t> ell_slices(int32_t n, const std::vector<int32_t> &rowptr) {
    std::vector<int32_t> sb((size_t)(n + 31) / 32 + 1, 0);
    for (size_t s = 0; s + 1 < sb.size(); ++s) {
        int32_t w = 0;
        for (int32_t i = (int32_t)(32 * s); i < std::min<int64_t>(n, 32 * (int64_t)(s + 1)); ++i)
            w = std::max(w, rowptr[i + 1] - rowptr[i]);
        sb[s + 1] = sb[s] + w;
    }
    return sb;
}

cudaError_t mesh_upload(felbm_mesh *m, void **d, const void *host, size_t bytes) {
    cudaError_t e = cudaMalloc(d, std::max<size_t>(bytes, 1));
    if (e != cudaSuccess) return e;
    m->device_bytes += (int64_t)bytes;
    return bytes ? cudaMemcpy(*d, host, bytes, cudaMemcpyHostToDevice) : cudaSuccess;
}

cudaError_t mesh_hold(felbm_mesh *m, void **d, const void *host, size_t bytes) {
    if (*d) return cudaSuccess;
    void *p = nullptr;
    cudaError_t e = cudaMalloc(&p, std::max<size_t>(bytes, 1));
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(p, host, bytes, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        cudaFree(p);
        return e;
    }
    *d = p;
    m->device_bytes += (int64_t)bytes;
    return cudaSuccess;
}

// The entries of DevELL<T> from the assembled rows, on the device; the b_xx,
// b_xy among them where wanted.
template <typename T>
static cudaError_t hold_ell(felbm_mesh *m, bool with_b) {
    const HostCSR &H = m->host;
    void **d = m->d_ell[sizeof(T) == 8];
    if (d[0] && d[2] && (d[1] || !with_b)) return cudaSuccess;
    const std::vector<int32_t> sb = ell_slices(H.n, H.rowptr);
    const size_t entries = (size_t)sb.back() * 32;
    std::vector<Ell2<T>> a(entries), b(entries), c(entries);
    for (size_t s = 0; s + 1 < sb.size(); ++s)
        for (int32_t k = 0; k < sb[s + 1] - sb[s]; ++k)
            for (int32_t l = 0; l < 32; ++l) {
                const size_t p = ((size_t)sb[s] + k) * 32 + l;
                const int64_t i = std::min<int64_t>(32 * (int64_t)s + l, H.n - 1);
                const int64_t q = (int64_t)H.rowptr[i] + k;
                if (q < H.rowptr[i + 1]) {
                    a[p] = {(T)H.ax[q], (T)H.ay[q]};
                    b[p] = {(T)H.bxx[q], (T)H.bxy[q]};
                    c[p] = {(T)H.byy[q], ell_id<T>(H.col[q])};
                } else {
                    a[p] = b[p] = {T(0), T(0)};
                    c[p] = {T(0), ell_id<T>((int32_t)i)};
                }
            }
    cudaError_t e = mesh_hold(m, &d[0], a.data(), entries * sizeof(Ell2<T>));
    if (e == cudaSuccess && with_b) e = mesh_hold(m, &d[1], b.data(), entries * sizeof(Ell2<T>));
    if (e == cudaSuccess) e = mesh_hold(m, &d[2], c.data(), entries * sizeof(Ell2<T>));
    return e;
}

template <typename T>
static Phys<T> phys_of(const felbm_params &p) {
    const double d = p.rho_l - p.rho_v;
    Phys<T> P;
    P.rho_l = (T)p.rho_l;
    P.rho_v = (T)p.rho_v;
    P.beta = (T)(12.0 * p.sigma / (p.xi * d * d * d * d));
    P.kappa = (T)(1.5 * p.xi * p.sigma / (d * d));
    P.inv_tau_l = (T)(1.0 / p.tau_l);
    P.inv_tau_v = (T)(1.0 / p.tau_v);
    P.dt = (T)p.dt;
    P.gx = (T)p.gravity[0];
    P.gy = (T)p.gravity[1];
    P.inv_drho = (T)(1.0 / (p.rho_l - p.rho_v));
    return P;
}

// Scratch: on general meshes the streamed h* (9 Np, population layout)
// first, then 6 N fields (rho, grad rho, mu, K).
static size_t hstar_elems(const felbm_mesh *m) { return m->kind == 0 ? 9 * pad4(pop_slots(m)) : 0; }

template <typename T>
static Fields<T> fields_of(felbm_state *s) {
    const size_t n = (size_t)s->mesh->n_nodes;
    T *base = reinterpret_cast<T *>(s->scratch);
    const size_t nh = hstar_elems(s->mesh);
    T *b = base + nh;
    Fields<T> F;
    F.hs = nh ? base : nullptr;
    F.rho = b;
    F.drx = b + n;
    F.dry = b + 2 * n;
    F.mu = b + 3 * n;
    F.kx = b + 4 * n;
    F.ky = b + 5 * n;
    return F;
}

static inline unsigned nblocks(int64_t n, int bs) { return (unsigned)((n + bs - 1) / bs); }

static constexpr size_t kProfMaxLaunches = 4096;

int prof_begin(felbm_state *s, int kind) {
    s->launches[kind]++;
    if (!s->prof_on || (s->prof_seen[kind]++ % s->prof_stride) != 0 || s->prof_used >= kProfMaxLaunches)
        return -1;
    const size_t slot = s->prof_used++;
    s->prof_kind[slot] = kind;
    cudaEventRecord(s->prof_ev[2 * slot], s->mesh->stream);
    return (int)slot;
}

void prof_end(felbm_state *s, int slot) {
    if (slot >= 0) cudaEventRecord(s->prof_ev[2 * slot + 1], s->mesh->stream);
}

template <typename T>
static DevLattice<T> dev_lattice(const felbm_mesh *m) {
    DevLattice<T> d;
    d.n = (int32_t)m->n_nodes;
    d.nx = m->sinfo.nx;
    d.ny = m->sinfo.ny;
    d.walls = m->sinfo.walls ? 1 : 0;
    d.pitch = m->sinfo.pitch;
    d.row0 = m->sinfo.row0;
    d.gny = m->sinfo.gny;
    for (int k = 0; k < 3; ++k)
        for (int o = 0; o < 6; ++o) {
            d.c[k][o][0] = (T)m->sinfo.a[k][o][0];
            d.c[k][o][1] = (T)m->sinfo.a[k][o][1];
            for (int q = 0; q < 3; ++q) d.c[k][o][2 + q] = (T)m->sinfo.b[k][o][q];
        }
    return d;
}

// Derivative chain shared by init and step: rho (already in F.rho) ->
// grad rho -> lap rho, K, mu.
// Threads per block of the general path's node kernels (one node per
// thread).
constexpr int kGenBlock = 128;

// Whether a general mesh's patches are all resident at once at two blocks
// per SM (152 SMs): its step is then bound by latency, and its kernels take
// more registers per thread.
constexpr int64_t kOneWave = 2 * 152 * kPatch;

// kappa in FP64 (the FP64 kappa lap rho term of FELBM_PARAM_LAP_FP64)
static double kappa64(const felbm_params &p) {
    const double d = p.rho_l - p.rho_v;
    return 1.5 * p.xi * p.sigma / (d * d);
}

static bool lap_fp64(const felbm_state *s) { return s->esize == 4 && (s->params.flags & FELBM_PARAM_LAP_FP64); }

// The mesh's operators with FP64 coefficients, for the FP64 Laplacian.
static DevELL<double> topo64(const felbm_mesh *m, const DevELL<float> &) { return dev_ell<double>(m, false); }
static DevLattice<double> topo64(const felbm_mesh *m, const DevLattice<float> &) { return dev_lattice<double>(m); }

template <typename T, typename Topo>
static void launch_chain(felbm_state *s, const Topo &d) {
    const felbm_mesh *m = s->mesh;
    const Fields<T> F = fields_of<T>(s);
    const Phys<T> P = phys_of<T>(s->params);
    const unsigned g = nblocks(m->n_nodes, kGenBlock);
    int sl = prof_begin(s, 1);
    launch_pdl(k_grad<T, Topo>, g, kGenBlock, 0, m->stream, d, F);
    prof_end(s, sl);
    sl = prof_begin(s, 2);
    if constexpr (sizeof(T) == 4) {
        if (lap_fp64(s)) {
            const auto d64 = topo64(m, d);
            launch_pdl(k_mu_lap64<std::decay_t<decltype(d64)>>, g, kGenBlock, 0, m->stream, d64, F, P, kappa64(s->params));
        } else {
            launch_pdl(k_mu<T, Topo>, g, kGenBlock, 0, m->stream, d, F, P);
        }
    } else {
        launch_pdl(k_mu<T, Topo>, g, kGenBlock, 0, m->stream, d, F, P);
    }
    prof_end(s, sl);
}

// The first launch of a general mesh's step: streamed h* and rho.
template <typename T, typename Topo>
static CollideArgs<T, Topo> step_rho(felbm_state *s, const Topo &d, bool write_mom) {
    const felbm_mesh *m = s->mesh;
    CollideArgs<T, Topo> A;
    A.m = d;
    A.fin = reinterpret_cast<const T *>(s->f[s->cur]);
    A.fout = reinterpret_cast<T *>(s->f[s->cur ^ 1]);
    A.F = fields_of<T>(s);
    A.P = phys_of<T>(s->params);
    A.mom = write_mom ? reinterpret_cast<T *>(s->mom) : nullptr;
    A.flag = s->d_flag;
    const int sl = prof_begin(s, 0);
    launch_pdl(m->n_nodes <= kOneWave ? k_rho<T, Topo, true> : k_rho<T, Topo, false>,
               nblocks(m->n_nodes, kGenBlock), kGenBlock, 0, m->stream, d, A.fin, A.P.dt, A.F.rho, A.F.hs);
    prof_end(s, sl);
    return A;
}

template <typename T, typename Topo>
static void step_topo(felbm_state *s, const Topo &d, bool write_mom) {
    const felbm_mesh *m = s->mesh;
    const CollideArgs<T, Topo> A = step_rho<T, Topo>(s, d, write_mom);
    launch_chain<T, Topo>(s, d);
    const int sl = prof_begin(s, 3);
    launch_pdl(k_collide<T, Topo>, nblocks(m->n_nodes, kGenBlock), kGenBlock, 0, m->stream, A);
    prof_end(s, sl);
    s->cur ^= 1;
}

template <typename T, typename Topo>
static void init_topo(felbm_state *s, const Topo &d) {
    const felbm_mesh *m = s->mesh;
    const Fields<T> F = fields_of<T>(s);
    const Phys<T> P = phys_of<T>(s->params);
    // F.rho <- rho0 (first quarter of the moments buffer)
    cudaMemcpyAsync(F.rho, s->mom, (size_t)m->n_nodes * sizeof(T), cudaMemcpyDeviceToDevice,
                    m->stream);
    launch_chain<T, Topo>(s, d);
    const unsigned g = nblocks(m->n_nodes, kGenBlock);
    k_init<T, Topo><<<g, kGenBlock, 0, m->stream>>>(d, reinterpret_cast<T *>(s->f[s->cur]), F, P,
                                              reinterpret_cast<const T *>(s->mom));
}

// Constant coefficient tables of a structured mesh for the state's dt.
template <typename T>
static LatCoef<T> lat_coef(const felbm_mesh *m, double dt) {
    LatCoef<T> c;
    for (int k = 0; k < 3; ++k)
        for (int o = 0; o < 6; ++o) {
            const double ax = m->sinfo.a[k][o][0], ay = m->sinfo.a[k][o][1];
            const double bxx = m->sinfo.b[k][o][0], bxy = m->sinfo.b[k][o][1],
                         byy = m->sinfo.b[k][o][2];
            c.r[k][o][0] = (T)ax;
            c.r[k][o][1] = (T)ay;
            T sv[9];
            for (int a = 1; a < 9; ++a) {
                const double ex = kEx(a), ey = kEy(a);
                sv[a] = (T)(ex * ax + ey * ay +
                            0.5 * dt * (ex * ex * bxx + 2.0 * ex * ey * bxy + ey * ey * byy));
            }
            for (int q = 0; q < 4; ++q) {
                c.s[k][o][q].x = sv[pair_dir(q, 0)];
                c.s[k][o][q].y = sv[pair_dir(q, 1)];
            }
        }
    return c;
}

template <typename T, bool LAP64>
static void step_lattice(felbm_state *s, LatArgs<T> &A, bool write_mom) {
    const felbm_mesh *m = s->mesh;
    A.fin = reinterpret_cast<const T *>(s->f[s->cur]);
    A.fout = reinterpret_cast<T *>(s->f[s->cur ^ 1]);
    A.mom = write_mom ? reinterpret_cast<T *>(s->mom) : nullptr;
    A.tmap = s->d_tmap ? s->d_tmap + 3 * s->cur : nullptr;
    const dim3 grd((A.nx + kLTX - 1) / kLTX, (A.yhi - A.ylo + kLTY - 1) / kLTY);
    const int sl = prof_begin(s, 4);
    launch_pdl(k_lat_step<T, LAP64>, grd, dim3(kLTX, kLTY), lat_smem<T>(), m->stream, A);
    prof_end(s, sl);
    s->cur ^= 1;
}

// One FP64 step of a lattice: its passes.  Few nodes are spread over the SMs
// in small blocks, many come in large ones, with fewer partial waves (us a step
// with blocks of 32, 64, 128: 100 x 100 24.6, 25.8, 26.7, 160 x 160 35.4, 35.0,
// 43.7, 256 x 256 76.1, 75.4, 81.4, 320 x 320 117.7, 117.3, 119.0, 512 x 512 all
// 269.7).
template <int S>
static void launch_pass(felbm_state *s, const LatArgs<double> &A) {
    int32_t lo, hi;
    pass_rows(A.ny, A.gny, A.ylo, A.yhi, 3 - S, lo, hi);
    const int64_t nodes = (int64_t)(hi - lo) * A.nx;
    const int bs = nodes >= 152 * 512 ? kPassBlock : (nodes >= 152 * 128 ? 64 : 32);
    const int sl = prof_begin(s, S);
    launch_pdl(k_lat_pass<double, S>, nblocks(nodes, bs), bs, 0, s->mesh->stream, A);
    prof_end(s, sl);
}

static void step_lattice64(felbm_state *s, LatArgs<double> &A, bool write_mom) {
    A.fin = reinterpret_cast<const double *>(s->f[s->cur]);
    A.fout = reinterpret_cast<double *>(s->f[s->cur ^ 1]);
    A.mom = write_mom ? reinterpret_cast<double *>(s->mom) : nullptr;
    launch_pass<0>(s, A);
    launch_pass<1>(s, A);
    launch_pass<2>(s, A);
    launch_pass<3>(s, A);
    s->cur ^= 1;
}

// The dynamic shared memory of k_lat_step is above the default limit: set
// the function attribute once per device (bit d of done, set only once the
// call succeeded; devices from 64 on set it at every call).  A refusal is
// returned to the caller of felbm_step.
template <typename T, bool LAP64>
static cudaError_t lat_smem_attr() {
    static std::atomic<uint64_t> done{0};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        dev = -1;
    }
    const uint64_t bit = (dev >= 0 && dev < 64) ? (uint64_t(1) << dev) : 0;
    if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
    const cudaError_t e =
        cudaFuncSetAttribute(k_lat_step<T, LAP64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lat_smem<T>());
    if (e != cudaSuccess) {
        cudaGetLastError();
        return e;
    }
    if (bit) done.fetch_or(bit, std::memory_order_release);
    return cudaSuccess;
}

// Shared memory of the patch kernel on a mesh.
template <typename T>
static size_t patch_bytes(const felbm_mesh *m) {
    const HostCSR &H = m->host;
    return patch_smem<T>(H.r1max, H.r2max, H.r3max, H.pemax, H.psmax);
}

// Two launches per step over a general triangle mesh with patches.
template <typename T, bool LAP64>
static cudaError_t patch_steps(felbm_state *s, int64_t n) {
    const felbm_mesh *m = s->mesh;
    const HostCSR &H = m->host;
    const size_t smem = patch_bytes<T>(m);
    const bool one = m->n_nodes <= kOneWave, lng = !H.ptail.empty();
    const auto kernel = one ? (lng ? k_patch_step<T, LAP64, true, true> : k_patch_step<T, LAP64, true, false>)
                            : (lng ? k_patch_step<T, LAP64, false, true> : k_patch_step<T, LAP64, false, false>);
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) {
        cudaGetLastError();
        return err;
    }
    const DevELL<T> d = dev_ell<T>(m);
    PatchArgs<T> A;
    A.nbase = m->d_pnbase;
    A.count = m->d_pcount;
    A.node = m->d_pnode;
    A.pslice = m->d_pslice;
    A.psbase = m->d_psbase;
    A.pcol = m->d_pcol;
    A.pstail = m->d_pstail;
    A.ptail = reinterpret_cast<const int2 *>(m->d_ptail);
    A.pa = reinterpret_cast<const V2<T> *>(m->d_pa[sizeof(T) == 8]);
    A.pa64 = reinterpret_cast<const V2<double> *>(m->d_pa[1]);
    A.r1max = H.r1max;
    A.r2max = H.r2max;
    A.r3max = H.r3max;
    A.pemax = H.pemax;
    A.psmax = H.psmax;
    A.kappa64 = kappa64(s->params);
    const unsigned blocks = (unsigned)(H.pnbase.size() - 1);
    for (int64_t k = 0; k < n; ++k) {
        A.c = step_rho<T>(s, d, k == n - 1);
        const int sl = prof_begin(s, 5);
        launch_pdl(kernel, blocks, kPatch, smem, m->stream, A);
        prof_end(s, sl);
        s->cur ^= 1;
    }
    return cudaSuccess;
}

// Whether a state on a general mesh takes the patch step: where the mesh has
// patches and a block their shared memory, always in FP32; in FP64, whose arithmetic on the rings costs more than two launches
// save beyond one wave of patches, up to there, where a row is so long that its
// one thread bounds a pass, or on a mesh made for it.  Jittered Delaunay meshes,
// us a step, patch step and four launches: FP64 300 x 300 223 and 192, 600 x 600
// 772 and 721, 1024 x 1024 2102 and 2030, with a hub of 150 neighbours 600 x 600
// 901 and 1065; FP64 Laplacian 300 x 300 29.1 and 31.3, 600 x 600 111 and 123,
// 1024 x 1024 272 and 347.
static bool patch_wanted(const felbm_state *s) {
    const felbm_mesh *m = s->mesh;
    if (m->kind != 0 || !m->patch_step ||
        (s->esize == 8 ? patch_bytes<double>(m) : patch_bytes<float>(m)) > 227 * 1024)
        return false;
    return (m->flags & FELBM_MESH_PATCH_STEP) || s->esize == 4 || m->n_nodes <= kOneWave || !m->host.ptail.empty();
}

// The device arrays of a general mesh that state s reads: its precision's
// rows, with the FP64 Laplacian the FP64 a_ij and neighbours too, and the
// patches if it takes the patch step.
static cudaError_t hold_rows(felbm_mesh *m, const felbm_state *s) {
    const HostCSR &H = m->host;
    const bool f32 = s->esize == 4, lap = lap_fp64(s);
    const std::lock_guard<std::mutex> guard(m->lock);
    cudaError_t e = f32 ? hold_ell<float>(m, true) : cudaSuccess;
    if (e == cudaSuccess && (!f32 || lap)) e = hold_ell<double>(m, !f32);
    if (e != cudaSuccess || !patch_wanted(s)) return e;
    auto hold = [&](auto *&d, const auto &v) {
        if (e == cudaSuccess && !v.empty()) e = mesh_hold(m, (void **)&d, v.data(), v.size() * sizeof(v[0]));
    };
    hold(m->d_pnbase, H.pnbase);
    hold(m->d_pcount, H.pcount);
    hold(m->d_pnode, H.pnode);
    hold(m->d_pslice, H.pslice);
    hold(m->d_psbase, H.psbase);
    hold(m->d_pstail, H.pstail);
    hold(m->d_ptail, H.ptail);
    hold(m->d_pcol, H.pcol);
    auto hold_a = [&](void *&d, auto zero) {
        if (e != cudaSuccess || d) return;
        std::vector<decltype(zero)> a(2 * H.pcsr.size(), zero);
        for (size_t k = 0; k < H.pcsr.size(); ++k)
            if (H.pcsr[k] >= 0) {
                a[2 * k] = (decltype(zero))H.ax[H.pcsr[k]];
                a[2 * k + 1] = (decltype(zero))H.ay[H.pcsr[k]];
            }
        hold(d, a);
    };
    if (f32) hold_a(m->d_pa[0], 0.0f);
    if (!f32 || lap) hold_a(m->d_pa[1], 0.0);
    return e;
}

template <typename T>
static int do_steps(felbm_state *s, int64_t n) {
    const felbm_mesh *m = s->mesh;
    if (patch_wanted(s)) {
        if constexpr (sizeof(T) == 4) {
            if (lap_fp64(s)) return cuda_status(patch_steps<T, true>(s, n));
        }
        return cuda_status(patch_steps<T, false>(s, n));
    }
    if (m->kind == 1) {
        const bool l64 = lap_fp64(s);
        cudaError_t ea = cudaSuccess;
        if constexpr (sizeof(T) == 4) ea = l64 ? lat_smem_attr<T, true>() : lat_smem_attr<T, false>();
        if (ea != cudaSuccess) return cuda_status(ea);
        LatArgs<T> A;
        A.nx = m->sinfo.nx;
        A.ny = m->sinfo.ny;
        A.pitch = m->sinfo.pitch;
        A.walls = m->sinfo.walls ? 1 : 0;
        A.row0 = m->sinfo.row0;
        A.gny = m->sinfo.gny;
        A.ylo = m->sinfo.ylo;
        A.yhi = m->sinfo.yhi;
        A.c = lat_coef<T>(m, s->params.dt);
        lat_uniform_consts<T>(m->sinfo, s->params.dt, A);
        A.P = phys_of<T>(s->params);
        A.rho = reinterpret_cast<T *>(s->scratch);
        A.flag = s->d_flag;
        A.al64 = 1.0 / (6.0 * m->sinfo.h);
        A.kappa64 = kappa64(s->params);
        for (int k = 0; k < 3; ++k)
            for (int o = 0; o < 6; ++o)
                for (int c = 0; c < 2; ++c) A.r64[k][o][c] = m->sinfo.a[k][o][c];
        for (int64_t k = 0; k < n; ++k) {
            if constexpr (sizeof(T) == 8)
                step_lattice64(s, A, k == n - 1);
            else if (l64)
                step_lattice<T, true>(s, A, k == n - 1);
            else
                step_lattice<T, false>(s, A, k == n - 1);
        }
    } else {
        const DevELL<T> d = dev_ell<T>(m);
        for (int64_t k = 0; k < n; ++k) step_topo<T>(s, d, k == n - 1);
    }
    return FELBM_OK;
}

template <typename T>
static void init_any(felbm_state *s) {
    if (s->mesh->kind == 1)
        init_topo<T>(s, dev_lattice<T>(s->mesh));
    else
        init_topo<T>(s, dev_ell<T>(s->mesh));
}

template <typename T>
static void launch_moments(felbm_state *s) {
    const felbm_mesh *m = s->mesh;
    const int32_t n = (int32_t)m->n_nodes;
    const int32_t *iperm = m->kind == 1 ? nullptr : m->d_perm + n;  // d_perm holds perm | iperm
    k_gather_moments<T><<<nblocks(n, 256), 256, 0, m->stream>>>(
        n, reinterpret_cast<const T *>(s->mom), iperm, s->params.rho_l, s->params.rho_v, s->d_out);
    double *part = s->d_out + 5 * (size_t)n;
    k_totals_partial<T><<<kTotalsBlocks, 256, 0, m->stream>>>(
        n, reinterpret_cast<const T *>(s->mom), m->d_mass, part);
    k_totals_final<<<1, 32, 0, m->stream>>>(kTotalsBlocks, part, part + 3 * kTotalsBlocks);
}

void mesh_free(felbm_mesh *m) {
    if (!m) return;
    cudaFree(m->d_sbase);
    cudaFree(m->d_deg);
    for (auto &p : m->d_ell)
        for (void *q : p) cudaFree(q);
    cudaFree(m->d_perm);
    cudaFree(m->d_mass);
    cudaFree(m->d_tag);
    cudaFree(m->d_pnbase);
    cudaFree(m->d_pcount);
    cudaFree(m->d_pnode);
    cudaFree(m->d_pslice);
    cudaFree(m->d_psbase);
    cudaFree(m->d_pstail);
    cudaFree(m->d_ptail);
    cudaFree(m->d_pcol);
    for (void *q : m->d_pa) cudaFree(q);
    delete m;
}

void state_free(felbm_state *s) {
    if (!s) return;
    for (auto &e : s->prof_ev)
        if (e) cudaEventDestroy(e);
    cudaFree(s->f[0]);
    cudaFree(s->f[1]);
    cudaFree(s->scratch);
    cudaFree(s->mom);
    cudaFree(s->d_out);
    cudaFree(s->d_flag);
    cudaFree(s->d_tmap);
    cudaFree(s->halo);
    delete s;
}

bool params_ok(const felbm_params *p) {
    const double v[] = {p->rho_l, p->rho_v, p->sigma, p->xi, p->tau_l, p->tau_v, p->dt,
                        p->gravity[0], p->gravity[1], p->gravity[2]};
    for (double x : v)
        if (!std::isfinite(x)) return false;
    return p->rho_l > p->rho_v && p->rho_v > 0.0 && p->sigma >= 0.0 && p->xi > 0.0 &&
           p->tau_l > 0.0 && p->tau_v > 0.0 && p->dt > 0.0 &&
           (p->precision == FELBM_FP64 || p->precision == FELBM_FP32) && (p->flags & ~FELBM_PARAM_LAP_FP64) == 0;
}

// One block waits on an mbarrier that nothing arrives on (phase 0 never
// completes), through the same bounded wait the tiles use for their TMA
// loads, and records the give-up in the flag as a tile does.
__global__ void k_wait_selftest(int *flag, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
    }
    __syncthreads();
    const bool ok = threadIdx.x != 0 || mbar_wait(&bar, 0u, limit_ns);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicOr(flag, 4);
}

FELBM_CHECK_READER(check_bits_api)

}  // namespace felbm

// ============================================================================
extern "C" {

int felbm_check_status(int32_t *checked_build, int32_t *bits) {
    if (!checked_build || !bits) return FELBM_ERR_INVALID_ARG;
#ifdef FELBM_CHECKED
    *checked_build = 1;
#else
    *checked_build = 0;
#endif
    *bits = (int32_t)(check_bits_api() | check_bits_api3() | check_bits_batch() | check_bits_slab());
    return FELBM_OK;
}

int felbm_wait_selftest(felbm_state *s, int64_t limit_ns) {
    if (!s || limit_ns < 1 || limit_ns > 2000000000LL) return FELBM_ERR_INVALID_ARG;
    k_wait_selftest<<<1, 32, 0, s->mesh->stream>>>(s->d_flag, (uint64_t)limit_ns);
    return cuda_status(cudaGetLastError());
}

const char *felbm_status_string(int st) {
    switch (st) {
        case FELBM_OK: return "ok";
        case FELBM_ERR_INVALID_ARG: return "invalid argument";
        case FELBM_ERR_INVALID_MESH: return "invalid mesh";
        case FELBM_ERR_OOM: return "out of memory";
        case FELBM_ERR_NONFINITE: return "non-finite value produced";
        case FELBM_ERR_TIMEOUT: return "bounded device wait gave up";
        case FELBM_ERR_CUDA: return "CUDA error";
        case FELBM_ERR_UNSUPPORTED: return "unsupported";
        default: return "unknown status";
    }
}


int felbm_mesh_create(const double *xy, int64_t n_nodes, const int32_t *tri, int64_t n_tri,
                      const double box[2], uint32_t flags, const uint8_t *node_tag, void *stream,
                      felbm_mesh **out) {
    if (!xy || !tri || !box || !out) return FELBM_ERR_INVALID_ARG;
    if (n_nodes < 3 || n_tri < 1 || n_nodes > 0x7fffffffLL || n_tri > 0x7fffffffLL / 3)
        return FELBM_ERR_INVALID_ARG;
    if ((flags & ~(FELBM_PERIODIC_X | FELBM_PERIODIC_Y | FELBM_MESH_GENERAL | FELBM_MESH_SPLIT_STEP |
                   FELBM_MESH_PATCH_STEP)) ||
        ((flags & FELBM_MESH_SPLIT_STEP) && (flags & FELBM_MESH_PATCH_STEP)))
        return FELBM_ERR_INVALID_ARG;
    felbm_mesh *m = new (std::nothrow) felbm_mesh();
    if (!m) return FELBM_ERR_OOM;
    m->n_nodes = n_nodes;
    m->n_tri = n_tri;
    m->flags = flags;
    m->stream = reinterpret_cast<cudaStream_t>(stream);
    // cheap checks every path relies on
    if (((flags & FELBM_PERIODIC_X) && !(box[0] > 0.0)) ||
        ((flags & FELBM_PERIODIC_Y) && !(box[1] > 0.0))) {
        delete m;
        return FELBM_ERR_INVALID_ARG;
    }
    for (int64_t t = 0; t < 3 * n_tri; ++t)
        if (tri[t] < 0 || tri[t] >= n_nodes) {
            delete m;
            return FELBM_ERR_INVALID_MESH;
        }
    int st = FELBM_OK;
    std::vector<double> lattice_mass;
    try {
        // a structured lattice needs no assembled CSR: its three row kinds'
        // coefficients come from the triangles around representative nodes
        if (!(flags & FELBM_MESH_GENERAL))
            detect_structured(xy, n_nodes, tri, n_tri, box, flags, node_tag, m->sinfo, lattice_mass);
        if (!m->sinfo.ok) st = build_csr(xy, n_nodes, tri, n_tri, box, flags, node_tag, m->host);
    } catch (const std::bad_alloc &) {
        st = FELBM_ERR_OOM;
    }
    if (st != FELBM_OK) {
        delete m;
        return st;
    }
    m->kind = m->sinfo.ok ? 1 : 0;
    const HostCSR &H = m->host;
    const size_t N = (size_t)n_nodes;
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **p, size_t bytes) {
        if (e == cudaSuccess) {
            e = cudaMalloc(p, bytes);
            if (e == cudaSuccess) m->device_bytes += (int64_t)bytes;
        }
    };
    alloc((void **)&m->d_mass, N * sizeof(double));
    if (m->kind == 0) {
        alloc((void **)&m->d_perm, 2 * N * sizeof(int32_t));
        if (!H.tag.empty()) alloc((void **)&m->d_tag, N);
        m->patch_step = !H.pnbase.empty() && !(flags & FELBM_MESH_SPLIT_STEP);
    }
    if (e != cudaSuccess) {
        int rs = cuda_status(e);
        mesh_free(m);
        return rs;
    }
    // uploads (synchronous: host vectors are temporaries of this call)
    if (m->kind == 1) {
        // structured kernels use the caller's (lattice) order
        e = cudaMemcpy(m->d_mass, lattice_mass.data(), N * sizeof(double), cudaMemcpyHostToDevice);
    } else {
        e = cudaMemcpy(m->d_mass, H.mass.data(), N * sizeof(double), cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(m->d_perm, H.perm.data(), N * sizeof(int32_t), cudaMemcpyHostToDevice);
        if (e == cudaSuccess)
            e = cudaMemcpy(m->d_perm + N, H.iperm.data(), N * sizeof(int32_t), cudaMemcpyHostToDevice);
        if (e == cudaSuccess && m->d_tag)
            e = cudaMemcpy(m->d_tag, H.tag.data(), N, cudaMemcpyHostToDevice);
        try {
            auto up = [&](void *d, const void *h, size_t b) {
                if (e == cudaSuccess) e = mesh_upload(m, (void **)d, h, b);
            };
            const std::vector<int32_t> sb = ell_slices(H.n, H.rowptr);
            std::vector<uint8_t> deg(N);
            for (size_t k = 0; k < N; ++k) deg[k] = (uint8_t)std::min(255, H.rowptr[k + 1] - H.rowptr[k]);
            up(&m->d_sbase, sb.data(), sb.size() * sizeof(int32_t));
            up(&m->d_deg, deg.data(), N);
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    if (e != cudaSuccess) {
        int rs = cuda_status(e);
        mesh_free(m);
        return rs;
    }
    *out = m;
    return FELBM_OK;
}

int felbm_mesh_info(const felbm_mesh *m, int64_t *n_nodes, int64_t *n_tri, int32_t *kind,
                    int64_t *device_bytes) {
    if (!m) return FELBM_ERR_INVALID_ARG;
    if (n_nodes) *n_nodes = m->n_nodes;
    if (n_tri) *n_tri = m->n_tri;
    if (kind) *kind = m->kind;
    if (device_bytes) {
        const std::lock_guard<std::mutex> guard(m->lock);
        *device_bytes = m->device_bytes;
    }
    return FELBM_OK;
}

void felbm_mesh_destroy(felbm_mesh *m) { mesh_free(m); }



int felbm_state_init(const felbm_mesh *mesh, const felbm_params *params, const double *rho0,
                     const double *u0, const double *p0, felbm_state **out) {
    felbm::NvtxRange nvtx_range("felbm_state_init");
    if (!mesh || !params || !rho0 || !out) return FELBM_ERR_INVALID_ARG;
    if (!params_ok(params)) return FELBM_ERR_INVALID_ARG;
    if (mesh->kind >= 2) return state_init3(mesh, params, rho0, u0, p0, out);
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
    alloc(&s->f[0], 18 * pad4(pop_slots(mesh)) * es);
    alloc(&s->f[1], 18 * pad4(pop_slots(mesh)) * es);
    alloc(&s->scratch, (hstar_elems(mesh) + 6 * N) * es);
    alloc(&s->mom, 4 * N * es);
    alloc((void **)&s->d_out, (5 * N + 3 * (kTotalsBlocks + 1)) * sizeof(double));
    alloc((void **)&s->d_flag, sizeof(int));
    if (e == cudaSuccess && mesh->kind == 0) {
        try {
            e = hold_rows(const_cast<felbm_mesh *>(mesh), s);
        } catch (const std::bad_alloc &) {
            e = cudaErrorMemoryAllocation;
        }
    }
    if (e != cudaSuccess) {
        int rs = cuda_status(e);
        state_free(s);
        return rs;
    }
    // initial moments in the kernels' node order and precision
    const bool perm = mesh->kind == 0;
    std::vector<unsigned char> hm(4 * N * es);
    for (size_t k = 0; k < N; ++k) {
        const size_t c = perm ? (size_t)mesh->host.perm[k] : k;
        const double v[4] = {rho0[c], u0 ? u0[2 * c] : 0.0, u0 ? u0[2 * c + 1] : 0.0,
                             p0 ? p0[c] : 0.0};
        for (int q = 0; q < 4; ++q) {
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
    // padding slots of structured rows are never read; zeroed all the same
    for (int c = 0; c < 2 && e == cudaSuccess; ++c)
        e = cudaMemsetAsync(s->f[c], 0, 18 * pad4(pop_slots(mesh)) * es, mesh->stream);
    if (e == cudaSuccess) {
        if (es == 8)
            init_any<double>(s);
        else
            init_any<float>(s);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(mesh->stream);  // hm is a temporary
    if (e != cudaSuccess) {
        int rs = cuda_status(e);
        state_free(s);
        return rs;
    }
    lattice_tmaps(s);  // optional: tiles fall back to cp.async fills without maps
    s->have_moments = true;
    *out = s;
    return FELBM_OK;
}

int felbm_step(felbm_state *s, int64_t n_steps) {
    felbm::NvtxRange nvtx_range("felbm_step");
    if (!s || n_steps < 0) return FELBM_ERR_INVALID_ARG;
    if (n_steps == 0) return FELBM_OK;
    if (s->mesh->kind >= 2) {
        steps3(s, n_steps);
    } else {
        const int st = s->esize == 8 ? do_steps<double>(s, n_steps) : do_steps<float>(s, n_steps);
        if (st != FELBM_OK) return st;
    }
    s->steps_done += n_steps;
    s->have_moments = true;
    return cuda_status(cudaGetLastError());
}

static int check_flag(felbm_state *s) {
    int h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, s->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s->mesh->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->mesh->stream);
    if (e != cudaSuccess) return cuda_status(e);
    return (h & 1) ? FELBM_ERR_NONFINITE : (h & 4) ? FELBM_ERR_TIMEOUT : FELBM_OK;
}

int felbm_state_sync(felbm_state *s) {
    if (!s) return FELBM_ERR_INVALID_ARG;
    return check_flag(s);
}

int felbm_moments_get(felbm_state *s, double *rho, double *C, double *u, double *p, double totals[3]) {
    felbm::NvtxRange nvtx_range("felbm_moments_get");
    if (!s) return FELBM_ERR_INVALID_ARG;
    if (!s->have_moments) return FELBM_ERR_INVALID_ARG;
    if (s->mesh->kind >= 2) {
        const int st3 = moments3(s, rho, C, u, p, totals);
        return st3 != FELBM_OK ? st3 : check_flag(s);
    }
    const size_t N = (size_t)s->mesh->n_nodes;
    const cudaStream_t st = s->mesh->stream;
    if (s->esize == 8)
        launch_moments<double>(s);
    else
        launch_moments<float>(s);
    cudaError_t e = cudaGetLastError();
    double *o = s->d_out;
    if (e == cudaSuccess && rho) e = cudaMemcpyAsync(rho, o, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && C) e = cudaMemcpyAsync(C, o + N, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && u) e = cudaMemcpyAsync(u, o + 2 * N, 2 * N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && p) e = cudaMemcpyAsync(p, o + 4 * N, N * 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && totals)
        e = cudaMemcpyAsync(totals, o + 5 * N + 3 * kTotalsBlocks, 3 * 8, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return cuda_status(e);
    return check_flag(s);
}

int felbm_state_export(felbm_state *s, double *hbar, double *gbar) {
    if (!s || !hbar || !gbar) return FELBM_ERR_INVALID_ARG;
    if (s->mesh->kind >= 2) {
        const int st3 = export3(s, hbar, gbar);
        return st3 != FELBM_OK ? st3 : check_flag(s);
    }
    const size_t N = (size_t)s->mesh->n_nodes, es = s->esize, S = pop_slots(s->mesh);
    std::vector<unsigned char> buf(18 * pad4(S) * es);
    cudaError_t e = cudaMemcpyAsync(buf.data(), s->f[s->cur], buf.size(), cudaMemcpyDeviceToHost,
                                    s->mesh->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->mesh->stream);
    if (e != cudaSuccess) return cuda_status(e);
    const bool perm = s->mesh->kind == 0;
    for (int a = 0; a < 18; ++a)
        for (size_t k = 0; k < N; ++k) {
            const size_t c = perm ? (size_t)s->mesh->host.perm[k] : k;
            const size_t q = pop_index(a, pop_slot(s->mesh, k), S);
            const double v = es == 8 ? reinterpret_cast<double *>(buf.data())[q]
                                     : (double)reinterpret_cast<float *>(buf.data())[q];
            (a < 9 ? hbar : gbar)[(a % 9) * N + c] = v;
        }
    return check_flag(s);
}

int felbm_state_import(felbm_state *s, const double *hbar, const double *gbar) {
    if (!s || !hbar || !gbar) return FELBM_ERR_INVALID_ARG;
    if (s->mesh->kind >= 2) return import3(s, hbar, gbar);
    const size_t N = (size_t)s->mesh->n_nodes, es = s->esize, S = pop_slots(s->mesh);
    std::vector<unsigned char> buf(18 * pad4(S) * es, 0);
    const bool perm = s->mesh->kind == 0;
    for (int a = 0; a < 18; ++a)
        for (size_t k = 0; k < N; ++k) {
            const size_t c = perm ? (size_t)s->mesh->host.perm[k] : k;
            const double v = (a < 9 ? hbar : gbar)[(a % 9) * N + c];
            if (!std::isfinite(v)) return FELBM_ERR_INVALID_ARG;
            const size_t q = pop_index(a, pop_slot(s->mesh, k), S);
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

void felbm_state_destroy(felbm_state *s) {
    if (!s) return;
    cudaStreamSynchronize(s->mesh->stream);
    state_free(s);
}

int felbm_profile_enable(felbm_state *s, int on) {
    if (!s || on < 0) return FELBM_ERR_INVALID_ARG;
    if (on && s->prof_ev.empty()) {
        try {
            s->prof_ev.assign(2 * kProfMaxLaunches, nullptr);
            s->prof_kind.assign(kProfMaxLaunches, 0);
        } catch (const std::bad_alloc &) {
            return FELBM_ERR_OOM;
        }
        for (auto &e : s->prof_ev) {
            cudaError_t r = cudaEventCreate(&e);
            if (r != cudaSuccess) return cuda_status(r);
        }
    }
    s->prof_on = on != 0;
    s->prof_stride = on > 0 ? on : 1;
    s->prof_used = 0;
    for (auto &c : s->launches) c = 0;
    for (auto &c : s->prof_seen) c = 0;
    return FELBM_OK;
}

int felbm_profile_read(felbm_state *s, double *ms, int64_t *timed, int64_t *launches) {
    if (!s) return FELBM_ERR_INVALID_ARG;
    cudaError_t e = cudaStreamSynchronize(s->mesh->stream);
    if (e != cudaSuccess) return cuda_status(e);
    double acc[8] = {0};
    int64_t cnt[8] = {0};
    for (size_t k = 0; k < s->prof_used; ++k) {
        float t = 0.f;
        e = cudaEventElapsedTime(&t, s->prof_ev[2 * k], s->prof_ev[2 * k + 1]);
        if (e != cudaSuccess) return cuda_status(e);
        acc[s->prof_kind[k]] += t;
        cnt[s->prof_kind[k]]++;
    }
    for (int k = 0; k < FELBM_PROFILE_KINDS; ++k) {
        if (ms) ms[k] = acc[k];
        if (timed) timed[k] = cnt[k];
        if (launches) launches[k] = s->launches[k];
        s->launches[k] = 0;
    }
    s->prof_used = 0;
    return FELBM_OK;
}

const char *felbm_profile_kind_name(int k) {
    static const char *names[FELBM_PROFILE_KINDS] = {
        "k_rho", "k_grad", "k_mu", "k_collide", "k_lattice_step", "k_patch_step", "unused6",
        "unused7"};
    return (k >= 0 && k < FELBM_PROFILE_KINDS) ? names[k] : nullptr;
}

}  // extern "C"
