// Internal declarations of the FE-LBM library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>
#include <stdint.h>

#include <mutex>
#include <utility>
#include <vector>

#include "../../include/felbm.h"

namespace felbm {

// ---- checked build (FELBM_CHECKED) -----------------------------------------
// Kernels bounds-check the indices they gather with and record a violation
// as a bit of a device status word (no assert, no trap: the access is
// skipped); felbm_check_status reads and clears it.  Bits: 1 a gathered node
// or slot index out of range, 2 a shared-memory (region) index out of range,
// 4 a TMA box coordinate off its 16-byte rule (the tile then loads by
// cp.async), 8 a slab halo copy out of range.  Without FELBM_CHECKED every
// check is the constant true.  Each translation unit holds its own status
// word (no relocatable device code) and a reader, check_bits_<unit>().
#ifdef __CUDACC__
#ifdef FELBM_CHECKED
static __device__ unsigned g_check_bits;
__device__ __forceinline__ bool chk_idx(long long i, long long n, unsigned bit) {
    if (i >= 0 && i < n) return true;
    atomicOr(&g_check_bits, bit);
    return false;
}
#define FELBM_CHECK_READER(name)                                                  \
    unsigned name() {                                                             \
        unsigned v = 0, z = 0;                                                    \
        cudaDeviceSynchronize();                                                  \
        if (cudaMemcpyFromSymbol(&v, g_check_bits, sizeof v) != cudaSuccess) v = ~0u; \
        cudaMemcpyToSymbol(g_check_bits, &z, sizeof z);                           \
        return v;                                                                 \
    }
#else
__device__ __forceinline__ constexpr bool chk_idx(long long, long long, unsigned) { return true; }
#define FELBM_CHECK_READER(name) \
    unsigned name() { return 0u; }
#endif
#endif
// NVTX range around an entry point (seen by nsys / ncu; a no-op otherwise).
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

// ---- programmatic dependent launch -----------------------------------------
// The kernels of a step are launched with programmatic stream serialisation
// (batches in FP64 and those that walk their tiles apart, plain launches):
// a kernel may start while its predecessor drains, reads only what no kernel
// writes (mesh tables) before pdl_wait(), and everything else after it.
// pdl_wait() returns once the predecessor has completed, which itself waited
// for its own, so the order of all memory accesses is that of plain launches.
// Kernels do not trigger before their end (griddepcontrol.launch_dependents),
// the patch step of meshes whose blocks are all resident apart: the blocks of
// the next launch then come as blocks of this one leave, and spread evenly.
// With a trigger behind the wait they took the slots that were free,
// the emptier SMs' first: a 357 x 203 lattice in FP32 ran 11.1 us a step with
// it, 8.3 without and 10.3 as plain launches (512 x 2048: 46.3, 45.8, 47.8; 32
// x 32: 4.2, 4.1, 6.2; 357 x 203 in FP64: 98.5 with it, 82.2 without).
// What other kernels write is read with plain loads or ldp(): the compiler
// may move non-coherent ones (__ldg, const __restrict__) ahead of the wait.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A pointer to what the kernels before wrote, taken after pdl_wait(), and
// coherent loads through it that the compiler may move across the kernel's
// own stores (it cannot tell that fields and populations do not overlap), but
// not above that point: the address comes from a volatile statement behind
// the wait.  Only for arrays that the kernel does not write.
template <typename T>
__device__ __forceinline__ const T *pdl_ptr(const T *p) {
    asm volatile("" : "+l"(p));
    return p;
}
__device__ __forceinline__ float ldp(const float *p) {
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double ldp(const double *p) {
    double v;
    asm("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 ldp(const float2 *p) {
    float2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ldp(const float4 *p) {
    float4 v;
    asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ldp(const double2 *p) {
    double2 v;
    asm("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A &&...args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
#endif

unsigned check_bits_api();
unsigned check_bits_api3();
unsigned check_bits_batch();
unsigned check_bits_slab();

// ---- host-side mesh preprocessing (felbm_mesh.cu) -------------------------

// Assembled per-node operators in the internal (reverse Cuthill-McKee) order.
// For node i and each neighbour j != i sharing a triangle:
//   a_ij = sum_{T∋i,j} |T| grad N_j^T / (3 m_i)                 (2-vector)
//   b_ij = sum_{T∋i,j} |T| / m_i * sym(grad N_i^T (x) grad N_j^T)  (2x2, symmetric part)
// so that, with sum_j a_ij = 0 and sum_j b_ij = 0 (P1 partition of unity),
//   recovered gradient  (R f)_i   = sum_{j!=i} a_ij (f_j - f_i)
//   lumped TG streaming psi*_i    = psi_i - dt sum_{j!=i} (e.a_ij + dt/2 e.b_ij.e)(psi_j - psi_i)
struct HostCSR {
    int32_t n = 0;
    std::vector<int32_t> rowptr, col;
    std::vector<double> ax, ay, bxx, bxy, byy;
    std::vector<double> mass;      // lumped mass, internal order
    std::vector<uint8_t> tag;      // internal order, empty if no walls
    std::vector<int32_t> perm;     // perm[internal] = caller id
    std::vector<int32_t> iperm;    // iperm[caller] = internal id
    // Patches (internal order is patch-major: patch p owns the nodes
    // [p kPatch, min(n, (p + 1) kPatch))).  Per patch its region: its own
    // nodes, then the nodes 1, 2 and 3 edges away, as internal ids in
    // pnode[pnbase[p] ..); pcount[4 p ..] the counts of rings <= 0, 1, 2, 3.
    // The rows of rings <= 2 lie in slices of 32 (as DevELL's), with up to
    // kPatchRow entries of a row; the rest of longer rows follows behind the
    // patch's slices, row by row, padded to a multiple of 32 (a slice as wide
    // as its longest row would be 32 times that row).  pslice[p] is the
    // patch's first entry of psbase, which holds its slices' first rows of 32
    // entries, their end and the patch's; pcol has the region index and pcsr
    // the CSR entry of each (-1: padding, index of the row).  pstail (as
    // psbase) is -1 or the number t of a slice with longer rows, whose row l
    // has its further entries at [ptail[64 t + 2 l], + ptail[64 t + 2 l + 1])
    // from the patch's first; both are empty where no row is longer.
    std::vector<int32_t> pnbase, pcount, pnode, pslice, psbase, pcsr, pstail, ptail;
    std::vector<uint16_t> pcol;
    int32_t r1max = 0, r2max = 0, r3max = 0;  // largest ring <= 1, 2, 3 sizes
    int32_t pemax = 0, psmax = 0;             // most rows of 32 entries, most slices of a patch
};

constexpr int kPatch = 256;   // nodes per patch of general triangle meshes
constexpr int kPatchRow = 32;  // entries of a row in a patch's slices

// General tetrahedral mesh (3-D), same conventions: for each neighbour j != i
// a_ij = sum_{T∋i,j} |T| grad N_j / (4 m_i) (3 components) and the symmetric
// part of b_ij = sum |T|/m_i grad N_i (x) grad N_j (6 components: xx, xy, xz,
// yy, yz, zz).
struct HostCSR3 {
    int32_t n = 0;
    std::vector<int32_t> rowptr, col;
    std::vector<double> coef;      // 9 * nnz, SoA: ax, ay, az, bxx, bxy, bxz, byy, byz, bzz
    std::vector<double> mass;      // lumped mass m_i = sum |T|/4, internal order
    std::vector<uint8_t> tag;      // internal order, empty if no walls (1..18: inward e_k)
    std::vector<int32_t> perm;     // perm[internal] = caller id
    std::vector<int32_t> iperm;    // iperm[caller] = internal id
};

// Kuhn-split cube lattice (3-D): node i = x + nx (y + ny z) at (x, y, z) h,
// every cube cut into the six tetrahedra around its (0,0,0)-(1,1,1)
// diagonal, periodic in x and y, periodic in z or walled (tags 5 on z = 0,
// 6 on z = nz - 1).  The 14 neighbour offsets are lat3_d*(o); c holds the
// assembled coefficients (HostCSR3 order) per z-layer kind (0 interior, 1
// bottom wall layer, 2 top wall layer) and offset, zero where the offset
// leaves a walled domain.
struct Lattice3Info {
    bool ok = false;
    int32_t nx = 0, ny = 0, nz = 0;
    bool walls = false;
    double c[3][14][9];
};

#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int lat3_dx(int o) {
    return (o == 0 || o == 6 || o == 8 || o == 12) ? 1 : (o == 1 || o == 7 || o == 9 || o == 13) ? -1 : 0;
}
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int lat3_dy(int o) {
    return (o == 2 || o == 6 || o == 10 || o == 12) ? 1 : (o == 3 || o == 7 || o == 11 || o == 13) ? -1 : 0;
}
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int lat3_dz(int o) {
    return (o == 4 || o == 8 || o == 10 || o == 12) ? 1 : (o == 5 || o == 9 || o == 11 || o == 13) ? -1 : 0;
}

struct StructuredInfo {
    bool ok = false;
    int32_t nx = 0, ny = 0;
    int32_t pitch = 0;   // population row pitch: nx rounded up to a multiple of 4
    bool walls = false;  // non-periodic y with walls on the first and last row
    double h = 1.0;
    // A slab of a sharded lattice (felbm_mesh_slab): storage row r is row
    // r + row0 of the whole lattice of gny rows, the slab's own rows are the
    // storage rows [ylo, yhi), with 4 halo rows below and above.  A whole
    // lattice: row0 = ylo = 0, gny = yhi = ny.
    int32_t row0 = 0, gny = 0, ylo = 0, yhi = 0;
    // 6 neighbour offsets (dx, dy) and their assembled a/b coefficients of an
    // interior node; wall rows get their own sets (bottom, top).
    double a[3][6][2];
    double b[3][6][3];
};

int build_csr(const double *xy, int64_t n_nodes, const int32_t *tri, int64_t n_tri,
              const double box[2], uint32_t flags, const uint8_t *tag, HostCSR &out);
// Tetrahedral mesh: validation, geometry, assembly, RCM (felbm_mesh3.cu).
int build_csr3(const double *xyz, int64_t n_nodes, const int32_t *tet, int64_t n_tet,
               const double box[3], uint32_t flags, const uint8_t *tag, HostCSR3 &out);
// Recognise the Kuhn lattice in an assembled tetrahedral mesh (H in RCM
// order); on success fills info (felbm_mesh3.cu).
void detect_lattice3(const double *xyz, int64_t n_nodes, const double box[3], uint32_t flags,
                     const uint8_t *tag, const HostCSR3 &H, Lattice3Info &info);
// Reverse Cuthill-McKee order of a node graph given as CSR without self loops.
std::vector<int32_t> rcm_order(int32_t n, const std::vector<int32_t> &rp,
                               const std::vector<int32_t> &cl);
// Recognise the structured lattice split; on success fills info (sizes and
// the coefficients of the three row kinds) and the lumped mass (lattice order).
void detect_structured(const double *xy, int64_t n_nodes, const int32_t *tri, int64_t n_tri,
                       const double box[2], uint32_t flags, const uint8_t *tag,
                       StructuredInfo &info, std::vector<double> &mass);

// ---- device-side views --------------------------------------------------

// Neighbour topologies.  each(row(i), fn) calls fn(j, ax, ay, bxx, bxy, byy)
// for every neighbour j != i of node i with the assembled coefficients a_ij,
// b_ij; tag_of(i) is the wall tag (0 = fluid).

// Rows of a general mesh in slices of 32 nodes (a warp's), internal order:
// slice s holds rows sbase[s] .. sbase[s+1] of 32 entries, row k the k-th
// neighbour of each of its nodes, in the order of the CSR row.  A warp's
// loads of one row are then consecutive 16- and 8-byte words: against CSR
// arrays, where lanes step by a whole row, a pass over the rows touches a
// sixth of the cache lines.  Entries past a node's degree hold the node
// itself and zero coefficients; they are not read.
template <typename T>
struct alignas(2 * sizeof(T)) Ell2 {
    T x, y;
};
template <typename T>
struct alignas(16) Ell4 {
    T x, y, z, w;
};
#ifdef __CUDACC__
#define FELBM_HD __host__ __device__
#else
#define FELBM_HD
#endif
// a node id in a T (its bits, or its value in FP64), and back
template <typename T>
FELBM_HD inline T ell_id(int32_t c) {
    if (sizeof(T) == 8) return (T)c;
    union {
        int32_t i;
        float f;
    } u;
    u.i = c;
    return (T)u.f;
}
#ifdef __CUDACC__
__device__ __forceinline__ Ell2<float> ell_load(const Ell2<float> *p) {
    const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ Ell2<double> ell_load(const Ell2<double> *p) {
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ Ell4<float> ell_load(const Ell4<float> *p) {
    const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
    return {v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ Ell4<double> ell_load(const Ell4<double> *p) {
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p)), b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
    return {a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ int32_t ell_get(float w) { return __float_as_int(w); }
__device__ __forceinline__ int32_t ell_get(double w) { return __double2int_rn(w); }
#endif

// General triangle mesh: {a_x, a_y}, {b_xx, b_xy} and {b_yy, neighbour}.
// row(i) reads the first entries of node i, which no kernel writes;
// each(row, fn) calls fn(j, ax, ay, bxx, bxy, byy) for all of them, in
// chunks.  Within a chunk the code has no branch, so that all its gathers are
// in flight at once: a pass waits for one L2 access per chunk and not per
// neighbour.  Chunks of 4 in FP32, 2 in FP64 (jittered Delaunay, us a step,
// chunks of 4 / 2, twice and half as long: FP32 256 x 256 10.8, 12.8, 12.0, 600
// x 600 62, 75, 64; FP64 153, 152, 161 and 770, 762, 802).
template <typename T>
struct DevELL {
    static constexpr int kChunk = sizeof(T) == 4 ? 4 : 2;
    int32_t n;
    const int32_t *sbase;
    const Ell2<T> *a, *b, *c;
    const uint8_t *deg;   // neighbours of each node (255: as many as its slice has rows)
    const uint8_t *tag;   // nullptr if no walls
#ifdef __CUDACC__
    struct Chunk {
        Ell2<T> a[kChunk], b[kChunk], c[kChunk];
    };
    struct Row {
        size_t p;  // first entry
        int32_t i, deg;
        Chunk k[2];
    };
    // entries k0 .. k0 + kChunk - 1 of a row (A: with a)
    template <bool A>
    __device__ __forceinline__ void load(size_t p, int32_t i, int32_t deg, int k0, Chunk &r) const {
#pragma unroll
        for (int k = 0; k < kChunk; ++k) {
            r.a[k] = r.b[k] = {T(0), T(0)};
            r.c[k] = {T(0), ell_id<T>(i)};
            if (k0 + k < deg) {
                const size_t e = p + 32 * (k0 + k);
                if (A) r.a[k] = ell_load(a + e);
                r.b[k] = ell_load(b + e);
                r.c[k] = ell_load(c + e);
            }
        }
    }
    template <bool A = true>
    __device__ __forceinline__ Row row(int32_t i) const {
        Row r;
        r.i = i;
        r.deg = __ldg(deg + i);
        const int32_t s0 = __ldg(sbase + (i >> 5));
        if (r.deg == 255) r.deg = __ldg(sbase + (i >> 5) + 1) - s0;  // (entries past its own: itself, zero)
        r.p = (size_t)s0 * 32 + (i & 31);
        load<A>(r.p, i, r.deg, 0, r.k[0]);
        load<A>(r.p, i, r.deg, kChunk, r.k[1]);
        return r;
    }
    // fn for the entries of a chunk; get(k, a): the recovery coefficients of
    // the row's k-th entry where the chunk was loaded without them
    template <typename Fn, typename Get>
    __device__ __forceinline__ void chunk(const Chunk &r, int k0, Fn &&fn, Get &&get) const {
#pragma unroll
        for (int k = 0; k < kChunk; ++k) {
            const int32_t j = ell_get(r.c[k].y);
            const Ell2<T> a = get(k0 + k, r.a[k]);
            if (chk_idx(j, n, 1u)) fn(j, a.x, a.y, r.b[k].x, r.b[k].y, r.c[k].x);
        }
    }
    template <bool A = true, typename Fn, typename Get>
    __device__ __forceinline__ void each_get(const Row &r, Fn &&fn, Get &&get) const {
        chunk(r.k[0], 0, fn, get);
        if (r.deg > kChunk) chunk(r.k[1], kChunk, fn, get);
        for (int k = 2 * kChunk; k < r.deg; k += kChunk) {
            Chunk c2;
            load<A>(r.p, r.i, r.deg, k, c2);
            chunk(c2, k, fn, get);
        }
    }
    template <typename Fn>
    __device__ __forceinline__ void each(const Row &r, Fn &&fn) const {
        each_get(r, fn, [](int, Ell2<T> v) { return v; });
    }
    __device__ __forceinline__ int tag_of(int32_t i) const { return tag ? (int)tag[i] : 0; }
    // population storage: slot of node i, slots per population array
    __device__ __forceinline__ size_t slot(int32_t i) const { return (size_t)i; }
    __device__ __forceinline__ size_t slots() const { return (size_t)n; }
#endif
};

// Structured lattice split (node i = x + nx*y): six neighbours at fixed
// offsets, coefficients of three row kinds (0 interior, 1 bottom wall row,
// 2 top wall row) held in the kernel parameters.  Populations are stored in
// rows of `pitch` slots (x + pitch*y), pitch = nx rounded up to a multiple
// of 4, so that every row starts 16-byte aligned.
// offsets o = 0..5: (1,0), (1,1), (0,1), (-1,0), (-1,-1), (0,-1)
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int lat_dx(int o) { return o == 0 || o == 1 ? 1 : (o == 3 || o == 4 ? -1 : 0); }
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int lat_dy(int o) { return o == 1 || o == 2 ? 1 : (o == 4 || o == 5 ? -1 : 0); }

template <typename T>
struct DevLattice {
    int32_t n, nx, ny, walls, pitch;
    int32_t row0, gny;  // storage row y is row y + row0 of a lattice of gny rows
    T c[3][6][5];  // ax, ay, bxx, bxy, byy
#ifdef __CUDACC__
    using Row = int32_t;
    __device__ __forceinline__ Row row(int32_t i) const { return i; }
    template <typename Fn>
    __device__ __forceinline__ void each(Row i, Fn &&fn) const {
        const int32_t y = i / nx, x = i - y * nx, gy = y + row0;
        const int kind = walls ? (gy == 0 ? 1 : (gy == gny - 1 ? 2 : 0)) : 0;
#pragma unroll
        for (int o = 0; o < 6; ++o) {
            int32_t yy = y + lat_dy(o);
            if (walls && (yy + row0 < 0 || yy + row0 >= gny)) continue;
            // (a slab's halo rows at the ends of its storage wrap onto its
            // own rows: their values feed only halo rows, which the halo
            // exchange replaces)
            yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
            int32_t xx = x + lat_dx(o);
            xx = xx < 0 ? xx + nx : (xx >= nx ? xx - nx : xx);
            if (!chk_idx(xx + nx * yy, n, 1u)) continue;
            fn(xx + nx * yy, c[kind][o][0], c[kind][o][1], c[kind][o][2], c[kind][o][3],
               c[kind][o][4]);
        }
    }
    __device__ __forceinline__ int tag_of(int32_t i) const {
        if (!walls) return 0;
        const int32_t gy = i / nx + row0;
        return gy == 0 ? 2 : (gy == gny - 1 ? 4 : 0);
    }
    __device__ __forceinline__ size_t slot(int32_t i) const {
        const int32_t y = i / nx;
        return (size_t)(i - y * nx) + (size_t)pitch * (size_t)y;
    }
    __device__ __forceinline__ size_t slots() const { return (size_t)pitch * (size_t)ny; }
#endif
};

// Model constants of one state (Sec. 2.1), in the state's precision.
template <typename T>
struct Phys {
    T rho_l, rho_v, beta, kappa, inv_tau_l, inv_tau_v, dt, gx, gy;
    T inv_drho;  // 1 / (rho_l - rho_v)
};

// Storage of the 18 populations of a state: direction pairs interleaved.
// Each population array has S slots (S = N on general meshes, pitch * ny on
// structured ones; slot i of node i, or x + pitch*y).  With Np = S rounded up
// to a multiple of 4 (keeps every pair array 16-byte aligned): h_0 at
// [0, S); the h pairs q = 0..3 of opposite directions (1,3), (2,4), (5,7),
// (6,8) at Np + 2 Np q + 2 i + s, slot s = 0 for 1, 2, 5, 6 and s = 1 for 3,
// 4, 7, 8; g the same from offset 9 Np.  A state buffer holds 18 Np values.
// A pair is one 8-byte (FP32) or 16-byte (FP64) word per node, read and
// streamed together with packed two-wide arithmetic.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int pair_of(int d) { return d == 1 || d == 3 ? 0 : (d == 2 || d == 4 ? 1 : (d == 5 || d == 7 ? 2 : 3)); }
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int slot_of(int d) { return d == 3 || d == 4 || d == 7 || d == 8 ? 1 : 0; }
// first direction of pair q (slot 0): 1, 2, 5, 6
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int pair_dir(int q, int s) { return s == 0 ? (q == 0 ? 1 : (q == 1 ? 2 : (q == 2 ? 5 : 6)))
                                                     : (q == 0 ? 3 : (q == 1 ? 4 : (q == 2 ? 7 : 8))); }
#ifdef __CUDACC__
__host__ __device__
#endif
#ifdef __CUDACC__
__host__ __device__
#endif
inline size_t pad4(size_t n) { return (n + 3) & ~(size_t)3; }
#ifdef __CUDACC__
__host__ __device__
#endif
inline size_t pop_index(int a, size_t i, size_t n) {
    const size_t np = pad4(n);
    const size_t base = a < 9 ? 0 : 9 * np;
    const int d = a % 9;
    return d == 0 ? base + i : base + np + 2 * np * (size_t)pair_of(d) + 2 * i + (size_t)slot_of(d);
}

template <typename T>
struct Fields {
    T *rho, *drx, *dry, *mu, *kx, *ky;  // N each
    // general meshes: the streamed, bounced-back h* of k_rho (population
    // layout: rest at [0, Np), pair q at Np + 2 Np q); nullptr otherwise
    T *hs;
};

}  // namespace felbm

// ---- opaque handles ---------------------------------------------------------

// Opaque storage of one TMA tensor map (CUtensorMap: 128 bytes, 64-byte
// aligned), encoded on the host and read by cp.async.bulk.tensor from
// global memory.
struct alignas(64) TMap {
    unsigned char bytes[128];
};

struct felbm_mesh {
    int64_t n_nodes = 0, n_tri = 0;
    uint32_t flags = 0;
    cudaStream_t stream = nullptr;
    int kind = 0;  // 0 general triangles, 1 structured triangles, 2 general tetrahedra, 3 tet lattice
    felbm::HostCSR host;
    felbm::HostCSR3 host3;
    felbm::Lattice3Info linfo3;
    felbm::StructuredInfo sinfo;
    // device arrays
    int32_t *d_perm = nullptr;
    // general meshes (kinds 0 and 2): rows in slices of 32 nodes, per
    // precision {FP32, FP64} the entries of DevELL / DevELL3.  These and the
    // patches' arrays are uploaded for the first state that reads them
    // (mesh_hold) and stay as long as the mesh.
    int32_t *d_sbase = nullptr;
    void *d_ell[2][4] = {};
    uint8_t *d_deg = nullptr;  // neighbours of each node (kind 0)
    double *d_mass = nullptr;
    uint8_t *d_tag = nullptr;
    // patches of general triangle meshes (HostCSR), with the recovery
    // coefficients a of their rows per precision {FP32, FP64}
    int32_t *d_pnbase = nullptr, *d_pcount = nullptr, *d_pnode = nullptr, *d_pslice = nullptr, *d_psbase = nullptr;
    int32_t *d_pstail = nullptr, *d_ptail = nullptr;
    uint16_t *d_pcol = nullptr;
    void *d_pa[2] = {nullptr, nullptr};
    bool patch_step = false;
    mutable std::mutex lock;  // of the uploads for new states and device_bytes
    int64_t device_bytes = 0;
};

// Population slots per array of a state on mesh m, and the slot of node i
// (internal order).
inline int mesh_dim(const felbm_mesh *m) { return m->kind >= 2 ? 3 : 2; }
inline int mesh_q(const felbm_mesh *m) { return m->kind >= 2 ? 19 : 9; }
inline size_t pop_slots(const felbm_mesh *m) {
    return m->kind == 1 ? (size_t)m->sinfo.pitch * (size_t)m->sinfo.ny : (size_t)m->n_nodes;
}
inline size_t pop_slot(const felbm_mesh *m, size_t i) {
    if (m->kind != 1) return i;
    const size_t nx = (size_t)m->sinfo.nx;
    return i % nx + (size_t)m->sinfo.pitch * (i / nx);
}

struct felbm_state {
    const felbm_mesh *mesh = nullptr;
    felbm_params params{};
    int precision = FELBM_FP64;
    size_t esize = 8;
    void *f[2] = {nullptr, nullptr};  // 18 pad4(N) each, layout of pop_index
    int cur = 0;
    void *scratch = nullptr;          // 6 N: rho, drx, dry, mu, kx, ky
    void *mom = nullptr;              // 4 N: rho, ux, uy, p (internal order)
    double *d_out = nullptr;          // 5 N staging in caller order + reduction partials
    int *d_flag = nullptr;            // bit 0: non-finite field, bit 2: bounded wait gave up
    TMap *d_tmap = nullptr;           // structured meshes: 2 buffers x {h pairs, h rest, g pairs}
    void *halo = nullptr;             // slabs: halo messages send lo, send hi, recv lo, recv hi
    bool have_moments = false;
    int64_t steps_done = 0;
    // profiling: event pairs around launches (felbm_profile_enable)
    bool prof_on = false;
    int prof_stride = 1;                  // time every prof_stride-th launch of a kind
    int64_t prof_seen[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    std::vector<cudaEvent_t> prof_ev;     // 2 per timed launch
    std::vector<int> prof_kind;           // kind of each timed launch
    size_t prof_used = 0;
    int64_t launches[8] = {0, 0, 0, 0, 0, 0, 0, 0};
};

namespace felbm {
// Record the launch of a kernel of the given kind; when profiling, the
// returned event index brackets it (-1: not timed).
int prof_begin(felbm_state *s, int kind);
// Shared helpers of the C ABI (felbm_api.cu) and its 3-D part (felbm_api3.cu).
constexpr int kTotalsBlocks = 304;  // 2 x 152 SMs
int cuda_status(cudaError_t e);
// Upload `bytes` of host data to a new device array of mesh m (counted in
// its device_bytes).
cudaError_t mesh_upload(felbm_mesh *m, void **d, const void *host, size_t bytes);
// Upload `bytes` of host data to the device array *d of mesh m unless it is
// there already, on the mesh's stream and waiting for it (as state creation
// does); *d stays null where that fails.  Under m's lock.
cudaError_t mesh_hold(felbm_mesh *m, void **d, const void *host, size_t bytes);
// Slices of 32 rows: sbase[s] is the first of slice s's rows of 32 entries,
// as many as the longest of its CSR rows.
std::vector<int32_t> ell_slices(int32_t n, const std::vector<int32_t> &rowptr);
bool params_ok(const felbm_params *p);
void mesh_free(felbm_mesh *m);
void state_free(felbm_state *s);
// Tetrahedral meshes (felbm_api3.cu): the state entry points of mesh kind 2.
int state_init3(const felbm_mesh *mesh, const felbm_params *params, const double *rho0,
                const double *u0, const double *p0, felbm_state **out);
void steps3(felbm_state *s, int64_t n);
int moments3(felbm_state *s, double *rho, double *C, double *u, double *p, double *totals);
int export3(felbm_state *s, double *hbar, double *gbar);
int import3(felbm_state *s, const double *hbar, const double *gbar);
// Encode and upload the tensor maps of a state on a structured mesh
// (felbm_tmap.cu); leaves d_tmap null where TMA is not usable.
void lattice_tmaps(felbm_state *s);
void prof_end(felbm_state *s, int slot);
}  // namespace felbm
