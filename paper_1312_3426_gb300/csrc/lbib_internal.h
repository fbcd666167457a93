// Internal declarations shared by the translation units of the CUDA library.
//
// Device data layout (one simulation):
//   fluid cells      only the fluid rows are stored; fluid index
//                    f = x + nx * (y' + nyf * z), y' = y - 1 with walls
//                    (nyf = ny - 2), y' = y without (nyf = ny).
//   populations      pop[2][19][nfp] of the storage type, direction-major
//                    (plane stride nfp = nf rounded up to 64 elements), the
//                    deviation h_i = f_i - w_i rho0 (times 2^s for FP16/BF16).
//                    Step t pulls from pop[t&1] and writes pop[(t+1)&1].
//   active cells     bit f of amask[nwords] marks the cells the objects
//                    touch: the 8 interpolation corners of every node, where
//                    it stands and where it will stand at the next step (the
//                    node update marks them, when its lower corner changes,
//                    before the fluid update of the same step).  Marks
//                    persist until a periodic reset, after which all nodes
//                    mark the corners of their position and of the one a
//                    step before (whose force the coming step clears).
//   coupling force   G[2][nf] float4, dense, non-zero only at active cells.
//                    Step t spreads into G[t&1]; the fluid step t adds
//                    G[t&1] at active cells and zeroes G[(t+1)&1] there (the
//                    buffer step t+1 spreads into), so after step t the
//                    buffer of step t is still readable.
//   velocity samples ufield[nf] float4 (u, rho) written by the fluid step at
//                    active cells and read at the node corners by the next
//                    step.
//   nodes            positions and velocities as unevaluated sums of two
//                    FP32 numbers (hi + lo, about 48 significant bits):
//                    Xh, Xl, Vh, Vl each [3][nn_total], structure of arrays,
//                    objects contiguous in id order.
#pragma once

#include <cuda_runtime.h>

#include <mutex>
#include <stdint.h>

#include "lbib.h"

namespace lbib {

constexpr int NQ = 19;
constexpr int FLUID_THREADS = 256;
constexpr int IB_THREADS = 256;          // largest LBIB_TUNE_MEMBRANE_THREADS
// Nodes per block of the node kernel (LBIB_TUNE_NODE_THREADS).  A node waits for two
// rounds of memory, one after the other, and small blocks leave and refill an
// SM one by one (steps with 32 / 64 / 128: 200 cells 256x128x128 FP16 82.9 / 83.1 /
// 83.3 us, 2000 cells FP32 934 / 934 / 937, 24 serving requests 229.9 / 230.6 /
// 231.8; 256 was slower still).
constexpr int NODE_CHUNK_DEFAULT = 64;
constexpr int MAX_TEMPLATE_NODES = 5120;  // k_rep_forces: 36 bytes of shared memory a node
constexpr int ACTIVE_RESET_STEPS = 128;    // period of the active-cell re-marking

// D3Q19 directions of this library: rest, the 6 axis directions in +/- pairs,
// then the 12 face diagonals in +/- pairs; opposite(q) = q+1 for odd q,
// q-1 for even q > 0.
__host__ __device__ constexpr int d3q19_ex(int q) {
    constexpr int t[NQ] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
    return t[q];
}
__host__ __device__ constexpr int d3q19_ey(int q) {
    constexpr int t[NQ] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
    return t[q];
}
__host__ __device__ constexpr int d3q19_ez(int q) {
    constexpr int t[NQ] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
    return t[q];
}
__host__ __device__ constexpr int d3q19_opp(int q) { return q == 0 ? 0 : ((q & 1) ? q + 1 : q - 1); }
__host__ __device__ constexpr double d3q19_w(int q) { return q == 0 ? 1.0 / 3.0 : (q < 7 ? 1.0 / 18.0 : 1.0 / 36.0); }

// Device status bits (sticky per simulation).
enum : uint32_t {
    ST_UNSTABLE = 1u,     // NaN or |u|^2 > 0.09 in a fluid cell
    ST_NODE_NAN = 2u,     // non-finite node position
    ST_TIMEOUT = 4u,      // a bounded device-side wait gave up
    ST_PAIRS = 8u,        // more close object pairs than the repulsion pair list holds
};

// Element lists of one template (device), all node ids local to an object:
//   tri:        (a, b, c, rest area S0 as float bits), inward-ordered, in the
//               mesh's order (read-outs)
struct TplDev {
    int nn, nt;
    const int4 *tri;
};

// Everything the membrane kernel needs of one object, in one record (one
// load instead of object, then template): its nodes, its template's element
// lists (node ids local to the object) and moduli.
//   edge:       per edge (b, c), b < c, in the bank-aware order, three arrays of
//               16-byte vectors, edge_stride apart: (a | b << 16, c | d << 16, t1, t2),
//               where (a,b,c) and (d,c,b) are the inward cyclic orders of the
//               two triangles sharing it, t1 and t2 their numbers where this
//               edge owns them (each triangle is owned by one edge), else -1;
//               (rest length L0, 1/L0, 1/theta0, pi - theta0), theta0 the rest
//               inner angle; the rest areas of t1 and t2 (8-byte vectors)
//   slot:       per slot of the node pass (nodes by number of records, so the
//               lanes of a warp walk equally far; padded to whole warps):
//               (node or -1, its first record, number of records, 0)
//   ring:       the records of the walk around each node v: the next neighbour
//               q (with the RING_START flag), edge (v,q), edge (p,q) opposite v,
//               triangle (v,p,q), p the neighbour before; record j of the 32
//               slots of a warp lie side by side (stride 32).  16 bits each
//               (uint2), or 32 bits (uint4, MEM_WIDE) where a mesh has more
//               than 65536 edges or triangles.  Edges count in the order of
//               `edge`.
constexpr uint32_t RING_START = 0x8000u;  // a fan starts at q: no triangle
enum : int { MEM_NONLINEAR = 1, MEM_ALTITUDE = 2, MEM_WIDE = 4 };
struct alignas(16) MemDev {
    int first, nn, ne, n_slots;
    const int4 *edge;
    const void *ring;
    const int4 *slot;
    int edge_stride, flags;  // MEM_ALTITUDE: local-area force along the altitudes (else centroid -> vertex)
    float ks, kb, kal, kag;
    double Sg0, V0;
    float kv;
    unsigned scal;  // the object's place in SimDev::edge_scal, in 16 bytes
    float pad[2];
};

// One object: its template, first global node, node count and 1/m.
struct ObjDev {
    int tid, first, nn;
    float inv_mass;
};

// Division by a fixed divisor d >= 1 of any 32-bit unsigned n with one
// multiply-high (Granlund and Montgomery, "Division by invariant integers
// using multiplication", PLDI 1994): l = ceil(log2 d),
// m = floor(2^32 (2^l - d) / d) + 1, q = (t + ((n - t) >> 1)) >> (l - 1)
// with t = mulhi(n, m); l = 0 (d = 1) gives q = n.
struct FastDiv {
    uint32_t m;
    int l;
    void init(uint32_t d) {
        l = 0;
        while ((1ull << l) < d) ++l;
        m = (uint32_t)((((1ull << 32) * ((1ull << l) - d)) / d) + 1);
    }
#ifdef __CUDACC__
    __device__ __forceinline__ uint32_t div(uint32_t n) const {
        if (l == 0) return n;
        const uint32_t t = __umulhi(n, m);
        return (t + ((n - t) >> 1)) >> (l - 1);
    }
#endif
};

// Everything a kernel needs to know about one simulation (POD, passed by
// value to single-simulation kernels and stored in an array for batches).
struct SimDev {
    int nx, ny, nz, walls;
    FastDiv div_nx, div_nyf;  // cell index -> (x, row), row -> (y, z)
    int nyf, nf, nfp, nwords;
    int prec;                 // lbib_precision
    float omega, fpre, rho0;  // 1/tau, 1 - 1/(2 tau), rest density
    float gx, gy, gz;         // body force
    float scale, inv_scale;   // 2^s, 2^-s
    float xi;
    void *pop[2];
    float4 *G[2];
    uint32_t *amask;
    float4 *ufield;
    float *Xh, *Xl, *Vh, *Vl; // [3][nn_total] each
    float *Fel;               // [3][nn_total] membrane force of the current step
    char *edge_scal;          // edge and triangle scalars of every object, where shared memory does not serve
    const int *node_obj;      // [nn_total] object of each node
    int nn_total, nobj;
    const ObjDev *obj;
    const float *fext;        // [nobj][3] external force per node of each object
    const TplDev *tpl;
    const MemDev *mem;        // [nobj]
    uint32_t *status;
    double *dropped;          // [3]
    // soft-sphere repulsion (a, n, cutoff): object-object and object-wall
    float rep_a, rep_n, rep_rc;
    float rep_wa, rep_wn, rep_wrc;
    int rep_on, rep_wall_on;
    float *aabb;              // [nobj][8]: min x,y,z, max x,y,z of each object's nodes
    int4 *pairs;              // close object pairs (i | j << 16, image shift x, y, z)
    unsigned *npairs;
    int pair_cap;
    // velocity inlet: cells x in [in_box[0], in_box[1]), y (lattice row, walls
    // included) in [in_box[2], in_box[3]), z in [in_box[4], in_box[5])
    int in_on;
    int in_box[6];
    float in_u[3];
    // obstacle cells (bit per fluid cell, nwords words; null: none): solid
    // like the wall rows; then as many words of near_bit
    const uint32_t *solid;
    int nsolid;
    // 16-bit storage: fluid kernel preference (0 and 1 two cells per thread
    // where the shape allows, 2 the warp-specialised two-cells kernel, 3 one
    // cell per thread)
    int fkern;
};

#ifdef __CUDACC__
__device__ __forceinline__ bool solid_bit(const SimDev &s, int f) {
    return (__ldg(s.solid + (f >> 5)) >> (f & 31)) & 1u;
}
// a neighbour (18 directions, periodic) is an obstacle cell
__device__ __forceinline__ bool near_bit(const SimDev &s, int f) {
    return (__ldg(s.solid + s.nwords + (f >> 5)) >> (f & 31)) & 1u;
}
#endif

// Raises a kernel's dynamic shared-memory limit (and, for cluster kernels,
// allows non-portable cluster sizes) once per device and size; safe to call
// from several threads.
struct SmemAttr {
    std::mutex mu;
    size_t done[64] = {};
    cudaError_t ensure(const void *fn, size_t bytes, bool cluster) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lock(mu);
        if (bytes <= done[dev] && done[dev] != 0) return cudaSuccess;
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e == cudaSuccess && cluster) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess) done[dev] = bytes > 0 ? bytes : 1;
        return e;
    }
};

// How the body of a step runs: by a kernel of its own; by one that may be
// launched early (programmatic dependent launch); or as one of many steps of
// one launch, where populations and velocity samples were written by other
// blocks of the same kernel and have to be read through the L2.
enum : int { MODE_PLAIN = 0, MODE_EARLY = 1, MODE_MANY = 2 };

// ---- programmatic dependent launch -------------------------------------------
// A kernel launched with `pdl` may start while the kernel before it in the
// stream finishes.  It reads, before dep_wait(), only data that no kernel
// still running can be writing (see lbib_step), and after dep_wait() lets
// the next such kernel start (dep_release()).  Without the launch attribute
// both are no-ops.
#if defined(__CUDACC__)
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launches k<<<grid, block, 0, st>>>(args...), with programmatic stream
// serialization when pdl.
template <typename... KArgs, typename... Args>
cudaError_t launch_dep(void (*k)(KArgs...), unsigned grid, unsigned block, cudaStream_t st, bool pdl, Args... args) {
    if (!pdl) {
        k<<<grid, block, 0, st>>>(args...);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}
#endif

// ---- launchers (fluid.cu) -------------------------------------------------
// pdl: launch with programmatic stream serialization (only right after the
// node kernel of the same step)
cudaError_t launch_fluid(const SimDev &s, int par, long long t, cudaStream_t st, bool pdl = false);
// the near_bit words of the obstacle bits
cudaError_t launch_near_bits(const SimDev &s, uint32_t *near, cudaStream_t st);
// the kernel launch_fluid picks (lbib_info out[7]): 0 one cell per thread,
// 1 two cells per thread, 2 warp-specialised two cells per thread
int fluid_kernel_kind(const SimDev &s);
// L2 prefetch distance (in blocks) of a fluid launch of that kernel kind
int fluid_prefetch(int prec, int kind, int sms);
// fluid_tma.cu: the warp-specialised kernel and whether the shape allows it
bool fluid_tma_shape(const SimDev &s);
cudaError_t launch_fluid_tma(const SimDev &s, int par, uint32_t seed, cudaStream_t st);
// the bounded-wait check of fluid_tma.cu (lbib_check_bounded_wait)
cudaError_t run_wait_probe(uint32_t *status, unsigned long long bound_ns, int arrive, cudaStream_t st);
cudaError_t launch_fields(const SimDev &s, int pop_par, int gmode, float *u_full, float *rho_full, int to_ufield,
                          cudaStream_t st);
cudaError_t launch_read_coupling(const SimDev &s, int gpar, float *g_full, cudaStream_t st);
cudaError_t launch_set_coupling(const SimDev &s, int gpar, const float *g_full, cudaStream_t st);
cudaError_t launch_read_pops(const SimDev &s, int pop_par, double *h_full, cudaStream_t st);
cudaError_t launch_set_pops(const SimDev &s, int pop_par, const double *h_full, cudaStream_t st);
cudaError_t launch_mass(const SimDev &s, int pop_par, double *acc, cudaStream_t st);
// allocation-free mass reduction: per-block partials into a static scratch
// array of MASS_SCRATCH_SLOTS doubles (8 KB) per device
constexpr int MASS_SCRATCH_SLOTS = 1024;
constexpr int MASS_SCRATCH_DEVICES = 64;
cudaError_t mass_scratch(double **ptr);
cudaError_t launch_mass_partials(const SimDev &s, int pop_par, double *part, int blocks, cudaStream_t st);

// ---- steps.cu ------------------------------------------------------------
// n steps from step t on in one cooperative launch, where steps_fit; sync:
// 192 device bytes of counters.  The membrane forces of the first step's
// positions are in Fel, and those of the final positions will be.
// shared: simulations on other streams may run beside it
bool steps_fit(const SimDev &s, int max_nodes, int max_edges, bool shared);
cudaError_t launch_steps(const SimDev &s, int max_nodes, int max_edges, long long t, int n, unsigned *sync,
                         cudaStream_t st);
// the bounded-wait check of its barriers (c: a zero counter)
cudaError_t run_steps_wait_probe(uint32_t *status, unsigned *c, unsigned long long bound_ns, int arrive, cudaStream_t st);

// ---- launchers (ib.cu) -----------------------------------------------------
// membrane part: clusters of `cluster` blocks, one per object or at most
// max_clusters (> 0) looping over the objects (max_nodes and max_edges size
// shared memory)
// threads: block size (a multiple of 32, at most 1024)
// group > 1: `group` objects per block of group * threads threads instead
cudaError_t launch_membrane(const SimDev &s, int max_nodes, int max_edges, int cluster, int max_clusters, int threads,
                            int group, cudaStream_t st);
// whether a launch of one object per cluster keeps the edge scalars in
// SimDev::edge_scal: several blocks per object, or more than one block's
// shared memory holds
bool membrane_in_global(int max_nodes, int max_edges, int cluster);
size_t membrane_scalar_bytes(int edges);  // of an object, a multiple of 16
// Threads per object of a membrane launch of nobj objects (one per block)
// beside a fluid update of fluid_us microseconds (0: nothing beside it).
int membrane_threads(int nobj, int max_edges, double fluid_us);
// Whether fewer blocks than objects go through them, with how many blocks and threads.
bool membrane_share(int nobj, int max_nodes, int max_edges, double fluid_us, int &blocks, int &threads);
// Time of the fluid update of nf cells: its populations in and out at 6 TB/s.
inline double fluid_time_us(int64_t nf, int prec) { return (double)nf * 38 * (prec == LBIB_POP_F32 ? 4 : 2) / 6.0e6; }
// SM count of the current device (cached per device)
int device_sms();
// pdl: launch with programmatic stream serialization (only right after the
// previous step's fluid kernel, a mask rebuild or a membrane kernel)
cudaError_t launch_nodes(const SimDev &s, int par, int threads, cudaStream_t st, bool pdl = false);
// object-object repulsion added to Fel (after the membrane kernel, which
// also writes the object bounding boxes); max_nodes sizes shared memory
cudaError_t launch_repulsion(const SimDev &s, int max_nodes, cudaStream_t st);
// oid >= 0: one object into out[14]; oid < 0: every object into out[nobj][14]
cudaError_t launch_mark_all(const SimDev &s, cudaStream_t st);
cudaError_t launch_pack_nodes(const SimDev &s, double *out, cudaStream_t st);
cudaError_t launch_unpack_nodes(const SimDev &s, const double *in, cudaStream_t st);
cudaError_t launch_analyze(const SimDev &s, int oid, double *out, cudaStream_t st);

}  // namespace lbib
