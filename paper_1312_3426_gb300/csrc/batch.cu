// Batched step: many independent simulations advanced together.
//
// A step of the batch is the step of lbib_step (see capi.cu) with every
// kernel launched once for all simulations over a flat work list:
//   node kernel      one block per (simulation, run of nodes of the chunk knob)
//   fluid kernel     one block per (simulation, run of FLUID_THREADS cells or
//                    PAIR_THREADS pairs), one launch per variant present (fluid_group)
//   membrane kernel  one block (or cluster, or group of a block's threads) per
//                    (simulation, object), in one or two launches by size on
//                    streams of their own while the fluid kernel runs (it
//                    prepares the next step)
// so the launch count per step does not grow with the number of
// simulations, and small simulations fill the GPU together.  Every block
// reads its simulation's descriptor and step counter from device arrays;
// the step offset inside a chunk is a kernel argument.  Chunks of
// LBIB_BATCH_GRAPH_STEPS steps are captured once as a CUDA graph (both
// streams) and replayed; a small kernel at the end of the graph advances
// the per-simulation step counters, so one graph serves every chunk of a
// call and later calls on the same set of simulations.
//
// The per-item device code is the code of the single-simulation kernels, so
// a simulation advanced in a batch computes what lbib_step computes for it
// alone, up to the order of the FP32 atomics of the spreading and of the
// repulsion (as between two runs of lbib_step); membrane forces are sums of a
// fixed order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "fluid_core.cuh"
#include "ib_core.cuh"
#include "sim.h"

namespace lbib {

constexpr int LBIB_BATCH_GRAPH_STEPS = 16;  // steps per captured graph
constexpr int FLUID_GROUPS = 10;            // fluid kernel variants (see fluid_group)

extern __shared__ float batch_smem[];

// One launch per storage type and boundary-condition variant present in the
// batch (items grouped by both; BC: obstacles or an inlet).
// L2 prefetch of the sources of work item blockIdx.x + pf of the same
// launch (items of one launch run roughly in index order); CELLS cells per
// item.
template <int ESZ, int CELLS>
__device__ __forceinline__ void prefetch_item(const SimDev *__restrict__ sims, const long long *__restrict__ t_base,
                                              int step_off, const int2 *__restrict__ items, int pf) {
    if (threadIdx.x >= NQ || (int)(blockIdx.x + pf) >= (int)gridDim.x) return;
    const int2 it = items[blockIdx.x + pf];
    const SimDev &s = sims[it.x];
    prefetch_cells<ESZ, CELLS>(s, s.pop[(t_base[it.x] + step_off) & 1], (long long)it.y * CELLS);
}

template <typename T, bool BC>
__global__ void __launch_bounds__(FLUID_THREADS, 5)
    k_batch_fluid(const SimDev *__restrict__ sims, const long long *__restrict__ t_base, int step_off,
                  const int2 *__restrict__ items, int pf) {
    prefetch_item<sizeof(T), FLUID_THREADS>(sims, t_base, step_off, items, pf);
    const int2 it = items[blockIdx.x];  // (simulation, block of cells)
    const SimDev &s = sims[it.x];
    const long long t = t_base[it.x] + step_off;
    fluid_block<T, BC, MODE_PLAIN>(s, (int)(t & 1), it.y * FLUID_THREADS, step_seed(t));
}

// 16-bit storage without obstacles or an inlet: two cells per thread (ODD: nx odd).
template <typename T, bool ODD>
__global__ void __launch_bounds__(PAIR_THREADS, pair_blocks<T>())
    k_batch_fluid_pair(const SimDev *__restrict__ sims, const long long *__restrict__ t_base, int step_off,
                       const int2 *__restrict__ items, int pf) {
    prefetch_item<sizeof(T), 2 * PAIR_THREADS>(sims, t_base, step_off, items, pf);
    const int2 it = items[blockIdx.x];  // (simulation, block of PAIR_THREADS cell pairs)
    const SimDev &s = sims[it.x];
    const long long t = t_base[it.x] + step_off;
    const int f = 2 * (it.y * PAIR_THREADS + (int)threadIdx.x);
    if (f < s.nf) fluid_pair<T, MODE_PLAIN, ODD>(s, (int)(t & 1), f, step_seed(t));
}

// NT nodes per work item (the plan's node chunk), two threads each, as in k_nodes
template <int NT>
__global__ void __launch_bounds__(2 * NT, 512 / NT)
    k_batch_nodes(const SimDev *__restrict__ sims, const long long *__restrict__ t_base, int step_off,
                  const int2 *__restrict__ items) {
    const int2 it = items[blockIdx.x];  // (simulation, first node)
    const SimDev &s = sims[it.x];
    node_step<MODE_PLAIN>(s, it.y + (int)(threadIdx.x >> 1), (int)((t_base[it.x] + step_off) & 1));
}

template <bool EG>
__global__ void __launch_bounds__(1024, 1)
    k_batch_membrane(const SimDev *__restrict__ sims, const int2 *__restrict__ items) {
    cg::cluster_group cl = cg::this_cluster();
    const int2 it = items[blockIdx.x / cl.num_blocks()];  // (simulation, object)
    membrane_object<EG>(sims[it.x], it.y, batch_smem, ClusterTeam());
}

// Several (simulation, object) items per block: group g of block b takes
// item b G + g with its own shared memory and named barrier g + 1.
__global__ void __launch_bounds__(1024, 1)
    k_batch_membrane_groups(const SimDev *__restrict__ sims, const int2 *__restrict__ items, int n_items, int T,
                            int group_floats) {
    const int g = (int)threadIdx.x / T, G = (int)blockDim.x / T;
    const int k = (int)blockIdx.x * G + g;
    if (k >= n_items) return;  // whole groups only
    const int2 it = items[k];
    const GroupTeam tm{(int)threadIdx.x - g * T, T, g + 1};
    membrane_object<false>(sims[it.x], it.y, batch_smem + (size_t)g * group_floats, tm);
}

__global__ void k_batch_advance(long long *t_base, int n, int steps) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) t_base[i] += steps;
}

// A batch plan: device copies of the descriptors and the work lists, and
// the captured graph; rebuilt when the set of simulations, their objects or
// the cluster size change.
struct BatchPlan {
    std::vector<lbib_sim *> sims;
    std::vector<uint64_t> serial;  // identity of each simulation (addresses can be reused)
    std::vector<int> nobj, nn, group;  // group: fluid kernel variant (fluid_group)
    std::vector<SimDev> dev;  // descriptors the device copy holds
    int cluster = 0, device = -1, mthreads = IB_THREADS, nthreads = NODE_CHUNK_DEFAULT, mgroup = 1;
    SimDev *d_sims = nullptr;
    long long *d_t = nullptr;
    int2 *d_items = nullptr;  // fluid (by storage type x obstacles), then node, then membrane items
    int n_flp[FLUID_GROUPS] = {};  // fluid items per kernel variant (see fluid_group)
    int n_fl = 0, n_nd = 0, n_mb = 0;
    int max_nodes = 0, max_edges = 0;
    // size classes of the membrane items (largest first): the n_big items
    // within a factor 2 of the largest, and the rest, whose largest has
    // rest_nodes nodes and rest_edges edges (0: one class)
    int n_big = 0, rest_nodes = 0, rest_edges = 0;
    // threads per object of the two classes by the rule, and whether it holds
    int big_threads = 0, rest_threads = 0;
    bool mrule = false;
    int pf_cell = 0, pf_pair = 0;  // L2 prefetch distances of the fluid launches (work items)
    cudaStream_t aux = nullptr;   // membrane kernel
    cudaStream_t aux2 = nullptr;  // membrane kernel of the smaller size class
    cudaEvent_t ev_rest = nullptr;
    cudaStream_t gst = nullptr;   // graph launches (the caller's stream may be the legacy one, which cannot be captured)
    cudaEvent_t ev_nodes = nullptr, ev_membrane = nullptr, ev_join = nullptr;
    cudaGraphExec_t graph = nullptr;

    void release_graph() {
        if (graph) cudaGraphExecDestroy(graph);
        graph = nullptr;
    }
    void release() {
        release_graph();
        cudaFree(d_sims);
        cudaFree(d_t);
        cudaFree(d_items);
        d_sims = nullptr;
        d_t = nullptr;
        d_items = nullptr;
        sims.clear();
        serial.clear();
        nobj.clear();
        nn.clear();
        group.clear();
        dev.clear();
    }
};

// One plan per process; lbib_batch_step calls are serialised on it.
static BatchPlan g_plan;
static std::mutex g_plan_mu;

// Fluid kernel variant of a simulation: 2 * precision + BC (obstacles or an
// inlet) for the one-cell-per-thread kernels; for 16-bit storage 5 + precision
// for the two-cells kernel, 7 + precision for that of an odd nx.  FP32 takes the
// one-cell kernel here, with 40 warps an SM instead of 20: the boxes of a batch
// are narrow and many, and even and odd widths share a launch (64 mixed channels
// 309.2 us a step against 318.3, 24 channels up to 192x96x96 272.7 against 279.7).
static int fluid_group(const lbib_sim *s) {
    if (s->d.prec != LBIB_POP_F32 && fluid_kernel_kind(s->d) != 0) return (s->d.nx & 1 ? 7 : 5) + s->d.prec;
    return 2 * s->d.prec + (s->d.solid || s->d.in_on ? 1 : 0);
}

static bool plan_matches(lbib_sim *const *sims, int n, int cluster) {
    if ((int)g_plan.sims.size() != n || g_plan.cluster != cluster || g_plan.device != sims[0]->device ||
        g_plan.nthreads != sims[0]->node_threads)
        return false;
    for (int i = 0; i < n; ++i)
        if (g_plan.sims[i] != sims[i] || g_plan.serial[i] != sims[i]->serial ||
            g_plan.nobj[i] != (int)sims[i]->objs.size() || g_plan.group[i] != fluid_group(sims[i]) ||
            g_plan.nn[i] != sims[i]->nn_total)
            return false;
    return true;
}

static cudaError_t build_plan(lbib_sim *const *sims, int n, int cluster, cudaStream_t st) {
    g_plan.release();
    const int nthreads = sims[0]->node_threads;  // of the batch
    if (!g_plan.aux) {
        int lo = 0, hi = 0;
        cudaError_t e = cudaDeviceGetStreamPriorityRange(&lo, &hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&g_plan.aux, cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&g_plan.aux2, cudaStreamNonBlocking, hi);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g_plan.ev_rest, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&g_plan.gst, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g_plan.ev_join, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g_plan.ev_nodes, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g_plan.ev_membrane, cudaEventDisableTiming);
        if (e != cudaSuccess) return e;
    }
    std::vector<int2> flp[FLUID_GROUPS], fl, nd, mb;
    int max_nodes = 0, max_edges = 0;
    for (int i = 0; i < n; ++i) {
        const lbib_sim *s = sims[i];
        const int grp = fluid_group(s);
        const int cells_per_block = grp >= 6 ? 2 * PAIR_THREADS : FLUID_THREADS;
        const int blocks = (s->d.nf + cells_per_block - 1) / cells_per_block;
        for (int b = 0; b < blocks; ++b) flp[grp].push_back(make_int2(i, b));
        if (!s->objs.empty()) {
            for (int f = 0; f < s->nn_total; f += nthreads) nd.push_back(make_int2(i, f));
            for (int o = 0; o < (int)s->objs.size(); ++o) mb.push_back(make_int2(i, o));
            max_nodes = std::max(max_nodes, s->max_nodes);
            max_edges = std::max(max_edges, s->max_edges);
        }
    }
    // largest objects first: their clusters start in the first wave and the
    // small ones fill in behind them (longest-processing-time-first order),
    // so a level-4 cell does not start late and set the launch's tail
    std::stable_sort(mb.begin(), mb.end(), [&](const int2 &a, const int2 &b) {
        return sims[a.x]->objs[a.y].nn > sims[b.x]->objs[b.y].nn;
    });
    for (int k = 0; k < FLUID_GROUPS; ++k) {
        g_plan.n_flp[k] = (int)flp[k].size();
        fl.insert(fl.end(), flp[k].begin(), flp[k].end());
    }
    std::vector<int2> items(fl);
    items.insert(items.end(), nd.begin(), nd.end());
    items.insert(items.end(), mb.begin(), mb.end());
    cudaError_t e;
    if ((e = cudaMalloc(&g_plan.d_sims, n * sizeof(SimDev))) != cudaSuccess) return e;
    if ((e = cudaMalloc(&g_plan.d_t, n * sizeof(long long))) != cudaSuccess) return e;
    if ((e = cudaMalloc(&g_plan.d_items, std::max<size_t>(1, items.size()) * sizeof(int2))) != cudaSuccess) return e;
    if (!items.empty() &&
        (e = cudaMemcpyAsync(g_plan.d_items, items.data(), items.size() * sizeof(int2), cudaMemcpyHostToDevice, st)) !=
            cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    g_plan.sims.assign(sims, sims + n);
    for (int i = 0; i < n; ++i) {
        g_plan.serial.push_back(sims[i]->serial);
        g_plan.group.push_back(fluid_group(sims[i]));
        g_plan.nobj.push_back((int)sims[i]->objs.size());
        g_plan.nn.push_back(sims[i]->nn_total);
    }
    g_plan.n_fl = (int)fl.size();
    g_plan.n_nd = (int)nd.size();
    g_plan.n_mb = (int)mb.size();
    g_plan.cluster = cluster;
    g_plan.nthreads = nthreads;
    g_plan.device = sims[0]->device;
    {
        int sms = 0;
        if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g_plan.device)) != cudaSuccess) return e;
        g_plan.pf_cell = fluid_prefetch(LBIB_POP_F32, 0, sms);  // as in the single-simulation launches
        g_plan.pf_pair = fluid_prefetch(LBIB_POP_F16S, 1, sms);
    }
    g_plan.max_nodes = max_nodes;
    g_plan.max_edges = max_edges;
    auto nodes_of = [&](const int2 &it) { return sims[it.x]->objs[it.y].nn; };
    g_plan.n_big = g_plan.rest_nodes = g_plan.rest_edges = 0;
    while (g_plan.n_big < (int)mb.size() && 2 * nodes_of(mb[g_plan.n_big]) > max_nodes) ++g_plan.n_big;
    for (size_t k = g_plan.n_big; k < mb.size(); ++k) {
        g_plan.rest_nodes = std::max(g_plan.rest_nodes, nodes_of(mb[k]));
        g_plan.rest_edges = std::max(g_plan.rest_edges, sims[mb[k].x]->topo[sims[mb[k].x]->objs[mb[k].y].tid].ne);
    }
    double fluid_us = 0.0;
    for (int i = 0; i < n; ++i) fluid_us += fluid_time_us(sims[i]->d.nf, sims[i]->d.prec);
    g_plan.big_threads = membrane_threads(g_plan.n_big, max_edges, fluid_us);
    g_plan.rest_threads = membrane_threads((int)mb.size() - g_plan.n_big, g_plan.rest_edges, fluid_us);
    return cudaSuccess;
}

static cudaError_t launch_repulsion_batch(cudaStream_t st) {
    for (lbib_sim *s : g_plan.sims) {
        if (!s->d.rep_on) continue;
        cudaError_t e = launch_repulsion(s->d, s->max_nodes, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// shared-memory limits of k_batch_membrane<false>, <true> and the groups kernel
static SmemAttr g_attr_one, g_attr_global, g_attr_groups;

// Membrane items [first, first + n) with up to G per block of T threads each,
// each with a shared-memory slice of `per` bytes (G drops to what fits).
static cudaError_t launch_membrane_groups(cudaStream_t st, int first, int n, size_t per, int G, int T) {
    while (G > 1 && (G * T > 1024 || per * G > IB_SMEM_MAX)) --G;
    const SimDev *sims = g_plan.d_sims;
    const int2 *items = g_plan.d_items + g_plan.n_fl + g_plan.n_nd + first;
    const void *fn = G > 1 ? (const void *)k_batch_membrane_groups : (const void *)k_batch_membrane<false>;
    cudaError_t e = (G > 1 ? g_attr_groups : g_attr_one).ensure(fn, per * G, G == 1);
    if (e != cudaSuccess) return e;
    if (G > 1)
        k_batch_membrane_groups<<<(n + G - 1) / G, G * T, per * G, st>>>(sims, items, n, T, (int)(per / sizeof(float)));
    else
        k_batch_membrane<false><<<n, T, per, st>>>(sims, items);
    return cudaGetLastError();
}

// On `st` (which waits for the node update): the membrane forces, then the
// repulsion.  The objects within a factor 2 of the largest run in one launch
// (their slices sized for the largest) and the others beside it on a second
// stream (slices sized for theirs), so a level-2 object does not hold the
// shared memory of a level-4 one, and each class has threads for its size
// (a step of 64 channels with objects of levels 2 to 4 takes 328 us, of 6
// larger ones 44.6; 390 and 87.5 with one launch of 192 threads per object).
// One launch, one object per cluster, where other threads or another cluster
// size were set without a group, or a block cannot hold an object.
static cudaError_t launch_membrane_batch(cudaStream_t st) {
    if (g_plan.n_mb == 0) return cudaSuccess;
    const int G = g_plan.mgroup;
    const size_t per = ib_smem_bytes(g_plan.max_nodes, g_plan.max_edges);
    const bool own = g_plan.mrule && g_plan.cluster == 1;
    const int T1 = own ? g_plan.big_threads : g_plan.mthreads, T2 = own ? g_plan.rest_threads : g_plan.mthreads;
    if ((G > 1 || own) && g_plan.n_big < g_plan.n_mb && per <= IB_SMEM_MAX) {
        cudaError_t e;
        if ((e = cudaStreamWaitEvent(g_plan.aux2, g_plan.ev_nodes, 0)) != cudaSuccess) return e;
        if ((e = launch_membrane_groups(g_plan.aux2, g_plan.n_big, g_plan.n_mb - g_plan.n_big,
                                        ib_smem_bytes(g_plan.rest_nodes, g_plan.rest_edges), G, T2)) != cudaSuccess)
            return e;
        if ((e = cudaEventRecord(g_plan.ev_rest, g_plan.aux2)) != cudaSuccess) return e;
        if ((e = launch_membrane_groups(st, 0, g_plan.n_big, per, G, T1)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(st, g_plan.ev_rest, 0)) != cudaSuccess) return e;
        return launch_repulsion_batch(st);
    }
    if ((G > 1 || own) && G * T1 <= 1024 && per * G <= IB_SMEM_MAX) {
        cudaError_t e = launch_membrane_groups(st, 0, g_plan.n_mb, per, G, T1);
        return e == cudaSuccess ? launch_repulsion_batch(st) : e;
    }
    const bool global = membrane_in_global(g_plan.max_nodes, g_plan.max_edges, g_plan.cluster);
    const size_t smem = global ? ib_smem_bytes(g_plan.max_nodes, 0) : per;
    cudaError_t e = (global ? g_attr_global : g_attr_one).ensure(
        global ? (const void *)k_batch_membrane<true> : (const void *)k_batch_membrane<false>, smem, true);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g_plan.n_mb * g_plan.cluster));
    cfg.blockDim = dim3((unsigned)g_plan.mthreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)g_plan.cluster;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, global ? k_batch_membrane<true> : k_batch_membrane<false>,
                           (const SimDev *)g_plan.d_sims, (const int2 *)(g_plan.d_items + g_plan.n_fl + g_plan.n_nd));
    // object-object repulsion of the simulations that set it (per simulation)
    return e == cudaSuccess ? launch_repulsion_batch(st) : e;
}

// Steps step_off .. step_off + k - 1 relative to the device step counters,
// on `st` and the plan's second stream; `st` has caught up with the second
// stream at the end.
static cudaError_t enqueue_steps(cudaStream_t st, int step_off, int k) {
    cudaError_t e = cudaSuccess;
    const int2 *fl = g_plan.d_items, *nd = g_plan.d_items + g_plan.n_fl;
    for (int j = 0; j < k && e == cudaSuccess; ++j) {
        const int off = step_off + j;
        if (g_plan.n_nd) {
            switch (g_plan.nthreads) {
                case 32: k_batch_nodes<32><<<g_plan.n_nd, 64, 0, st>>>(g_plan.d_sims, g_plan.d_t, off, nd); break;
                case 64: k_batch_nodes<64><<<g_plan.n_nd, 128, 0, st>>>(g_plan.d_sims, g_plan.d_t, off, nd); break;
                case 128: k_batch_nodes<128><<<g_plan.n_nd, 256, 0, st>>>(g_plan.d_sims, g_plan.d_t, off, nd); break;
                default: k_batch_nodes<256><<<g_plan.n_nd, 512, 0, st>>>(g_plan.d_sims, g_plan.d_t, off, nd); break;
            }
            if ((e = cudaGetLastError()) != cudaSuccess) break;
            if ((e = cudaEventRecord(g_plan.ev_nodes, st)) != cudaSuccess) break;
            if ((e = cudaStreamWaitEvent(g_plan.aux, g_plan.ev_nodes, 0)) != cudaSuccess) break;
            if ((e = launch_membrane_batch(g_plan.aux)) != cudaSuccess) break;
            if ((e = cudaEventRecord(g_plan.ev_membrane, g_plan.aux)) != cudaSuccess) break;
        }
        {
            const int2 *g = fl;
            const int *n = g_plan.n_flp;
            const SimDev *ds = g_plan.d_sims;
            const long long *dt = g_plan.d_t;
            const int p1 = g_plan.pf_cell, p2 = g_plan.pf_pair;
            if (n[0]) k_batch_fluid<float, false><<<n[0], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[0];
            if (n[1]) k_batch_fluid<float, true><<<n[1], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[1];
            if (n[2]) k_batch_fluid<__half, false><<<n[2], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[2];
            if (n[3]) k_batch_fluid<__half, true><<<n[3], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[3];
            if (n[4]) k_batch_fluid<__nv_bfloat16, false><<<n[4], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[4];
            if (n[5]) k_batch_fluid<__nv_bfloat16, true><<<n[5], FLUID_THREADS, 0, st>>>(ds, dt, off, g, p1);
            g += n[5];
            if (n[6]) k_batch_fluid_pair<__half, false><<<n[6], PAIR_THREADS, 0, st>>>(ds, dt, off, g, p2);
            g += n[6];
            if (n[7]) k_batch_fluid_pair<__nv_bfloat16, false><<<n[7], PAIR_THREADS, 0, st>>>(ds, dt, off, g, p2);
            g += n[7];
            if (n[8]) k_batch_fluid_pair<__half, true><<<n[8], PAIR_THREADS, 0, st>>>(ds, dt, off, g, p2);
            g += n[8];
            if (n[9]) k_batch_fluid_pair<__nv_bfloat16, true><<<n[9], PAIR_THREADS, 0, st>>>(ds, dt, off, g, p2);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) break;
        if (g_plan.n_nd) e = cudaStreamWaitEvent(st, g_plan.ev_membrane, 0);
    }
    return e;
}

// Captures LBIB_BATCH_GRAPH_STEPS steps and the advance of the counters
// (on the plan's graph stream).
static cudaError_t capture_graph(cudaStream_t st) {
    g_plan.release_graph();
    cudaError_t e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    cudaError_t e2 = enqueue_steps(st, 0, LBIB_BATCH_GRAPH_STEPS);
    if (e2 == cudaSuccess) {
        const int n = (int)g_plan.sims.size();
        k_batch_advance<<<(n + 127) / 128, 128, 0, st>>>(g_plan.d_t, n, LBIB_BATCH_GRAPH_STEPS);
        e2 = cudaGetLastError();
    }
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(st, &graph);
    if (e2 != cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&g_plan.graph, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    return e;
}

}  // namespace lbib

using namespace lbib;

extern "C" lbib_status lbib_batch_step(lbib_sim *const *sims, int n, int n_steps) {
    if (!sims || n <= 0 || n_steps < 0) return LBIB_ERR_ARG;
    std::lock_guard<std::mutex> plan_lock(g_plan_mu);
    for (int i = 0; i < n; ++i) {
        if (!sims[i]) return LBIB_ERR_ARG;
        if (sims[i]->sticky != LBIB_OK) return sims[i]->sticky;
        if (sims[i]->device != sims[0]->device) return LBIB_ERR_ARG;
        for (int j = 0; j < i; ++j)
            if (sims[j] == sims[i]) return LBIB_ERR_ARG;
    }
    if (cudaSetDevice(sims[0]->device) != cudaSuccess) return LBIB_ERR_CUDA;
    for (int i = 0; i < n; ++i) {
        lbib_status r = sim_prepare_step(sims[i]);
        if (r != LBIB_OK) return r;
    }
    cudaStream_t st = sims[0]->stream;
    // other simulations' pending work (uploads, refreshes, their own second
    // streams) must be done
    for (int i = 0; i < n; ++i) {
        if (sims[i]->stream != st && cudaStreamSynchronize(sims[i]->stream) != cudaSuccess) return LBIB_ERR_CUDA;
        if (cudaStreamSynchronize(sims[i]->aux) != cudaSuccess) return LBIB_ERR_CUDA;
        if (cudaStreamSynchronize(sims[i]->side) != cudaSuccess) return LBIB_ERR_CUDA;
    }
    cudaError_t e = cudaSuccess;
    const int cluster = sims[0]->cluster;
    int max_nodes = 0, max_edges = 0;
    for (int i = 0; i < n; ++i)
        if (!sims[i]->objs.empty()) {
            max_nodes = std::max(max_nodes, sims[i]->max_nodes);
            max_edges = std::max(max_edges, sims[i]->max_edges);
        }
    if (membrane_in_global(max_nodes, max_edges, cluster))
        for (int i = 0; i < n; ++i) {
            const lbib_status r = sims[i]->objs.empty() ? LBIB_OK : sim_edge_scratch(sims[i]);
            if (r != LBIB_OK) return r;
        }
    if (!plan_matches(sims, n, cluster)) e = build_plan(sims, n, cluster, st);
    if (g_plan.mthreads != membrane_block(sims[0]) || g_plan.mgroup != sims[0]->membrane_group ||
        g_plan.mrule != membrane_by_rule(sims[0])) {
        g_plan.mthreads = membrane_block(sims[0]);  // captured in the graph
        g_plan.mgroup = sims[0]->membrane_group;
        g_plan.mrule = membrane_by_rule(sims[0]);
        g_plan.release_graph();
    }
    // descriptors (node arrays may have been reallocated, tables uploaded)
    // and the step counters of this call
    std::vector<long long> tb(n);
    for (int i = 0; i < n; ++i) tb[i] = (long long)sims[i]->t;
    bool same_dev = (int)g_plan.dev.size() == n;
    for (int i = 0; i < n && same_dev; ++i) same_dev = std::memcmp(&g_plan.dev[i], &sims[i]->d, sizeof(SimDev)) == 0;
    if (e == cudaSuccess && !same_dev) {
        // the batched kernels read the descriptors from the device copy, but
        // the repulsion launches of a captured graph hold them by value: a
        // changed descriptor (repulsion switched or retuned, node arrays
        // reallocated) needs a new graph
        g_plan.release_graph();
        g_plan.dev.resize(n);
        for (int i = 0; i < n; ++i) g_plan.dev[i] = sims[i]->d;
        e = cudaMemcpyAsync(g_plan.d_sims, g_plan.dev.data(), n * sizeof(SimDev), cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(g_plan.d_t, tb.data(), n * sizeof(long long), cudaMemcpyHostToDevice, st);
    // membrane forces of the current positions where they are not ready
    bool need_membrane = false;
    for (int i = 0; i < n; ++i) need_membrane |= !sims[i]->objs.empty() && !sims[i]->fel_valid;
    if (e == cudaSuccess && need_membrane && n_steps > 0) {
        // the launch waits for ev_nodes: recorded here, on what st has done
        // so far (a record of the captured graph cannot be waited for)
        e = cudaEventRecord(g_plan.ev_nodes, st);
        if (e == cudaSuccess) e = launch_membrane_batch(st);
    }

    int done = 0;
    while (e == cudaSuccess && done < n_steps) {
        for (int i = 0; i < n && e == cudaSuccess; ++i)
            if (sims[i]->since_mark >= ACTIVE_RESET_STEPS) e = sim_remark(sims[i], st);
        if (e != cudaSuccess) break;
        const int left = n_steps - done;
        const int k = left >= LBIB_BATCH_GRAPH_STEPS ? LBIB_BATCH_GRAPH_STEPS : left;
        if (k == LBIB_BATCH_GRAPH_STEPS) {
            // the graph advances the device counters by its own step count;
            // it runs on the graph stream, ordered after and before `st`
            if (!g_plan.graph) e = capture_graph(g_plan.gst);
            if (e == cudaSuccess) e = cudaEventRecord(g_plan.ev_join, st);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(g_plan.gst, g_plan.ev_join, 0);
            if (e == cudaSuccess) e = cudaGraphLaunch(g_plan.graph, g_plan.gst);
            if (e == cudaSuccess) e = cudaEventRecord(g_plan.ev_join, g_plan.gst);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st, g_plan.ev_join, 0);
        } else {
            e = enqueue_steps(st, 0, k);
        }
        for (int i = 0; i < n; ++i) sims[i]->since_mark += k;
        done += k;
    }
    // host copies of the descriptors and counters must outlive the copies
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        g_plan.release();
        for (int i = 0; i < n; ++i) {
            sims[i]->sticky = LBIB_ERR_CUDA;
            sims[i]->err = std::string("batch step: ") + cudaGetErrorString(e);
        }
        return LBIB_ERR_CUDA;
    }
    for (int i = 0; i < n; ++i) {
        lbib_sim *s = sims[i];
        if (n_steps > 0) {
            s->gmode = (int)((s->t + n_steps - 1) & 1);
            s->t += n_steps;
            if (s->nn_total > 0) {
                s->dev_newer = true;
                s->fel_valid = true;  // the last membrane pass used the final positions
                s->side_ok = false;   // the batch ran on its own streams
            }
        }
    }
    return LBIB_OK;
}
