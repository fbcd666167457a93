// Many steps of one small simulation in one launch.
//
// A step of a small channel is a chain of short kernels (node update, then
// membrane forces of the next step beside the fluid update), and the launches
// and cross-stream events between them take longer than the kernels: 14.5 us
// a step for one sphere in a 40x20x20 channel, 7 of them between kernels, and
// the host enqueues no faster than 11 us a step.  Here one cooperative launch
// runs all steps of a call, with two barriers over its blocks in each:
//   node update    8 nodes per warp, spread over all blocks (on one SM the
//                  scattered gathers and reductions of a level-3 cell's 642
//                  nodes take 7 us, at about one sector a cycle);
//   [barrier]
//   then, by role  the first blocks: the membrane forces of one object each, for
//                  the next step (and, with repulsion between objects, a
//                  barrier over these blocks and the repulsion on its nodes);
//                  the others: the fluid cells, a warp's 32 or 64 at a time;
//   [barrier]
// The barriers are counters in global memory that only grow (reset before the
// launch), added to after a block barrier and a fence, read with acquire by
// one thread before a block barrier.  All blocks are resident (cooperative
// launch) and arrive at every barrier in order, so every wait ends; as
// everywhere it is bounded all the same (bounded_wait.h): one that runs out
// sets ST_TIMEOUT and the block leaves.  What another block writes during the
// launch is read through the L2 (populations, velocity samples, mask, forces,
// and the positions of an object by its membrane block); a node's own state
// stays with its warp.
#include "bounded_wait.h"
#include "fluid_core.cuh"
#include "ib_core.cuh"

namespace lbib {

// One block per SM.  768 threads (80 registers each) take a level-3 cell's 642
// nodes in one round; the FP32 two-cells update spills at 80 registers, so
// its blocks have 512 (128x64x64 without objects 12.0 us a step against 18.7).
template <typename T, bool PAIR>
constexpr int STEPS_THREADS = sizeof(T) == 4 && PAIR ? 512 : 768;
constexpr unsigned long long STEPS_WAIT_NS = 10000000000ull;

extern __shared__ float steps_smem[];

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long steps_clock() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Until *c has reached target (all threads of the block call it); false when
// the bound ran out.
__device__ __forceinline__ bool steps_wait(uint32_t *status, const unsigned *c, unsigned target,
                                           unsigned long long bound_ns = STEPS_WAIT_NS) {
    bool late = false;
    if (threadIdx.x == 0 && ld_acquire(c) < target) {
        WaitClock clock;
        clock.start(steps_clock());
        for (unsigned i = 1; ld_acquire(c) < target; ++i) {
            if ((i & 1023u) == 0u && clock.over(steps_clock(), bound_ns)) {
                atomicOr(status, ST_TIMEOUT);
                late = true;
                break;
            }
        }
    }
    return __syncthreads_or(late) == 0;
}

__device__ __forceinline__ void steps_signal(unsigned *c) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(c, 1u);
    }
}

// Check of the wait itself: one block waits for a counter that nothing adds to, or
// that it has added to first.
__global__ void k_steps_wait_probe(uint32_t *status, unsigned *c, unsigned long long bound_ns, int arrive) {
    if (arrive) steps_signal(c);
    steps_wait(status, c, 1u, bound_ns);
}

cudaError_t run_steps_wait_probe(uint32_t *status, unsigned *c, unsigned long long bound_ns, int arrive, cudaStream_t st) {
    k_steps_wait_probe<<<1, 64, 0, st>>>(status, c, bound_ns, arrive);
    return cudaGetLastError();
}

// PAIR: two cells per thread (BC: nx odd), else one (BC: obstacles or an inlet)
template <typename T, bool PAIR, bool BC>
__global__ void __launch_bounds__(STEPS_THREADS<T, PAIR>, 1) k_steps(SimDev s, long long t0, int n, unsigned *sync) {
    constexpr int THREADS = STEPS_THREADS<T, PAIR>;
    unsigned *nodes_done = sync, *boxes_done = sync + 16, *done = sync + 32;
    const unsigned blocks = gridDim.x;
    const int nobj = s.nobj, b = (int)blockIdx.x, nfluid = (int)blocks - nobj;
    const int groups = (s.nf + (PAIR ? 63 : 31)) / (PAIR ? 64 : 32);
    for (int k = 0; k < n; ++k) {
        const long long t = t0 + k;
        const int par = (int)(t & 1);
        if (k > 0 && !steps_wait(s.status, done, blocks * (unsigned)k)) return;
        if (nobj > 0) {
            constexpr int L = NODE_LANES<MODE_MANY>;
            for (int i = 32 / L * (int)((threadIdx.x >> 5) * blocks + blockIdx.x); i < s.nn_total; i += THREADS / L * (int)blocks)
                node_step<MODE_MANY>(s, i + (int)(threadIdx.x & 31) / L, par);
            steps_signal(nodes_done);
            if (!steps_wait(s.status, nodes_done, blocks * (unsigned)(k + 1))) return;
        }
        if (b < nobj) {
            membrane_object<false, MODE_MANY>(s, b, steps_smem, BlockTeam());
            if (s.rep_on) {  // the other objects' boxes
                steps_signal(boxes_done);
                if (!steps_wait(s.status, boxes_done, (unsigned)nobj * (unsigned)(k + 1))) return;
                repel_object(s, b, steps_smem);
            }
        } else {
            const uint32_t seed = step_seed(t);
            // groups of a warp's cells, one after the other to different blocks,
            // so that in the last round every block has as many warps at work
            constexpr int GROUP = PAIR ? 64 : 32;
            const int lane = (int)threadIdx.x & 31;
            for (int g = b - nobj + nfluid * (int)(threadIdx.x >> 5); g < groups; g += nfluid * (THREADS / 32)) {
                if constexpr (PAIR) {
                    const int f = GROUP * g + 2 * lane;
                    if (f < s.nf) fluid_pair<T, MODE_MANY, BC>(s, par, f, seed);
                } else {
                    const int f = GROUP * g + lane;
                    if (f < s.nf) fluid_cell<T, BC, MODE_MANY>(s, par, f, active_word(s, f), seed);
                }
            }
        }
        steps_signal(done);
    }
}

// Two cells per thread where the kernel allows; FP32 (the same bits either
// way) only where one cell per thread takes more than two rounds of the
// blocks (64x48x48 with 3 cells 12.1 against 13.0 us a step, without objects 101x37x53
// 5.7 against 6.3; 128x64x64 with 20 cells 17.6 against 15.9) and the objects are not
// so large that the step waits for their membrane blocks, which then have 512
// threads (8 level-4 cells in 128x64x64 27.9 against 31.4).
static bool steps_pair(const SimDev &s, int max_edges) {
    if (fluid_kernel_kind(s) == 0) return false;
    return s.prec != LBIB_POP_F32 ||
           (s.nf > 2 * STEPS_THREADS<float, false> * (device_sms() - s.nobj) && (s.nobj == 0 || max_edges <= 4096));
}
static int steps_tiles(const SimDev &s, int max_edges) {
    const int cells = !steps_pair(s, max_edges)         ? STEPS_THREADS<float, false>
                      : s.prec == LBIB_POP_F32 ? 2 * STEPS_THREADS<float, true>
                                               : 2 * STEPS_THREADS<__half, true>;
    return (s.nf + cells - 1) / cells;
}

// Blocks for the fluid cells: what is left of the SMs, one tile each if that is
// fewer.  Beside objects, whose membrane blocks take as long as two or three
// rounds of tiles, half as many do (64x48x48 with 3 cells: 49 blocks instead of
// 95 at the same time a step), and simulations on other streams find room (8 of
// these on 8 streams 4.5 us a simulation and step against 12.8 with 95 blocks,
// 7.9 with separate launches, which the host bounds).
static int steps_fluid_blocks(const SimDev &s, int max_edges) {
    const int sms = device_sms() - s.nobj, tiles = steps_tiles(s, max_edges);
    if (s.nobj > 0 && tiles > sms / 4 && tiles <= sms) return (tiles + 1) / 2;
    return tiles < sms ? tiles : sms;
}

// Up to 8 rounds of the fluid blocks (6 of the FP32 two-cells blocks, which
// have 16 warps; without objects 5), and objects on half of the SMs at most.
// Without objects from 32 tiles on, and from 64 where a thread has two cells of one
// row (16 bits, even width): a separate launch takes 4.1 us, or 6.2 where the
// kernel is longer, a step of a launch 4.0 to 4.7.  us a step, one launch against separate ones:
//   sphere 40x20x20                 8.2 / 12.7
//   no objects 101x37x53            5.7 /  6.2    128x96x96 FP16  16.7 / 18.6
//     30x32x31 FP32                 4.0 /  4.1    FP16 4.6 / 4.1; 40x40x40 4.0 / 5.7, 4.7 / 4.1; 41x40x39 FP16 5.3 / 6.2
//     48x40x40 FP16                 4.7 /  4.1    48x48x48 4.9 / 5.1, 64x48x48 4.8 / 6.2
//   3 cells 64x48x48 FP16          11.5 / 20.5
//   20 cells 117x70x66 FP32        17.0 / 22.5
//   20 cells 128x64x64 FP32        16.0 / 22.8    FP16  12.9 / 22.1
//   8 level-4 cells 128x64x64 FP32 28.1 / 37.7
//   20 cells 120x80x80 FP32        25.9 / 26.6    160x96x96 FP16  29.3 / 30.9
//   10 bodies with repulsion among posts FP16: 199x50x30 12.8 / 32.4, 200x64x64 26.0 / 33.8
// beyond (6.4 rounds at 96x96x96 FP32 30.6 / 28.8, 9.5 at 160x128x96 FP16 37.3 /
// 37.4) they are equal or worse.
//
// Beside simulations on other streams, half of the SMs at most, so that two such
// launches fit: the blocks hold their SMs while they wait, where separate launches
// fill one simulation's gaps with another's work.  us a simulation and step on 8
// streams, one launch against separate ones:
//   sphere 40x20x20                 2.1 /  4.1    3 cells 64x48x48 FP16  4.3 /  4.8
// and with more SMs
//   20 cells 117x70x66 FP32        17.0 / 15.0    128x64x64 FP16  12.9 / 11.2
//   20 cells 160x96x96 FP16        29.1 / 22.8    8 level-4 cells 128x64x64 FP32 28.1 / 15.5
//   no objects 64x48x48             5.2 /  2.9    101x37x53  5.7 / 4.4    128x96x96 FP16 16.7 / 15.5
bool steps_fit(const SimDev &s, int max_nodes, int max_edges, bool shared) {
    const int sms = device_sms();
    if (shared && 2 * (s.nobj + steps_fluid_blocks(s, max_edges)) > sms) return false;
    if ((s.rep_on && s.nobj > REPEL_MAX_OBJECTS) || (s.nobj > 0 && ib_smem_bytes(max_nodes, max_edges) > IB_SMEM_MAX)) return false;
    const int tiles = steps_tiles(s, max_edges);
    if (s.nobj == 0) {
        const bool row = s.prec != LBIB_POP_F32 && steps_pair(s, max_edges) && s.nx % 2 == 0;
        return tiles >= (row ? 64 : 32) && tiles <= 5 * sms;
    }
    const int rounds = s.prec == LBIB_POP_F32 && steps_pair(s, max_edges) ? 6 : 8;
    return 2 * s.nobj <= sms && tiles <= rounds * (sms - s.nobj);
}

template <typename T, bool PAIR, bool BC>
static cudaError_t launch_steps_t(const SimDev &s, size_t smem, int fluid, long long t, int n, unsigned *sync,
                                  cudaStream_t st) {
    static SmemAttr attr;
    void *fn = (void *)k_steps<T, PAIR, BC>;
    cudaError_t e = attr.ensure(fn, smem, false);
    if (e == cudaSuccess) e = cudaMemsetAsync(sync, 0, 192, st);
    if (e != cudaSuccess) return e;
    SimDev d = s;
    void *args[] = {&d, &t, &n, &sync};
    return cudaLaunchCooperativeKernel(fn, dim3((unsigned)(s.nobj + fluid)), dim3(STEPS_THREADS<T, PAIR>), args, smem, st);
}

template <typename T>
static cudaError_t launch_steps_v(const SimDev &s, int max_nodes, int max_edges, long long t, int n, unsigned *sync,
                                  cudaStream_t st) {
    const size_t smem = s.nobj > 0 ? ib_smem_bytes(max_nodes, max_edges) : 0;
    const int fluid = steps_fluid_blocks(s, max_edges);
    if (steps_pair(s, max_edges)) {
        if (s.nx & 1) return launch_steps_t<T, true, true>(s, smem, fluid, t, n, sync, st);
        return launch_steps_t<T, true, false>(s, smem, fluid, t, n, sync, st);
    }
    if (s.solid || s.in_on) return launch_steps_t<T, false, true>(s, smem, fluid, t, n, sync, st);
    return launch_steps_t<T, false, false>(s, smem, fluid, t, n, sync, st);
}

cudaError_t launch_steps(const SimDev &s, int max_nodes, int max_edges, long long t, int n, unsigned *sync,
                         cudaStream_t st) {
    switch (s.prec) {
        case LBIB_POP_F32: return launch_steps_v<float>(s, max_nodes, max_edges, t, n, sync, st);
        case LBIB_POP_F16S: return launch_steps_v<__half>(s, max_nodes, max_edges, t, n, sync, st);
        default: return launch_steps_v<__nv_bfloat16>(s, max_nodes, max_edges, t, n, sync, st);
    }
}

}  // namespace lbib
