// mc_internal.cuh -- structures shared by the kernels and the C ABI layer of
// libmc.so.  Nothing here is visible through include/mc.h.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <set>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/mc.h"
#include "fastdiv.cuh"
#include "philox.cuh"

namespace mc {

constexpr int kMaxChains = 4096;
constexpr int kDefaultThreads = 256;
constexpr int kSu2DefaultThreads = 128; // SU(2) phase kernels (launch bound 256 threads)
constexpr int kMaxOverrelax = 64;   // overrelaxation sweeps per heat-bath sweep
constexpr size_t kAlign = 256;

// Per-chain descriptor of a 2D Ising chain, resident in the workspace.
struct IsingChain {
    uint32_t Lx, Ly;    // extents (even)
    uint32_t W;         // MSC words per row per colour = Lx / 64
    uint32_t T2, T4;    // Metropolis thresholds for dE = 4 and dE = 8 (floor(e^{-beta dE} 2^32))
    PhiloxKey key;      // seed
    uint32_t chain_id;  // Philox counter word 3
    uint32_t runs, run; // grid mode: a column's row pairs in `runs` runs of `run` or, the first ones, one more
    uint64_t spin_off;  // byte offset of the chain's spins in the lattice region
    double beta;        // coupling (the Metropolis-Hastings step of the learned proposal needs it)
    FastDiv div_half;   // by Lx / 2: colour-linear site index -> row
    FastDiv div_inner;  // int8, Lx no multiple of 8: by Lx / 8, the groups inside a row (Lx >= 8)
};

// Per-chain descriptor of a 4D SU(2) chain.
struct Su2Chain {
    int32_t L[4];       // extents, mu = 0 time (all even)
    uint32_t nh;        // sites per parity = N / 2
    float beta;
    PhiloxKey key;
    uint32_t chain_id;
    uint32_t pad0;
    uint64_t link_off;  // byte offset of the links: float4 [parity][mu][nh]
    uint64_t tries_off; // byte offset of the try record: uint8 [s][mu]
    FastDiv div1h, div1, div2, div3; // by L1 / 2, L1, L2, L3: site index -> coordinates
    // Byte distance, within one (parity, mu) link array, of a step along directions 2, 3 and 0 (a step
    // changes the canonical index by an even number, so the index within the parity by half of it), and
    // the bytes of the array: step[2] = 8 L1, step[3] = step[2] L2, step[0] = step[3] L3, bytes = step[0] L0.
    uint32_t step2, step3, step0, bytes;
};

// Device-resident run state: lets one captured CUDA graph be replayed.
struct DevState {
    unsigned long long sweep_base;   // sweeps completed before the running call
    unsigned long long rec_head;     // records written before the running call
    unsigned long long hb_failures;  // SU(2) link updates with every try rejected
    int err_code;                    // first latched device fault (0 = none)
    int err_info;
    unsigned long long pad[4];
};

// Measurement record as kept on the device.  Ising: a = anti-aligned bonds,
// b = up spins (E = 2a - 2N, M = 2b - N are formed on the host).  SU(2): a, b =
// the exact int64 fixed-point sums of the spatial and temporal plaquettes (two's
// complement), from which the host forms P, P_s, P_t in FP64 (the device's FP64
// pipe is narrow, and the measuring thread would hold up the next phase).
constexpr double kPlaqUnfix = 1.0 / 536870912.0; // 2^-29, the unit of the plaquette sums
struct DevRecord {
    long long sweep;
    unsigned long long a, b;
    double d0, d1, d2;
};
static_assert(sizeof(DevRecord) == 48, "record size");

// Device fault codes latched in DevState::err_code.
enum DevErr : int { kErrNone = 0, kErrChainLookup = 1, kErrBounds = 2, kErrTimeout = 3 };

__device__ __forceinline__ void latch_error(DevState *st, int code, int info)
{
    if (atomicCAS(&st->err_code, 0, code) == 0)
        st->err_info = info;
}

// Lattice load policy.  Kernels that never read a location written during the
// same launch use the read-only path (kLdReadOnly).  Kernels whose later phases
// read what earlier phases wrote (possibly on other SMs of the cluster) either
// load through L2, the device's point of coherence (kLdCoherent: the SU(2)
// resident kernel, where L1-cacheable loads measured no faster), or use plain
// loads ordered by the barrier's acquire (kLdPlain: the batch kernel).
constexpr int kLdReadOnly = 0, kLdPlain = 1, kLdCoherent = 2;

// Threads per block of the SU(2) plaquette measurement; each thread measures
// one x1 pair of sites, so a chain of N sites has ceil(N / (2 kPlaqThreads))
// blocks.
constexpr int kPlaqThreads = 128;
// Largest cluster of the SU(2) resident mode (CTAs per chain; 16 is non-portable).
constexpr int kSu2ResidentMaxCluster = 16;
template <int LD, typename T>
__device__ __forceinline__ T lat_load(const T *p)
{
    if (LD == kLdCoherent)
        return __ldcg(p);
    else if (LD == kLdReadOnly)
        return __ldg(p);
    else
        return *p;
}

// Chained launches: the sweep kernels of a call depend each on the one before.
// Launched with programmatic serialisation, a kernel's blocks are set up while its
// predecessor still runs, do what needs nothing from it (chain lookup, index
// arithmetic, random numbers) and wait here for its completion, which makes its
// writes visible to the (plain) loads that follow.  Only then may the next kernel
// start likewise, so that at most one kernel is ever waiting: let off from the
// first instruction, kernels piled up several deep and displaced the running one's
// blocks (3.1 -> 7.3 us per half-sweep of a 2048^2 chain).
//
// The sweep counter is read before the wait.  k_advance writes it at the end of each chunk of a
// call, so the first kernel of a chunk is launched plainly (launch_chained).
//
// A kernel that uses tensor memory releases its successor only after its own allocation,
// and a barrier of the block behind it.  The successor's blocks allocate before they wait, and hold
// what they have until they end: let in earlier, two of them can take all 512 columns of an SM
// on which a block of the running kernel has yet to allocate, and each side waits for the other
// for ever (tcgen05.alloc has no limit).
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait(bool release)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (release)
        chain_release();
}

// Chain of a block of a grid-mode launch: one load (a binary search over the
// offsets is six dependent ones for 64 chains).
struct SweepArgs;
__device__ __forceinline__ int chain_of_block(const SweepArgs &a);

// Largest k in [0, n) with block_start[k] <= b (block_start ascending, [0] = 0).
__device__ __forceinline__ int find_chain(const uint32_t *__restrict__ block_start, int n, uint32_t b)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&block_start[mid]) <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Arguments common to the sweep kernels.
struct SweepArgs {
    const void *chains;          // IsingChain* or Su2Chain*
    const uint32_t *block_start; // grid-mode block offsets per chain (n_chains + 1 entries)
    const uint32_t *block_chain; // chain of each block (n_chains > 1)
    int n_chains;
    char *lattice;               // lattice region base
    DevRecord *series;           // [chain][cap]
    DevState *state;
    long long cap;               // records per chain in the ring
    uint32_t k;                  // sweep offset within the running call
    int measure;                 // 1: this sweep is measured
    uint32_t rec_k;              // index of this record within the running call
    uint8_t *tries;              // SU(2) try record base, or nullptr
    int release;                 // let the next kernel's blocks in once this one's are past chain_wait
};

__device__ __forceinline__ int chain_of_block(const SweepArgs &a)
{
    return a.n_chains == 1 ? 0 : (int)__ldg(&a.block_chain[blockIdx.x]);
}

}  // namespace mc

// Host-side context.  Lives in the global namespace because include/mc.h
// forward-declares `struct mc_ctx`.
struct mc_ctx {
    int kind = 0;
    int layout = 0;
    int n_chains = 0;
    long long cap = 0;
    cudaStream_t stream = nullptr;       // the caller's stream
    cudaStream_t ls = nullptr;           // stream kernels are launched on (== stream, or the
                                         // capture stream while a graph is being recorded)
    cudaStream_t cap_stream = nullptr;   // private non-blocking stream for graph capture/replay
    cudaEvent_t fence_in = nullptr, fence_out = nullptr;
    char *ws = nullptr;
    size_t ws_bytes = 0;
    // carve-out of the workspace
    void *d_chains = nullptr;
    uint32_t *d_block_start = nullptr;   // grid-mode sweep launches: first block of each chain
    uint32_t *d_block_chain = nullptr;   // and the chain of each block (more than one chain)
    uint32_t *d_meas_start = nullptr;    // measurement launches
    char *d_lattice = nullptr;
    mc::DevRecord *d_series = nullptr;
    mc::DevState *d_state = nullptr;
    char *d_staging = nullptr;
    size_t staging_bytes = 0;
    long long *d_partials = nullptr;     // SU(2) Polyakov loop: per-block partial sums (fixed point)
    uint8_t *d_tries = nullptr;
    mc::DevRecord *d_scratch_rec = nullptr; // one record per chain for mc_measure
    // host copies
    std::vector<mc::IsingChain> ising;
    std::vector<mc::Su2Chain> su2;
    std::vector<mc_chain_desc> desc;
    std::vector<uint32_t> block_start, block_chain, meas_start;
    uint32_t grid_blocks = 0, meas_blocks = 0;
    bool row_runs = true;                // Ising grid mode: threads take runs of row pairs (else int8, a group each)
    bool whole_rows = false;             // int8: every chain has rows of whole Philox groups
    // run bookkeeping
    long long sweeps_done = 0;
    long long rec_written = 0, rec_read = 0;
    int mode = MC_MODE_AUTO;
    int threads = mc::kDefaultThreads;
    bool threads_set = false;            // threads chosen by the caller (mc_set_mode), not the default
    bool record_tries = false;
    int n_or = 0;                        // SU(2): overrelaxation sweeps after each heat-bath sweep
    int su2_res_cluster = 0;             // SU(2) resident mode: CTAs per chain (0 = not prepared)
    std::map<std::tuple<long long, int, int, int, bool, int>, cudaGraphExec_t> graphs;
    std::set<std::tuple<long long, int, int, int, bool, int>> swept; // launched once, not recorded yet
    bool in_chunk = false;               // a sweep kernel of the chunk being enqueued has been launched
    mc::DevState state_copy{};           // the run state as of the last check_device
    mc::DevState *h_state = nullptr;     // page-locked block it comes back through, once there have been many
    int checks = 0;
    // kernel timing (mc_profile_enable)
    bool profiling = false;
    std::vector<cudaEvent_t> events; // pairs: [2i] before, [2i+1] after launch i
    size_t events_used = 0;
};

namespace mc {
// Launchers implemented in ising.cu / su2.cu; return a cudaError_t.
cudaError_t ising_init_launch(mc_ctx *c, const mc_chain_desc *desc);
cudaError_t ising_sweep_enqueue(mc_ctx *c, long long n, int every, int mode);
cudaError_t ising_measure_launch(mc_ctx *c, int chain, DevRecord *out);
cudaError_t ising_config_io(mc_ctx *c, int chain, int fmt, void *dev_buf, bool to_lattice);
size_t ising_config_bytes(const IsingChain &ch, int fmt);
bool ising_resident_fits(const mc_ctx *c, int *smem_bytes);
bool ising_resident_auto(const mc_ctx *c);
cudaError_t ising_prepare_resident(mc_ctx *c);
void ising_plan_grid(mc_ctx *c);

cudaError_t su2_init_launch(mc_ctx *c, const mc_chain_desc *desc);
cudaError_t su2_sweep_enqueue(mc_ctx *c, long long n, int every);
cudaError_t su2_measure_launch(mc_ctx *c, int chain, DevRecord *out);
cudaError_t su2_polyakov_launch(mc_ctx *c, int chain, DevRecord *out);
cudaError_t su2_config_io(mc_ctx *c, int chain, void *dev_buf, bool to_lattice);
size_t su2_config_bytes(const Su2Chain &ch);
void su2_plan_grid(mc_ctx *c);
cudaError_t su2_prepare_resident(mc_ctx *c);
cudaError_t su2_resident_enqueue(mc_ctx *c, long long n, int every);

cudaError_t advance_state_launch(mc_ctx *c, long long n, long long recs);

// A validated sweep call in three parts (capi.cu): the mode, and what can be refused before anything is launched (once a
// call: it looks at every chain, ~4 us for 4096); everything enqueued
// on the context's private stream, ordered after the caller's work, the host's counters advanced with each chunk that
// is launched; then the caller's stream made to wait for it.  A group prepares all its members first, and
// starts all of them before the last part.
mc_status sweep_prepare(mc_ctx *c, int &mode);
mc_status sweep_begin(mc_ctx *c, long long n, int every, int mode);
mc_status sweep_end(mc_ctx *c);

// Whether `s` is being captured into a graph of the caller's (with the error message set).  A captured sweep would be
// counted on the host once and run once per launch of the graph, so the sweep counter and the records kept
// would no longer be the device's.
bool refuse_capture(cudaStream_t s);

// Message returned by mc_last_error() on this thread.
void set_last_error(const std::string &msg);

// Launch a kernel chained to the one before it on the stream (chain_wait), or as a plain launch.
template <typename... P, typename... A>
cudaError_t launch_chained_on(cudaStream_t stream, bool chained, void (*kernel)(P...), unsigned blocks, unsigned threads,
                              size_t smem, const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// Launch one sweep kernel on the context's launch stream, chained to the sweep kernel before it: not the
// first of a chunk, which reads what k_advance wrote before it waits, nor between profiling events.
template <typename... P, typename... A>
cudaError_t launch_chained(mc_ctx *c, void (*kernel)(P...), unsigned blocks, unsigned threads, const A &...args)
{
    const bool chained = c->in_chunk && !c->profiling;
    c->in_chunk = true;
    return launch_chained_on(c->ls, chained, kernel, blocks, threads, 0, args...);
}

// Bracket one sweep-kernel launch with events when the context is profiling.
cudaError_t prof_begin(mc_ctx *c);
cudaError_t prof_end(mc_ctx *c);
}  // namespace mc
