// su2.cu -- 4D SU(2) pure-gauge heat-bath (Sec. 2.4).
//
// Links are the quaternions (U0, U1, U2, U3) of Eq. (4), one float4 per link,
// stored per chain as [parity][mu][site-within-parity] so that the 32 links a
// warp reads for one neighbour direction are 512 contiguous bytes.  Canonical
// site index s = x1 + L1 (x2 + L2 (x3 + L3 x0)) (mu = 0 is time); with L1 even,
// the index of s within its parity class is s >> 1.
//
// One kernel per (parity p, direction mu) phase, in the order of Sec. 2.4
// (mu = 0..3 on odd sites, then on even sites), one thread per site of parity p:
//   1. staple W of Eq. (6), summed over the six nu != mu (the paper's separate
//      staple kernel and its N_vect staple buffer are fused away: W lives in
//      registers only);
//   2. k = |W|, V = W / k, alpha = beta k;
//   3. a0 from Kennedy-Pendleton (up to 8 tries, the "8 attempts per start" of
//      Sec. 2.4), then Creutz (up to 64 tries); a link whose every try fails is
//      left unchanged and counted (still exact: the failure probability depends
//      on alpha only);
//   4. a uniform direction on S^2 for the remaining components;
//   5. U = X V (Eq. (5) with w = X/k) and reprojection onto SU(2) (U / |U|).
// Try t of the link at parity index e uses the Philox block
// (e, sweep, TAG_HB | p<<12 | mu<<8 | t, chain); the direction uses
// (e, sweep, TAG_DIR | p<<12 | mu<<8, chain).  Uniforms are ((r>>8)+1) 2^-24.
// FP32 throughout.  The heat-bath draw keeps the correctly rounded library
// functions (logf, cospif, expm1f, log1pf): a0 = 1 - 2 lambda^2 amplifies their
// error near a0 = 1, and __logf / __cosf there moved single links by more than
// 1e-5.  The normalisations (1 / |W|, |W|, sqrt(1 - a0^2), sin theta) use
// rsqrtf, 1 / (2 alpha) uses __fdividef, and the direction's angle uses
// __sincosf on an argument reduced to (-pi, pi] -- errors of a few 1e-7 per
// link, 5% less time per phase.  Lattice-wide plaquette and Polyakov sums in
// exact int64 fixed point, FP64 only for the final averages.  Site coordinates
// come from magic-number divisions.
#include "su2_dev.cuh"

namespace mc {
namespace {

// Chain descriptors of small batches as kernel parameters: the block's chain is
// found by comparisons with parameters, and the extents, steps, divisors and keys
// come from the constant bank instead of a lookup (by binary search, at that
// time) and some twenty dependent loads per thread: 16 against 20 us per measured sweep of 16 chains of 4^4, 55 against
// 61 for one 4 x 24^3 chain with overrelaxation; no difference where the launch is long
// (4 x 32^4).  Larger batches look the block's chain up in a table in memory.
constexpr int kTableChains = 16;
struct ChainTable {
    uint32_t start[kTableChains]; // first block of each chain (2^32 - 1 past the last)
    Su2Chain ch[kTableChains];
};
struct NoTable {
};

__device__ __forceinline__ const Su2Chain &block_chain(const SweepArgs &, const ChainTable &tab, uint32_t b, int &k, uint32_t &b0)
{
    k = 0;
#pragma unroll
    for (int i = 1; i < kTableChains; ++i)
        k += b >= tab.start[i] ? 1 : 0;
    b0 = tab.start[k];
    return tab.ch[k];
}
__device__ __forceinline__ Su2Chain block_chain(const SweepArgs &a, const NoTable &, uint32_t, int &k, uint32_t &b0)
{
    k = chain_of_block(a);
    b0 = a.block_start[k];
    return static_cast<const Su2Chain *>(a.chains)[k];
}

// The record of this launch's sweep of chain k.
__device__ __forceinline__ DevRecord *sweep_record(const SweepArgs &a, int k)
{
    const unsigned long long slot = (a.state->rec_head + a.rec_k) % (unsigned long long)a.cap;
    return &a.series[(long long)k * a.cap + (long long)slot];
}

// Blocks of up to 256 threads, MINB per SM.  The 18 neighbour links of an update
// are in flight together only when the registers hold them: 64 registers (MINB =
// 4, 32 warps per SM) take 503 us per heat-bath sweep of 4 x 32^4 against 528 with
// 40 registers and 48 warps, and a launch whose blocks are all resident with 85
// (MINB = 3) is shorter still: 8^4 13.5 against 15.1 us per sweep (20.3 with 40
// registers), 20 x 24 x 20 x 24 31.8 against 35.4, but 522 us for 4 x 32^4.  Bound by
// the schedulers' dispatch (~1150 cycles per warp and link: FP32 420, Philox 220,
// the divergent retries 20%) with the DRAM traffic of a 256 MiB lattice at 60% of
// its floor; launch and link-load latency on small lattices.
template <int P, int MU, bool REC, int MINB, typename TAB>
__global__ void __launch_bounds__(256, MINB) k_phase(const __grid_constant__ SweepArgs a, const __grid_constant__ TAB tab)
{
    int k;
    uint32_t b0;
    const auto &ch = block_chain(a, tab, blockIdx.x, k, b0);
    const uint32_t e = (blockIdx.x - b0) * blockDim.x + threadIdx.x;
    if (e >= ch.nh)
        return;
    float4 *U = reinterpret_cast<float4 *>(a.lattice + ch.link_off);
    const PhiloxSchedule ks = philox_schedule(ch.key);
    su2_update_link<P, MU, kLdPlain, REC, false, 3, true>(U, ch, ks, e, (uint32_t)(a.state->sweep_base + a.k), a.tries,
                                                          a.state, a.release != 0);
    if (P == 1 && MU == 0 && a.measure && e == 0) { // the plaquette kernel of this sweep adds into the record
        DevRecord *rec = sweep_record(a, k);
        rec->sweep = (long long)(a.state->sweep_base + a.k);
        rec->a = rec->b = 0;
        rec->d0 = rec->d1 = rec->d2 = 0.0;
    }
}

// Overrelaxation phase: same thread layout as k_phase, no random numbers; 4 blocks
// per SM for the same reason (52 against 55 us per phase of 4 x 32^4, 1.6 against 2.2
// of 8^4 with 40 registers).
template <int P, int MU, typename TAB>
__global__ void __launch_bounds__(256, 4) k_or_phase(const __grid_constant__ SweepArgs a, const __grid_constant__ TAB tab)
{
    int k;
    uint32_t b0;
    const auto &ch = block_chain(a, tab, blockIdx.x, k, b0);
    const uint32_t e = (blockIdx.x - b0) * blockDim.x + threadIdx.x;
    if (e >= ch.nh)
        return;
    float4 *U = reinterpret_cast<float4 *>(a.lattice + ch.link_off);
    su2_overrelax_link<P, MU, kLdPlain, true>(U, ch, e, a.release != 0);
}

// ------------------------------------------------------------------ plaquette
// Sums of (1/2) Tr U_munu(x) of Eq. (3), spatial and temporal separately (the two
// values per measuring thread of Sec. 2.4).  One thread per x1 pair of sites
// (su2_pair_plaquettes), kPlaqThreads pairs per block, at least 6 blocks per SM (80
// registers for the 29 links in flight: 74 us per measurement of 4 x 32^4, 78 with 8
// or 5 blocks, 85 with 4; 96 us for one site per thread): bound by the latency of
// its link loads.  Products in FP32, sums in exact int64
// fixed point (plaq_fixed), so that the blocks add them straight into the
// chain's record in any order.  The record (zeroed by the sweep's first phase) is the
// sweep's, or `out` for chain `only` (zeroed by the caller).
__global__ void __launch_bounds__(kPlaqThreads, 6) k_plaquette(const __grid_constant__ SweepArgs a,
                                                               const uint32_t *meas_start, int only, DevRecord *out)
{
    __shared__ long long ss[kPlaqThreads / 32], st[kPlaqThreads / 32];
    const uint32_t blk = only >= 0 ? meas_start[only] + blockIdx.x : blockIdx.x;
    const int k = only >= 0 ? only : find_chain(meas_start, a.n_chains, blk);
    const Su2Chain ch = static_cast<const Su2Chain *>(a.chains)[k];
    const uint32_t j = (blk - meas_start[k]) * kPlaqThreads + threadIdx.x;
    long long ps = 0, pt = 0;
    chain_wait(a.release != 0);
    if (j < ch.nh)
        su2_pair_plaquettes<kLdPlain>(reinterpret_cast<const float4 *>(a.lattice + ch.link_off), ch, j, ps, pt);
    ps = warp_sum_ll(ps);
    pt = warp_sum_ll(pt);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        ss[w] = ps;
        st[w] = pt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long sa = 0, sb = 0;
        for (int i = 0; i < kPlaqThreads / 32; ++i) {
            sa += ss[i];
            sb += st[i];
        }
        DevRecord *rec = out ? out : sweep_record(a, k);
        atomicAdd(&rec->a, (unsigned long long)sa); // the exact sums; P, P_s, P_t are formed on the host
        atomicAdd(&rec->b, (unsigned long long)sb);
    }
}

// ------------------------------------------------------------------ Polyakov loop
// One thread per spatial site xs = x1 + L1 (x2 + L2 x3): the time-ordered
// product U_0(0, xs) ... U_0(L0 - 1, xs) of FP32 quaternions; (1/2) Tr of an
// SU(2) quaternion is its first component.  Exact fixed-point sums as for the
// plaquette; partial[b] per block, then one block for the chain.
__global__ void __launch_bounds__(256) k_polyakov(Su2Chain ch, const float4 *__restrict__ U, long long *partial)
{
    __shared__ long long sp[8];
    const uint32_t nspace = (uint32_t)ch.L[1] * ch.L[2] * ch.L[3];
    const uint32_t xs = blockIdx.x * blockDim.x + threadIdx.x;
    long long v = 0;
    if (xs < nspace) {
        uint32_t q1, q2, x1, x2, x3;
        fast_divmod(xs, ch.div1, q1, x1);
        fast_divmod(q1, ch.div2, q2, x2);
        x3 = q2;
        const uint32_t sp0 = (x1 + x2 + x3) & 1u;
        float4 P = make_float4(1.f, 0.f, 0.f, 0.f);
        for (int t = 0; t < ch.L[0]; ++t) {
            const uint32_t s = xs + (uint32_t)t * nspace, p = (sp0 + (uint32_t)t) & 1u;
            P = qmul(P, __ldg(&U[(size_t)(p * 4 + 0) * ch.nh + (s >> 1)]));
        }
        v = plaq_fixed(P.x);
    }
    v = warp_sum_ll(v);
    if ((threadIdx.x & 31) == 0)
        sp[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long a = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i)
            a += sp[i];
        partial[blockIdx.x] = a;
    }
}

__global__ void __launch_bounds__(256) k_polyakov_final(const long long *partial, uint32_t nb, uint32_t nspace,
                                                        DevRecord *out)
{
    __shared__ long long sp[8];
    long long a = 0;
    for (uint32_t i = threadIdx.x; i < nb; i += blockDim.x)
        a += partial[i];
    a = warp_sum_ll(a);
    if ((threadIdx.x & 31) == 0)
        sp[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long A = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i)
            A += sp[i];
        out->a = out->b = 0;
        out->d0 = (double)A * kPlaqUnfix / (double)nspace;
        out->d1 = out->d2 = 0.0;
    }
}

// ------------------------------------------------------------------ init / I/O
// Hot start: Haar-random link = normalised 4-vector of four Box-Muller normals
// from the Philox block (s, 0, TAG_INIT | mu, chain); cold start: identity.
__global__ void k_su2_init(Su2Chain ch, float4 *U, int hot)
{
    const uint32_t n = 2 * ch.nh;
    const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 4 * n)
        return;
    const uint32_t s = idx >> 2, mu = idx & 3u;
    float4 v = make_float4(1.f, 0.f, 0.f, 0.f);
    if (hot) {
        const uint4 r = philox4x32_10(make_uint4(s, 0u, kTagSu2Init | mu, ch.chain_id), ch.key);
        const float ra = sqrtf(-2.0f * logf(uniform_open0(r.x)));
        const float rb = sqrtf(-2.0f * logf(uniform_open0(r.z)));
        float sa, ca, sb, cb;
        sincospif(2.0f * uniform_open0(r.y), &sa, &ca);
        sincospif(2.0f * uniform_open0(r.w), &sb, &cb);
        v = make_float4(ra * ca, ra * sa, rb * cb, rb * sb);
        const float inv = rsqrtf(qdot(v, v));
        v = make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
    }
    // parity of s from its coordinates
    uint32_t r = s;
    int x1 = (int)(r % (uint32_t)ch.L[1]);
    r /= (uint32_t)ch.L[1];
    int x2 = (int)(r % (uint32_t)ch.L[2]);
    r /= (uint32_t)ch.L[2];
    int x3 = (int)(r % (uint32_t)ch.L[3]);
    int x0 = (int)(r / (uint32_t)ch.L[3]);
    const int p = (x0 + x1 + x2 + x3) & 1;
    U[(size_t)(p * 4 + mu) * ch.nh + (s >> 1)] = v;
}

// canonical float q[s][mu][4] <-> internal [parity][mu][s >> 1]
__global__ void k_su2_io(Su2Chain ch, float4 *U, float4 *canon, int to_lattice)
{
    const uint32_t n = 2 * ch.nh;
    const uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 4 * n)
        return;
    const uint32_t s = idx >> 2, mu = idx & 3u;
    uint32_t r = s;
    int x1 = (int)(r % (uint32_t)ch.L[1]);
    r /= (uint32_t)ch.L[1];
    int x2 = (int)(r % (uint32_t)ch.L[2]);
    r /= (uint32_t)ch.L[2];
    int x3 = (int)(r % (uint32_t)ch.L[3]);
    int x0 = (int)(r / (uint32_t)ch.L[3]);
    const int p = (x0 + x1 + x2 + x3) & 1;
    float4 *in = &U[(size_t)(p * 4 + mu) * ch.nh + (s >> 1)];
    if (to_lattice)
        *in = canon[idx];
    else
        canon[idx] = *in;
}

inline unsigned blocks_for(size_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int P, bool REC, int MINB, typename TAB>
void launch_phase(mc_ctx *c, const SweepArgs &a, const TAB &tab, int mu)
{
    if (prof_begin(c) != cudaSuccess)
        return;
    const unsigned nt = (unsigned)c->threads;
    switch (mu) {
    case 0: launch_chained(c, k_phase<P, 0, REC, MINB, TAB>, c->grid_blocks, nt, a, tab); break;
    case 1: launch_chained(c, k_phase<P, 1, REC, MINB, TAB>, c->grid_blocks, nt, a, tab); break;
    case 2: launch_chained(c, k_phase<P, 2, REC, MINB, TAB>, c->grid_blocks, nt, a, tab); break;
    default: launch_chained(c, k_phase<P, 3, REC, MINB, TAB>, c->grid_blocks, nt, a, tab); break;
    }
    prof_end(c);
}

template <int P, typename TAB>
void launch_or_phase(mc_ctx *c, const SweepArgs &a, const TAB &tab, int mu)
{
    if (prof_begin(c) != cudaSuccess)
        return;
    const unsigned nt = (unsigned)c->threads;
    switch (mu) {
    case 0: launch_chained(c, k_or_phase<P, 0, TAB>, c->grid_blocks, nt, a, tab); break;
    case 1: launch_chained(c, k_or_phase<P, 1, TAB>, c->grid_blocks, nt, a, tab); break;
    case 2: launch_chained(c, k_or_phase<P, 2, TAB>, c->grid_blocks, nt, a, tab); break;
    default: launch_chained(c, k_or_phase<P, 3, TAB>, c->grid_blocks, nt, a, tab); break;
    }
    prof_end(c);
}

// The phases of one compound sweep: heat-bath, then n_or overrelaxation sweeps,
// each over the odd sites first (Sec. 2.4).  The last phase before a measurement
// keeps the plaquette kernel's blocks out until it is done: set up early they
// crowd the SMs that its own blocks leave first (20 x 24 x 20 x 24: 50 against 60 us
// per measured sweep).
template <bool REC, int MINB, typename TAB>
void launch_sweep(mc_ctx *c, const SweepArgs &a, const TAB &tab)
{
    for (int r = 0; r <= c->n_or; ++r)
        for (int ph = 0; ph < 8; ++ph) {
            SweepArgs b = a;
            b.release = !(a.measure && r == c->n_or && ph == 7);
            if (r == 0 && ph < 4)
                launch_phase<1, REC, MINB>(c, b, tab, ph);
            else if (r == 0)
                launch_phase<0, REC, MINB>(c, b, tab, ph - 4);
            else if (ph < 4)
                launch_or_phase<1>(c, b, tab, ph);
            else
                launch_or_phase<0>(c, b, tab, ph - 4);
        }
}

}  // namespace

// =========================================================================== host
size_t su2_config_bytes(const Su2Chain &ch) { return (size_t)2 * ch.nh * 4 * sizeof(float4); }

// Block tables.  All chains of the batch share each launch: sweeping L2-sized
// groups of chains one after another (to keep each group's links L2-resident
// across its eight phases) was measured slower on 4 x 32^4.
void su2_plan_grid(mc_ctx *c)
{
    c->block_start.assign(c->n_chains + 1, 0);
    c->meas_start.assign(c->n_chains + 1, 0);
    uint32_t acc = 0, macc = 0;
    for (int k = 0; k < c->n_chains; ++k) {
        c->block_start[k] = acc;
        c->meas_start[k] = macc;
        acc += blocks_for(c->su2[k].nh, c->threads);
        macc += blocks_for(c->su2[k].nh, kPlaqThreads);
    }
    c->block_start[c->n_chains] = acc;
    c->meas_start[c->n_chains] = macc;
    c->grid_blocks = acc;
    c->meas_blocks = macc;
}

cudaError_t su2_init_launch(mc_ctx *c, const mc_chain_desc *desc)
{
    for (int k = 0; k < c->n_chains; ++k) {
        const Su2Chain &ch = c->su2[k];
        k_su2_init<<<blocks_for((size_t)8 * ch.nh, 256), 256, 0, c->ls>>>(
            ch, reinterpret_cast<float4 *>(c->d_lattice + ch.link_off), desc[k].start == MC_HOT);
    }
    return cudaGetLastError();
}

static SweepArgs sweep_args(const mc_ctx *c)
{
    SweepArgs a{};
    a.chains = c->d_chains;
    a.block_start = c->d_block_start;
    a.block_chain = c->d_block_chain;
    a.n_chains = c->n_chains;
    a.lattice = c->d_lattice;
    a.series = c->d_series;
    a.state = c->d_state;
    a.cap = c->cap;
    a.tries = c->record_tries ? c->d_tries : nullptr;
    a.release = 1;
    return a;
}

cudaError_t su2_sweep_enqueue(mc_ctx *c, long long n, int every)
{
    SweepArgs a = sweep_args(c);
    ChainTable tab;
    const bool table = c->n_chains <= kTableChains;
    for (int k = 0; table && k < kTableChains; ++k) {
        tab.start[k] = k < c->n_chains ? c->block_start[k] : 0xFFFFFFFFu;
        tab.ch[k] = c->su2[k < c->n_chains ? k : 0];
    }
    // every block resident at 3 x 256 threads per SM: the 85-register phase kernel
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const bool resident = (long long)c->grid_blocks * c->threads <= 768ll * sms;
    for (long long t = 0; t < n; ++t) {
        a.k = (uint32_t)t;
        a.measure = every > 0 && ((t + 1) % every) == 0;
        a.rec_k = a.measure ? (uint32_t)((t + 1) / every - 1) : 0u;
        if (c->record_tries)
            launch_sweep<true, 4>(c, a, NoTable{});
        else if (!table)
            launch_sweep<false, 4>(c, a, NoTable{});
        else if (resident)
            launch_sweep<false, 3>(c, a, tab);
        else
            launch_sweep<false, 4>(c, a, tab);
        if (a.measure)
            launch_chained(c, k_plaquette, c->meas_blocks, (unsigned)kPlaqThreads, a,
                           static_cast<const uint32_t *>(c->d_meas_start), -1, static_cast<DevRecord *>(nullptr));
    }
    return cudaGetLastError();
}

cudaError_t su2_polyakov_launch(mc_ctx *c, int chain, DevRecord *out)
{
    const Su2Chain &ch = c->su2[chain];
    const uint32_t nspace = (uint32_t)ch.L[1] * ch.L[2] * ch.L[3];
    const unsigned nb = (nspace + 255) / 256;
    const float4 *U = reinterpret_cast<const float4 *>(c->d_lattice + ch.link_off);
    k_polyakov<<<nb, 256, 0, c->ls>>>(ch, U, c->d_partials);
    k_polyakov_final<<<1, 256, 0, c->ls>>>(c->d_partials, nb, nspace, out);
    return cudaGetLastError();
}

cudaError_t su2_measure_launch(mc_ctx *c, int chain, DevRecord *out)
{
    const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(DevRecord), c->ls);
    if (e != cudaSuccess)
        return e;
    k_plaquette<<<c->meas_start[chain + 1] - c->meas_start[chain], kPlaqThreads, 0, c->ls>>>(
        sweep_args(c), c->d_meas_start, chain, out);
    return cudaGetLastError();
}

cudaError_t su2_config_io(mc_ctx *c, int chain, void *dev_buf, bool to_lattice)
{
    const Su2Chain &ch = c->su2[chain];
    k_su2_io<<<blocks_for((size_t)8 * ch.nh, 256), 256, 0, c->ls>>>(
        ch, reinterpret_cast<float4 *>(c->d_lattice + ch.link_off), static_cast<float4 *>(dev_buf), to_lattice);
    return cudaGetLastError();
}

}  // namespace mc
