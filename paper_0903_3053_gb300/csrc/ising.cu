// ising.cu -- 2D Ising Metropolis sweep on the red/black checkerboard
// (Eq. (1), Sec. 2.3), two storage layouts:
//
//   int8  : s[y][x] = +-1, one byte per spin.
//   MSC32 : multi-spin coding, 32 spins per 32-bit word and one bit per spin
//           (the paper stores spins as 1-bit variables, Sec. 2.3).  Each
//           colour c has its own plane of Ly rows x W = Lx/64 words; bit b of
//           word w in row y of plane c is the site of colour c with in-row
//           index j = 32 w + b, i.e. x = 2 j + ((y + c) & 1).  With that packing
//           the four neighbours of a whole word are: the same word of the other
//           plane in rows y-1, y and y+1, and the row-y word of the other plane
//           shifted by one bit (towards w-1 or w+1 depending on the row parity).
//           Anti-aligned neighbours are counted bit-sliced for 32 spins at once.
//
// Random numbers: site i = y*(Lx/2) + j of colour c uses word (i & 3) of the
// Philox block with counter (i >> 2, sweep, TAG_METRO | c, chain_id), so the
// stream does not depend on layout, tiling or launch shape.  A spin flips when
// dE = 2 s h <= 0, or when its word is below T[dE] = floor(e^{-beta dE} 2^32)
// (integer thresholds, no floating point on the path).
//
// Execution modes:
//   grid     : one launch per colour over every chain of the batch; the chain of
//              a block is looked up in a table with an entry per block.
//   resident : one CTA per chain holding its whole lattice in shared memory and
//              running all sweeps of a call in one launch (small lattices).
// The energy/magnetisation measurement (the paper's sweep+measure kernels) is
// fused into the colour-1 half-sweep: each colour-1 site counts its
// anti-aligned bonds (every bond joins exactly one colour-1 site) and pairs
// itself with one colour-0 site for the magnetisation; exact integer sums via
// warp reductions and one 64-bit atomic per CTA.
#include <algorithm>
#include <cmath>

#include "ising_dev.cuh"

namespace mc {
namespace {

// ------------------------------------------------------------------ grid mode
// What a thread of an int8 launch takes: a group of any chain, a run of row pairs of
// a group column, or a group of chains that all have rows of whole groups.  A kernel without the
// code for groups over a row's end has the shorter chain of instructions (1024 x 512 4.1
// us per measured sweep against 4.5 with both in one, 1024 x 256 twice 4.5 / 4.8).
enum { kGroups, kRuns, kRows };
template <int C, int LAYOUT, int FORM>
__device__ __forceinline__ void half_sweep(const SweepArgs &a)
{
    const int k = chain_of_block(a);
    const IsingChain ch = static_cast<const IsingChain *>(a.chains)[k];
    const uint32_t t = (blockIdx.x - a.block_start[k]) * blockDim.x + threadIdx.x;
    const uint32_t sweep = (uint32_t)(a.state->sweep_base + a.k);
    const bool measure = (C == 1) && a.measure;
    uint32_t anti = 0, up = 0;
    chain_wait(a.release != 0); // the other colour's half-sweep is done (the run state changes only between chunks)
    if (LAYOUT == MC_LAYOUT_INT8) {
        int8_t *s = reinterpret_cast<int8_t *>(a.lattice + ch.spin_off);
        if (t < int8_units<FORM == kRuns>(ch)) {
            const PhiloxSchedule ks = philox_schedule(ch.key);
            if (measure)
                int8_unit<C, true, FORM == kRuns, kLdPlain, FORM == kRows ? 0 : 4>(s, ch, ks, t, sweep, anti, up);
            else
                int8_unit<C, false, FORM == kRuns, kLdPlain, FORM == kRows ? 0 : 4>(s, ch, ks, t, sweep, anti, up);
        }
    } else {
        const uint32_t W = ch.W, nw = W * ch.Ly;
        uint32_t *base = reinterpret_cast<uint32_t *>(a.lattice + ch.spin_off);
        uint32_t *pc = base + (size_t)C * nw;
        const uint32_t *po = base + (size_t)(1 - C) * nw;
        if (t < W * ch.runs) { // one thread per word column and run of row pairs
            const PhiloxSchedule ks = philox_schedule(ch.key);
            const uint32_t q = fast_div(32 * t, ch.div_half), w = t - q * W; // t / W: half a row is 32 W sites
            const uint32_t yy0 = run_start(ch, q), yy1 = run_start(ch, q + 1);
            if (measure)
                msc_row_pairs<C, true>(pc, po, yy0, yy1, w, ch, ks, sweep, anti, up);
            else
                msc_row_pairs<C, false>(pc, po, yy0, yy1, w, ch, ks, sweep, anti, up);
        }
    }
    if (!a.measure)
        return;
    const long long slot = (long long)((a.state->rec_head + a.rec_k) % (unsigned long long)a.cap);
    DevRecord *rec = &a.series[(long long)k * a.cap + slot];
    if (C == 0) {
        if (t == 0) { // zero the record before the colour-1 kernel accumulates into it
            rec->sweep = (long long)(a.state->sweep_base + a.k);
            rec->a = 0;
            rec->b = 0;
            rec->d0 = rec->d1 = rec->d2 = 0.0;
        }
        return;
    }
    block_sum2(anti, up);
    if (threadIdx.x == 0) {
        atomicAdd(&rec->a, (unsigned long long)anti);
        atomicAdd(&rec->b, (unsigned long long)up);
    }
}

// Two launch-bound flavours of the same half-sweep: blocks of at most 256
// threads with 4 resident per SM (64 registers, so that the Philox key schedule
// stays in registers; the kernel is bound by the schedulers' dispatch, which 32
// warps per SM keep busy: a 32768^2 chain in 32-spin words 730 us per sweep against
// 757 with 8 blocks and 32 registers, int8 groups need them for the bytes loaded ahead) or 5 for
// int8 rows of whole groups (48 registers; with 4 or 8 1024 x 512 takes 4.3 or 4.5 us against
// 4.1), and blocks of up to 1024 threads for callers that ask for them.
template <int C, int LAYOUT, int FORM>
__global__ void __launch_bounds__(256, FORM == kRows ? 5 : 4) k_half_sweep(SweepArgs a)
{
    half_sweep<C, LAYOUT, FORM>(a);
}
template <int C, int LAYOUT, int FORM>
__global__ void __launch_bounds__(1024) k_half_sweep_big(SweepArgs a)
{
    half_sweep<C, LAYOUT, FORM>(a);
}

template <int C, int LAYOUT, int FORM>
void launch_half_sweep(mc_ctx *c, const SweepArgs &a)
{
    launch_chained(c, c->threads <= 256 ? k_half_sweep<C, LAYOUT, FORM> : k_half_sweep_big<C, LAYOUT, FORM>,
                   c->grid_blocks, (unsigned)c->threads, a);
}

// ------------------------------------------------------------------ resident mode
template <int LAYOUT>
__global__ void __launch_bounds__(1024) k_resident(SweepArgs a, uint32_t n_sweeps, uint32_t every)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int k = blockIdx.x;
    const IsingChain ch = static_cast<const IsingChain *>(a.chains)[k];
    const uint32_t bytes = LAYOUT == MC_LAYOUT_INT8 ? ch.Lx * ch.Ly : 8u * ch.Ly * ch.W;
    uint32_t *gl = reinterpret_cast<uint32_t *>(a.lattice + ch.spin_off);
    uint32_t *sl = reinterpret_cast<uint32_t *>(smem);
    __shared__ uint32_t sums[2][2];
    if (threadIdx.x < 4)
        sums[threadIdx.x >> 1][threadIdx.x & 1] = 0;
    const bool nibbles = LAYOUT == MC_LAYOUT_INT8 && (ch.Lx & 7u) == 0;
    const uint32_t G = ch.Lx >> 3, groups = G * ch.Ly; // groups of a colour
    if (nibbles) { // eight sites of a row, both colours, at a time
        const uint2 *g8 = reinterpret_cast<const uint2 *>(gl);
        for (uint32_t u = threadIdx.x; u < groups; u += blockDim.x) {
            const uint32_t odd = fast_div(4 * u, ch.div_half) & 1u;
            const uint2 v = g8[u];
            smem[odd * groups + u] = (uint8_t)nibble_of(__byte_perm(v.x, v.y, 0x6420u));
            smem[(odd ^ 1u) * groups + u] = (uint8_t)nibble_of(__byte_perm(v.x, v.y, 0x7531u));
        }
    } else {
        for (uint32_t u = threadIdx.x; u < bytes / 4; u += blockDim.x)
            sl[u] = gl[u];
    }
    __syncthreads();
    const PhiloxSchedule ks = philox_schedule(ch.key);
    const unsigned long long base = a.state->sweep_base;
    int buf = 0;
    // the next record's slot and the sweeps until it: counted, not divided for (warp 0 writes the record on the way to the
    // next sweep's barrier)
    unsigned long long slot = a.state->rec_head % (unsigned long long)a.cap;
    DevRecord *const series = &a.series[(long long)k * a.cap];
    uint32_t until = every;
    for (uint32_t t = 0; t < n_sweeps; ++t) {
        const uint32_t sweep = (uint32_t)(base + t);
        const bool measure = every != 0 && --until == 0;
        uint32_t anti = 0, up = 0;
        if (nibbles) {
            uint8_t *p0 = smem, *p1 = smem + groups;
            for (uint32_t u = threadIdx.x; u < groups / 2; u += blockDim.x) {
                const uint32_t yy = fast_div(4 * u, ch.div_half);
                nibble_row_pair<0, false>(p0, p1, yy, u - yy * G, ch, ks, sweep, anti, up);
            }
            __syncthreads();
            if (measure) {
                for (uint32_t u = threadIdx.x; u < groups / 2; u += blockDim.x) {
                    const uint32_t yy = fast_div(4 * u, ch.div_half);
                    nibble_row_pair<1, true>(p1, p0, yy, u - yy * G, ch, ks, sweep, anti, up);
                }
            } else {
                for (uint32_t u = threadIdx.x; u < groups / 2; u += blockDim.x) {
                    const uint32_t yy = fast_div(4 * u, ch.div_half);
                    nibble_row_pair<1, false>(p1, p0, yy, u - yy * G, ch, ks, sweep, anti, up);
                }
            }
        } else if (LAYOUT == MC_LAYOUT_INT8) {
            int8_t *s = reinterpret_cast<int8_t *>(smem);
            const uint32_t units = int8_units<false>(ch);
            for (uint32_t u = threadIdx.x; u < units; u += blockDim.x)
                int8_unit<0, false, false, kLdPlain, 1>(s, ch, ks, u, sweep, anti, up);
            __syncthreads();
            if (measure) {
                for (uint32_t u = threadIdx.x; u < units; u += blockDim.x)
                    int8_unit<1, true, false, kLdPlain, 1>(s, ch, ks, u, sweep, anti, up);
            } else {
                for (uint32_t u = threadIdx.x; u < units; u += blockDim.x)
                    int8_unit<1, false, false, kLdPlain, 1>(s, ch, ks, u, sweep, anti, up);
            }
        } else {
            const uint32_t W = ch.W, nw = W * ch.Ly, pairs = W * (ch.Ly >> 1);
            uint32_t *p0 = sl, *p1 = sl + nw;
            for (uint32_t u = threadIdx.x; u < pairs; u += blockDim.x) {
                const uint32_t yy = fast_div(32 * u, ch.div_half), w = u - yy * W;
                msc_row_pair<0, false>(p0, p1, yy, w, ch, ks, sweep, anti, up);
            }
            __syncthreads();
            if (measure) {
                for (uint32_t u = threadIdx.x; u < pairs; u += blockDim.x) {
                    const uint32_t yy = fast_div(32 * u, ch.div_half), w = u - yy * W;
                    msc_row_pair<1, true>(p1, p0, yy, w, ch, ks, sweep, anti, up);
                }
            } else {
                for (uint32_t u = threadIdx.x; u < pairs; u += blockDim.x) {
                    const uint32_t yy = fast_div(32 * u, ch.div_half), w = u - yy * W;
                    msc_row_pair<1, false>(p1, p0, yy, w, ch, ks, sweep, anti, up);
                }
            }
        }
        if (measure) { // the warps add up in the sums' current buffer; no barrier besides the sweep's own
            anti = __reduce_add_sync(0xffffffffu, anti);
            up = __reduce_add_sync(0xffffffffu, up);
            if ((threadIdx.x & 31) == 0) {
                atomicAdd(&sums[buf][0], anti);
                atomicAdd(&sums[buf][1], up);
            }
        }
        __syncthreads();
        if (measure) {
            if (threadIdx.x == 0) {
                DevRecord *rec = &series[slot];
                rec->sweep = (long long)(base + t);
                rec->a = sums[buf][0];
                rec->b = sums[buf][1];
                rec->d0 = rec->d1 = rec->d2 = 0.0;
                sums[buf][0] = sums[buf][1] = 0; // next added to two measurements later, past further barriers
            }
            buf ^= 1;
            until = every;
            slot = slot + 1 == (unsigned long long)a.cap ? 0 : slot + 1;
        }
    }
    if (nibbles) {
        uint2 *g8 = reinterpret_cast<uint2 *>(gl);
        for (uint32_t u = threadIdx.x; u < groups; u += blockDim.x) {
            const uint32_t odd = fast_div(4 * u, ch.div_half) & 1u;
            const uint32_t even_x = bytes_of(smem[odd * groups + u]), odd_x = bytes_of(smem[(odd ^ 1u) * groups + u]);
            g8[u] = make_uint2(__byte_perm(even_x, odd_x, 0x5140u), __byte_perm(even_x, odd_x, 0x7362u));
        }
        return;
    }
    for (uint32_t u = threadIdx.x; u < bytes / 4; u += blockDim.x)
        gl[u] = sl[u];
}

// ------------------------------------------------------------------ init
// Hot start: spin +1 iff the top bit of its random word (sweep field 0, tag
// INIT | colour) is set; cold start: all +1 (Sec. 2.1).
__global__ void k_init_int8(IsingChain ch, int8_t *s, int hot)
{
    const uint32_t n = ch.Lx * ch.Ly;
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const uint32_t y = p / ch.Lx, x = p - y * ch.Lx;
        int8_t v = 1;
        if (hot) {
            const uint32_t c = (x + y) & 1u, i = y * (ch.Lx >> 1) + (x >> 1);
            const uint4 r = philox4x32_10(make_uint4(i >> 2, 0u, kTagIsingInit | c, ch.chain_id), ch.key);
            const uint32_t rr[4] = {r.x, r.y, r.z, r.w};
            v = (rr[i & 3u] >> 31) ? 1 : -1;
        }
        s[p] = v;
    }
}

__global__ void k_init_msc(IsingChain ch, uint32_t *base, int hot)
{
    const uint32_t nw = ch.Ly * ch.W;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < 2 * nw; u += gridDim.x * blockDim.x) {
        const uint32_t c = u / nw, t = u - c * nw, y = t / ch.W, w = t - y * ch.W;
        uint32_t word = 0xFFFFFFFFu;
        if (hot) {
            word = 0;
            const uint32_t blk0 = y * (ch.Lx >> 3) + 8 * w;
            for (int kk = 0; kk < 8; ++kk) {
                const uint4 r = philox4x32_10(make_uint4(blk0 + kk, 0u, kTagIsingInit | c, ch.chain_id), ch.key);
                word |= ((r.x >> 31) << (4 * kk)) | ((r.y >> 31) << (4 * kk + 1)) | ((r.z >> 31) << (4 * kk + 2)) |
                        ((r.w >> 31) << (4 * kk + 3));
            }
        }
        base[u] = word;
    }
}

// ------------------------------------------------------------------ measure (standalone)
template <int LAYOUT>
__global__ void k_measure(IsingChain ch, const char *lat, DevRecord *out)
{
    uint32_t anti = 0, up = 0;
    const uint32_t tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (LAYOUT == MC_LAYOUT_INT8) {
        const int8_t *s = reinterpret_cast<const int8_t *>(lat);
        const uint32_t Lx = ch.Lx, Ly = ch.Ly, half = Lx >> 1, nc = (Lx * Ly) >> 1;
        if (tid < nc) {
            const uint32_t y = tid / half, j = tid - y * half, x = 2 * j + ((y + 1) & 1u);
            const int sv = s[y * Lx + x];
            const int ne = s[y * Lx + inc_wrap(x, Lx)], nw = s[y * Lx + dec_wrap(x, Lx)];
            const int nn = s[dec_wrap(y, Ly) * Lx + x], ns = s[inc_wrap(y, Ly) * Lx + x];
            anti = (ne != sv) + (nw != sv) + (nn != sv) + (ns != sv);
            up = (sv > 0) + (((x & 1u) ? nw : ne) > 0);
        }
    } else {
        const uint32_t W = ch.W, Ly = ch.Ly, nw = W * Ly;
        const uint32_t *p0 = reinterpret_cast<const uint32_t *>(lat), *p1 = p0 + nw;
        if (tid < nw) {
            const uint32_t y = tid / W, w = tid - y * W;
            uint32_t nu, nd, ns, side;
            msc_neighbours<1>(p0, y, w, W, Ly, nu, nd, ns, side);
            const uint32_t s = p1[tid];
            anti = __popc(s ^ nu) + __popc(s ^ nd) + __popc(s ^ ns) + __popc(s ^ side);
            up = __popc(s) + __popc(ns);
        }
    }
    block_sum2(anti, up);
    if (threadIdx.x == 0) {
        atomicAdd(&out->a, (unsigned long long)anti);
        atomicAdd(&out->b, (unsigned long long)up);
    }
}

// ------------------------------------------------------------------ config I/O
// Canonical int8 s[y][x] <-> MSC planes; one thread per MSC word.
__global__ void k_msc_from_int8(IsingChain ch, const int8_t *src, uint32_t *dst)
{
    const uint32_t nw = ch.Ly * ch.W;
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= 2 * nw)
        return;
    const uint32_t c = u / nw, t = u - c * nw, y = t / ch.W, w = t - y * ch.W;
    uint32_t word = 0;
    for (int b = 0; b < 32; ++b) {
        const uint32_t x = 2 * (32 * w + b) + ((y + c) & 1u);
        word |= (uint32_t)(src[y * ch.Lx + x] > 0) << b;
    }
    dst[u] = word;
}

__global__ void k_msc_to_int8(IsingChain ch, const uint32_t *src, int8_t *dst)
{
    const uint32_t nw = ch.Ly * ch.W;
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= 2 * nw)
        return;
    const uint32_t c = u / nw, t = u - c * nw, y = t / ch.W, w = t - y * ch.W;
    const uint32_t word = src[u];
    for (int b = 0; b < 32; ++b) {
        const uint32_t x = 2 * (32 * w + b) + ((y + c) & 1u);
        dst[y * ch.Lx + x] = ((word >> b) & 1u) ? 1 : -1;
    }
}

// Canonical bit rows (bit b of word v of row y = site x = 32 v + b) <-> MSC.
// Even bits of x to its low half and odd bits to its high half (the outer
// perfect unshuffle written as four delta swaps; Warren, "Hacker's Delight",
// Sec. 7-2), and the inverse shuffle.
__device__ __forceinline__ uint32_t bit_unshuffle(uint32_t x)
{
    uint32_t t;
    t = (x ^ (x >> 1)) & 0x22222222u; x ^= t ^ (t << 1);
    t = (x ^ (x >> 2)) & 0x0C0C0C0Cu; x ^= t ^ (t << 2);
    t = (x ^ (x >> 4)) & 0x00F000F0u; x ^= t ^ (t << 4);
    t = (x ^ (x >> 8)) & 0x0000FF00u; x ^= t ^ (t << 8);
    return x;
}
__device__ __forceinline__ uint32_t bit_shuffle(uint32_t x)
{
    uint32_t t;
    t = (x ^ (x >> 8)) & 0x0000FF00u; x ^= t ^ (t << 8);
    t = (x ^ (x >> 4)) & 0x00F000F0u; x ^= t ^ (t << 4);
    t = (x ^ (x >> 2)) & 0x0C0C0C0Cu; x ^= t ^ (t << 2);
    t = (x ^ (x >> 1)) & 0x22222222u; x ^= t ^ (t << 1);
    return x;
}

// Canonical bit rows <-> the two colour planes.  One thread per 64-site chunk u
// = y W + w of a row (canonical words 2u, 2u + 1, read or written once, 8
// contiguous bytes per thread, so that a page-locked host buffer can be read
// or written by the kernel directly): its even-x sites are word u of plane
// y & 1, its odd-x sites word u of the other plane.
__global__ void k_msc_from_bits(IsingChain ch, const uint32_t *src, uint32_t *dst)
{
    const uint32_t nw = ch.Ly * ch.W;
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nw)
        return;
    const uint32_t y = u / ch.W;
    const uint32_t a = bit_unshuffle(src[2 * u]), b = bit_unshuffle(src[2 * u + 1]);
    dst[(y & 1u) * nw + u] = (a & 0xFFFFu) | (b << 16);          // x even
    dst[((y + 1u) & 1u) * nw + u] = (a >> 16) | (b & 0xFFFF0000u); // x odd
}

__global__ void k_msc_to_bits(IsingChain ch, const uint32_t *src, uint32_t *dst)
{
    const uint32_t nw = ch.Ly * ch.W;
    const uint32_t u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u >= nw)
        return;
    const uint32_t y = u / ch.W;
    const uint32_t even = src[(y & 1u) * nw + u], odd = src[((y + 1u) & 1u) * nw + u];
    dst[2 * u] = bit_shuffle((even & 0xFFFFu) | (odd << 16));
    dst[2 * u + 1] = bit_shuffle((even >> 16) | (odd & 0xFFFF0000u));
}

__global__ void k_int8_from_bits(IsingChain ch, const uint32_t *src, int8_t *dst)
{
    const uint32_t n = ch.Lx * ch.Ly;
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n)
        dst[p] = ((src[p >> 5] >> (p & 31u)) & 1u) ? 1 : -1;
}

__global__ void k_int8_to_bits(IsingChain ch, const int8_t *src, uint32_t *dst)
{
    const uint32_t nwords = (ch.Lx * ch.Ly) >> 5;
    const uint32_t v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nwords)
        return;
    uint32_t word = 0;
    for (int b = 0; b < 32; ++b)
        word |= (uint32_t)(src[32 * v + b] > 0) << b;
    dst[v] = word;
}

__global__ void k_advance(DevState *st, unsigned long long n, unsigned long long recs)
{
    st->sweep_base += n;
    st->rec_head += recs;
}

inline unsigned blocks_for(size_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

}  // namespace

// =========================================================================== host
size_t ising_config_bytes(const IsingChain &ch, int fmt)
{
    const size_t n = (size_t)ch.Lx * ch.Ly;
    if (fmt == MC_FMT_INT8)
        return n;
    if (fmt == MC_FMT_BITS)
        return (ch.Lx % 32 == 0) ? n / 8 : 0;
    return 0;
}

// Work units per chain for a grid-mode launch: Philox groups (int8) or row pairs (MSC).
static uint32_t grid_units(const mc_ctx *c, const IsingChain &ch)
{
    if (c->layout == MC_LAYOUT_INT8)
        return c->row_runs ? int8_units<true>(ch) : int8_units<false>(ch);
    return ch.runs * ch.W;
}

// Row pairs per thread: more of them spread a thread's prologue
// (chain lookup, descriptor, indices, key schedule) over more words and load each
// neighbour row once, fewer keep the last wave of blocks even.
// 32-spin words: as many, a power of two up to 8,
// as leave 2^18 threads (1.7 full waves of 1024 threads on 152 SMs).  Measured us
// per measured sweep with 1 / 2 / 4 / 8 row pairs: one 4096^2 chain (131072 row
// pairs) 18.2 / 20.0 / - / -, one 8192^2 or four 4096^2 chains (524288) 54.6 / 52.3 / 57.7 /
// 58.8, one 16384^2 chain (2097152) 199.5 / - / - / 189.2.
// int8: as few waves as 8 allow, filled by runs of two neighbouring lengths, the longer ones first:
// 2048^2 9.7 against 10.8 us with powers of two, 4096^2 23.1 / 25.4, 8192^2 79 / 82, three of 2000 x 1000
// 13.0 / 14.4 (32-spin words: 8192^2 50.1 / 51.2, but four 4096^2 54.9 / 51.3).  int8 chains of fewer than 2^17
// row pairs in all (a 2048 x 1024 lattice) take one group per thread instead: 3.5
// against 4.0 us for 1024 x 512, 5.5 against 4.8 for 1024^2, 11.4 against 10.8 for 2048^2.
constexpr uint64_t kInt8Pairs = 1u << 17;
constexpr uint64_t kRowPairThreads = 1u << 18;
constexpr uint64_t kWaveThreads = 152 * 1024; // 64 registers a thread
constexpr uint64_t kMaxRowPairs = 8;

void ising_plan_grid(mc_ctx *c)
{
    const bool int8 = c->layout == MC_LAYOUT_INT8;
    uint64_t pairs = 0;
    for (const auto &ch : c->ising)
        pairs += (uint64_t)(int8 ? ch.Lx / 8 : ch.W) * (ch.Ly >> 1);
    c->row_runs = !int8 || pairs >= kInt8Pairs;
    c->whole_rows = std::all_of(c->ising.begin(), c->ising.end(), [](const IsingChain &ch) { return (ch.Lx & 7u) == 0; });
    const uint64_t waves = (pairs + kMaxRowPairs * kWaveThreads - 1) / (kMaxRowPairs * kWaveThreads),
                   most = waves * (kWaveThreads / (uint64_t)c->threads);
    double rows = 1.0; // row pairs per thread
    if (int8)
        rows = std::max(1.0, (double)pairs / (double)(waves * kWaveThreads));
    else
        while (rows < (double)kMaxRowPairs && (double)pairs / (2.0 * rows) >= (double)kRowPairThreads)
            rows *= 2.0;
    c->block_start.assign(c->n_chains + 1, 0);
    for (;;) { // int8: until the last wave is not exceeded, or every chain is one block
        uint64_t acc = 0, fit = 0, least = 0; // blocks; those that take runs; chains that do
        for (int k = 0; k < c->n_chains; ++k) {
            IsingChain &ch = c->ising[k];
            const uint32_t np = ch.Ly >> 1;
            ch.runs = int8 ? std::max(1u, (uint32_t)(np / rows)) : (uint32_t)std::ceil(np / rows);
            ch.run = np / ch.runs;
            c->block_start[k] = (uint32_t)acc;
            const uint64_t blocks = blocks_for(grid_units(c, ch), c->threads);
            acc += blocks;
            if ((ch.Lx & 7u) == 0) {
                fit += blocks;
                ++least;
            }
        }
        c->block_start[c->n_chains] = c->grid_blocks = (uint32_t)acc;
        if (!int8 || !c->row_runs || fit <= std::max(most, least) || rows <= 1.0 || rows > 2.0 * (double)kMaxRowPairs)
            break;
        rows *= fit > most + most / 32 ? 1.03 : 1.004;
    }
}

static size_t resident_bytes(const mc_ctx *c, const IsingChain &ch)
{
    return c->layout == MC_LAYOUT_INT8 ? (size_t)ch.Lx * ch.Ly : (size_t)8 * ch.Ly * ch.W;
}

bool ising_resident_fits(const mc_ctx *c, int *smem_bytes)
{
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    size_t need = 0;
    for (const auto &ch : c->ising) {
        const size_t b = resident_bytes(c, ch);
        if (b % 4 != 0)
            return false;
        need = b > need ? b : need;
    }
    if (smem_bytes)
        *smem_bytes = (int)need;
    return need + 1024 <= (size_t)optin;
}

// Automatic choice between the resident and the grid launches: estimated us per
// sweep, from times measured over L = 16 .. 384 and 1 .. 4096 chains.  A resident
// chain costs its sites at one CTA's rate, and chains beyond one per SM queue up; a
// grid sweep costs two chained launches and all sites at the chip's rate.
// Resident / grid, measured us per measured sweep: int8 64^2 x 1 chain 1.25 / 3.1,
// 96^2 x 1 2.4 / 3.1, 128^2 x 1 3.4 / 3.1, 128^2 x 48 3.4 / 4.6, 256^2 x 1 11 / 3.1, 256^2 x 48 11 / 8.7, 256^2 x 152
// 10.7 / 15.0, 64^2 x 4096 20 / 170, 128^2 x 1024 18 / 53, 130^2 (ragged groups) x 1 7.1 / 5.1; 32-spin words 128^2
// x 1 4.3 / 5.4, 256^2 x 1 8.0 / 6.5, 256^2 x 152 8.3 / 10.3, 384^2 x 48 17.9 / 10.3.
bool ising_resident_auto(const mc_ctx *c)
{
    if (!ising_resident_fits(c, nullptr))
        return false;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    double one = 0.0, all = 0.0;
    bool ragged = false;
    for (const auto &ch : c->ising) {
        const double sites = (double)ch.Lx * ch.Ly;
        one = sites > one ? sites : one;
        all += sites;
        ragged = ragged || (ch.Lx & 7u) != 0;
    }
    const double rounds = (double)((c->n_chains + sms - 1) / sms);
    if (c->layout == MC_LAYOUT_MSC32)
        return std::max(4.2, 0.122e-3 * one * rounds) <= 5.4 + 0.6e-6 * all;
    return ragged ? 1.0 + 0.38e-3 * one * rounds <= 4.0 + 4.5e-6 * all
                  : 0.75 + 0.16e-3 * one * rounds <= 3.1 + 1.3e-6 * all;
}

// Threads of a resident CTA: the work units of the largest chain (int8: pairs of groups
// in a row pair, or groups where Lx is no multiple of 8; MSC32: row pairs) rounded up to a warp, at most
// the block size -- the caller's (mc_set_mode), else 1024 when every chain has
// an SM to itself and the default (256) when chains share SMs.  Threads past
// the last unit would idle through every half-sweep and hold the SM's warp
// slots: a 64^2 MSC32 lattice has 32 row pairs, and with one-warp CTAs a batch
// of 4096 such chains is resident on the 152 SMs in one wave (1.23e12 against
// 0.96e12 spin flips/s with 256-thread CTAs, four waves of one working warp
// each).  With a CTA per SM to spare, more threads shorten each half-sweep:
// one 256^2 MSC32 chain 7.8 against 9.2 us.
static int resident_threads(const mc_ctx *c)
{
    uint32_t units = 0;
    for (const auto &ch : c->ising) {
        const uint32_t u = c->layout == MC_LAYOUT_MSC32 ? ch.W * (ch.Ly >> 1)
                           : (ch.Lx & 7u) == 0          ? (ch.Lx >> 3) * (ch.Ly >> 1)
                                                        : int8_units<false>(ch);
        units = u > units ? u : units;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int cap = c->threads_set || c->n_chains > sms ? c->threads : 1024;
    const int t = (int)((units + 31) / 32 * 32);
    return t < 32 ? 32 : (t < cap ? t : cap);
}

static void (*resident_kernel(const mc_ctx *c))(SweepArgs, uint32_t, uint32_t)
{
    return c->layout == MC_LAYOUT_INT8 ? k_resident<MC_LAYOUT_INT8> : k_resident<MC_LAYOUT_MSC32>;
}

// Raise the dynamic shared-memory limit of the resident kernels (outside any
// graph capture).
cudaError_t ising_prepare_resident(mc_ctx *c)
{
    int smem = 0;
    if (!ising_resident_fits(c, &smem))
        return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(resident_kernel(c), cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

cudaError_t ising_init_launch(mc_ctx *c, const mc_chain_desc *desc)
{
    for (int k = 0; k < c->n_chains; ++k) {
        const IsingChain &ch = c->ising[k];
        char *p = c->d_lattice + ch.spin_off;
        if (c->layout == MC_LAYOUT_INT8) {
            k_init_int8<<<blocks_for((size_t)ch.Lx * ch.Ly, 256), 256, 0, c->ls>>>(
                ch, reinterpret_cast<int8_t *>(p), desc[k].start == MC_HOT);
        } else {
            k_init_msc<<<blocks_for((size_t)2 * ch.Ly * ch.W, 256), 256, 0, c->ls>>>(
                ch, reinterpret_cast<uint32_t *>(p), desc[k].start == MC_HOT);
        }
    }
    return cudaGetLastError();
}

cudaError_t advance_state_launch(mc_ctx *c, long long n, long long recs)
{
    k_advance<<<1, 1, 0, c->ls>>>(c->d_state, (unsigned long long)n, (unsigned long long)recs);
    return cudaGetLastError();
}

cudaError_t ising_sweep_enqueue(mc_ctx *c, long long n, int every, int mode)
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
    a.tries = nullptr;
    a.release = 1;
    if (mode == MC_MODE_RESIDENT) {
        int smem = 0;
        if (!ising_resident_fits(c, &smem))
            return cudaErrorInvalidValue;
        const int threads = resident_threads(c);
        cudaError_t e = prof_begin(c);
        if (e != cudaSuccess)
            return e;
        resident_kernel(c)<<<c->n_chains, threads, smem, c->ls>>>(a, (uint32_t)n, (uint32_t)every);
        e = cudaGetLastError();
        if (e != cudaSuccess)
            return e;
        return prof_end(c);
    }
    for (long long t = 0; t < n; ++t) {
        a.k = (uint32_t)t;
        a.measure = every > 0 && ((t + 1) % every) == 0;
        a.rec_k = a.measure ? (uint32_t)((t + 1) / every - 1) : 0u;
        for (int colour = 0; colour < 2; ++colour) {
            cudaError_t e = prof_begin(c);
            if (e != cudaSuccess)
                return e;
            if (c->layout == MC_LAYOUT_MSC32)
                (colour == 0 ? launch_half_sweep<0, MC_LAYOUT_MSC32, kRuns> : launch_half_sweep<1, MC_LAYOUT_MSC32, kRuns>)(c, a);
            else if (c->row_runs)
                (colour == 0 ? launch_half_sweep<0, MC_LAYOUT_INT8, kRuns> : launch_half_sweep<1, MC_LAYOUT_INT8, kRuns>)(c, a);
            else if (c->whole_rows)
                (colour == 0 ? launch_half_sweep<0, MC_LAYOUT_INT8, kRows> : launch_half_sweep<1, MC_LAYOUT_INT8, kRows>)(c, a);
            else
                (colour == 0 ? launch_half_sweep<0, MC_LAYOUT_INT8, kGroups>
                             : launch_half_sweep<1, MC_LAYOUT_INT8, kGroups>)(c, a);
            e = prof_end(c);
            if (e != cudaSuccess)
                return e;
        }
    }
    return cudaGetLastError();
}

cudaError_t ising_measure_launch(mc_ctx *c, int chain, DevRecord *out)
{
    const IsingChain &ch = c->ising[chain];
    const char *lat = c->d_lattice + ch.spin_off;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(DevRecord), c->ls);
    if (e != cudaSuccess)
        return e;
    if (c->layout == MC_LAYOUT_INT8)
        k_measure<MC_LAYOUT_INT8><<<blocks_for(((size_t)ch.Lx * ch.Ly) >> 1, 256), 256, 0, c->ls>>>(ch, lat, out);
    else
        k_measure<MC_LAYOUT_MSC32><<<blocks_for((size_t)ch.Ly * ch.W, 256), 256, 0, c->ls>>>(ch, lat, out);
    return cudaGetLastError();
}

cudaError_t ising_config_io(mc_ctx *c, int chain, int fmt, void *buf, bool to_lattice)
{
    const IsingChain &ch = c->ising[chain];
    char *lat = c->d_lattice + ch.spin_off;
    const size_t n = (size_t)ch.Lx * ch.Ly;
    if (c->layout == MC_LAYOUT_INT8) {
        if (fmt == MC_FMT_INT8) // buf: device memory or page-locked host memory
            return to_lattice ? cudaMemcpyAsync(lat, buf, n, cudaMemcpyDefault, c->ls)
                              : cudaMemcpyAsync(buf, lat, n, cudaMemcpyDefault, c->ls);
        if (to_lattice)
            k_int8_from_bits<<<blocks_for(n, 256), 256, 0, c->ls>>>(ch, static_cast<const uint32_t *>(buf),
                                                                        reinterpret_cast<int8_t *>(lat));
        else
            k_int8_to_bits<<<blocks_for(n / 32, 256), 256, 0, c->ls>>>(ch, reinterpret_cast<const int8_t *>(lat),
                                                                           static_cast<uint32_t *>(buf));
        return cudaGetLastError();
    }
    const size_t words = (size_t)2 * ch.Ly * ch.W;
    uint32_t *msc = reinterpret_cast<uint32_t *>(lat);
    if (fmt == MC_FMT_INT8) {
        if (to_lattice)
            k_msc_from_int8<<<blocks_for(words, 256), 256, 0, c->ls>>>(ch, static_cast<const int8_t *>(buf), msc);
        else
            k_msc_to_int8<<<blocks_for(words, 256), 256, 0, c->ls>>>(ch, msc, static_cast<int8_t *>(buf));
    } else {
        if (to_lattice)
            k_msc_from_bits<<<blocks_for(words / 2, 256), 256, 0, c->ls>>>(ch, static_cast<const uint32_t *>(buf), msc);
        else
            k_msc_to_bits<<<blocks_for(words / 2, 256), 256, 0, c->ls>>>(ch, msc, static_cast<uint32_t *>(buf));
    }
    return cudaGetLastError();
}

}  // namespace mc
