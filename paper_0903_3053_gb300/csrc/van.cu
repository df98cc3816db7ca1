// van.cu -- the learned global proposal: masked autoregressive conv net
// (forward, backward, Adam), autoregressive sampler, and the symmetrised
// Metropolis-Hastings round over the chains of an Ising context.  See
// van_dev.cuh for the network.  The paper has no learned component.
#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "tc_dev.cuh"
#include "van_dev.cuh"

using bf16 = __nv_bfloat16;

namespace mc {
namespace van {
namespace {

// Per-CTA partial gradient of a hidden layer (13 x 32 x 32 weights + 32 biases)
// and the most CTAs k_dw32_tc is launched with.
constexpr int kDwPart = kTapsB * kCh * kCh + kCh;
constexpr int kMaxDwBlocks = 512;

// ------------------------------------------------------------------ parameters
// Canonical FP32 parameter layout (the same as the FP64 oracle): for each layer
// l, W[o][i][5][5] then b[o]; cin = 1 for l = 0, cout = 1 for l = D - 1.
struct ParamLayout {
    int D;
    size_t w_off[kMaxDepth], b_off[kMaxDepth], total;
};

__host__ __device__ inline int layer_cin(int l) { return l == 0 ? 1 : kCh; }
__host__ __device__ inline int layer_cout(int l, int D) { return l == D - 1 ? 1 : kCh; }

ParamLayout param_layout(int D)
{
    ParamLayout p{};
    p.D = D;
    size_t off = 0;
    for (int l = 0; l < D; ++l) {
        p.w_off[l] = off;
        off += (size_t)layer_cout(l, D) * layer_cin(l) * 25;
        p.b_off[l] = off;
        off += (size_t)layer_cout(l, D);
    }
    p.total = off;
    return p;
}

struct DevParams {
    size_t w_off[kMaxDepth], b_off[kMaxDepth];
    int D;
};

__device__ __forceinline__ size_t canon_w(const DevParams &P, int l, int o, int i, int dy, int dx)
{
    return P.w_off[l] + (((size_t)o * layer_cin(l) + i) * 5 + (dy + 2)) * 5 + (dx + 2);
}

// Kernel-side copies of the weights, rounded to BF16: hidden layers as
// [l][tap][o][c] (BF16), layer 1 as [o][tap] and the last layer as [tap][c]
// (FP32 holding BF16-rounded values), biases FP32.
__global__ void k_prep_weights(const float *p, DevParams P, bf16 *wh, float *w1, float *wD, float *bias)
{
    const int D = P.D;
    const int nh = (D - 2) * kTapsB * kCh * kCh;
    const int total = nh + kCh * kTapsA + kTapsB * kCh + (D - 1) * kCh + 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        if (i < nh) {
            const int l = 1 + i / (kTapsB * kCh * kCh), r = i % (kTapsB * kCh * kCh);
            const int t = r / (kCh * kCh), o = (r / kCh) % kCh, c = r % kCh;
            wh[i] = __float2bfloat16(p[canon_w(P, l, o, c, tap_dy(t), tap_dx(t))]);
        } else if (i < nh + kCh * kTapsA) {
            const int r = i - nh, o = r / kTapsA, t = r % kTapsA;
            w1[r] = bf(__float2bfloat16(p[canon_w(P, 0, o, 0, tap_dy(t), tap_dx(t))]));
        } else if (i < nh + kCh * kTapsA + kTapsB * kCh) {
            const int r = i - nh - kCh * kTapsA, t = r / kCh, c = r % kCh;
            wD[r] = bf(__float2bfloat16(p[canon_w(P, D - 1, 0, c, tap_dy(t), tap_dx(t))]));
        } else {
            const int r = i - nh - kCh * kTapsA - kTapsB * kCh; // biases: layers 0..D-2 x 32, then the last
            const int l = r / kCh, o = r % kCh;
            bias[r] = l < D - 1 ? p[P.b_off[l] + o] : p[P.b_off[D - 1]];
        }
    }
}

// ------------------------------------------------------------------ forward
constexpr int kTcMaxPolls = 1 << 22; // bounded completion wait

// BF16 pair <-> two floats as plain bit operations (BF16 -> FP32 is exact);
// the pack rounds to nearest even, lo in the low half.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t u;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(u) : "f"(hi), "f"(lo));
    return u;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&d);
}
// max(., 0) of the pair: the same bits as packing max(lo, 0), max(hi, 0)
__device__ __forceinline__ uint32_t relu_pack(float lo, float hi)
{
    uint32_t u = pack_bf16x2(lo, hi);
    asm("max.bf16x2 %0, %0, %1;" : "+r"(u) : "r"(0u));
    return u;
}
__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// A lane's row of 128 bytes (two positions) to and from global memory, 32 bytes an instruction: whole sectors, so
// that rows stored by their own lanes need no detour through shared memory, whose bandwidth the
// convolutions' operands want.  L = 64, batch 512, a forward layer: 58 us; by 16-byte stores 81, by whole lines through
// shared memory 67.
__device__ __forceinline__ void store32(void *dst, const uint4 &a, const uint4 &b)
{
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(a.x), "r"(a.y), "r"(a.z),
                 "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
}
__device__ __forceinline__ void store_row(bf16 *dst, const uint4 (&row)[8])
{
#pragma unroll
    for (int c = 0; c < 8; c += 2)
        store32(dst + 8 * c, row[c], row[c + 1]);
}
// Which of a position's 32 activations are positive, for the backward pass: bit k for channel 2 k, bit 16 + k for
// channel 2 k + 1.  The backward convolution reads these 4 bytes per position instead of 64 of activations (a fifth
// of its traffic): 131 -> 110 us at L = 64, batch 512; the forward layers of a training step write them in
// 1 to 2 us each.
__device__ __forceinline__ uint32_t positive_bits(const uint32_t *w) // 16 packed pairs
{
    uint32_t bits = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
        bits |= __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(w + k), __floats2bfloat162_rn(0.f, 0.f)) & (0x00010001u << k);
    return bits;
}
// Zero the halves of channels 8 C .. 8 C + 7 of hi and lo whose bit is not set.
template <int C>
__device__ __forceinline__ void mask8(uint32_t bits, uint4 &hi, uint4 &lo)
{
    uint32_t on[4]; // bits k and 16 + k to the signs of the halves, the signs over the halves
#pragma unroll
    for (int k = 0; k < 4; ++k)
        asm("prmt.b32 %0, %1, 0, 0xBB99;" : "=r"(on[k]) : "r"(bits << (15 - (4 * C + k))));
    hi.x &= on[0], hi.y &= on[1], hi.z &= on[2], hi.w &= on[3];
    lo.x &= on[0], lo.y &= on[1], lo.z &= on[2], lo.w &= on[3];
}

// Layer 1 (1 -> 32 channels, mask A, ReLU) on the fifth-generation tensor
// cores: one MMA per tile of 128 consecutive positions (M = 128, N = 32,
// K = 16: the 12 taps and 4 zeros).  The A rows hold the (negated) spins --
// 0 outside the lattice, exact in BF16 -- in two K-major chunk planes; B holds the
// layer's weights (BF16 values, as k_prep_weights leaves them) as
// [chunk][out channel] rows.  A warp converts the spins of its 32 positions' three
// rows once into shared memory (the positions are consecutive, so each row is a
// run of 36 bytes, fetched a tile ahead), and a lane takes its five neighbours of a
// row as three words, shifted by half a word at odd positions and masked at the
// lattice's edges.  After the MMA each thread reads its position's 32 accumulator
// columns, adds the bias, applies ReLU and stores its BF16 row (store32).  Several CTAs per SM overlap
// one another's MMA waits; every wait on an mbarrier is bounded and a timeout latches *err (the tensor-memory
// allocation has no limit: see chain_wait for why it ends).  L = 64, 4096
// configurations: ~230 us against 436 when every tap was a byte load, a comparison and
// two conversions and every lane stored its own row 16 bytes an instruction (250 with the rows
// through shared memory into whole lines); the 1.07 GB it writes take 155.
constexpr int kL1Threads = 128;
constexpr uint32_t kL1Cols = 32;

__global__ void __launch_bounds__(kL1Threads, 8) k_layer1_tc(const int8_t *__restrict__ spins, int negate,
                                                             const float *__restrict__ w1, const float *__restrict__ b1,
                                                             bf16 *__restrict__ h1, uint32_t *__restrict__ bits, int n,
                                                             int L, int *err)
{
    __shared__ __align__(128) uint4 A[2][kL1Threads]; // chunk planes: taps 0-7, taps 8-15
    __shared__ __align__(128) uint4 B[2][kCh];        // chunk planes: [out channel] taps 0-7, 8-15
    __shared__ __align__(16) bf16 Win[kL1Threads / 32][3 * 40]; // a warp's spins, three rows of 36
    __shared__ __align__(16) float Bias[kCh];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tslot;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    chain_wait(false); // the next kernel's blocks come in only after this block's tensor memory is allocated (below)
    if (tid < kCh)
        Bias[tid] = b1[tid];
    if (tid < 2 * kCh) { // w1 is [o][t]
        const int pl = tid / kCh, o = tid % kCh;
        bf16 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int t = 8 * pl + k;
            v[k] = __float2bfloat16(t < kTapsA ? w1[o * kTapsA + t] : 0.f);
        }
        B[pl][o] = *reinterpret_cast<uint4 *>(v);
    }
    const uint32_t bar_s = smem_u32(&bar);
    if (warp == 0)
        tc::tmem_alloc(smem_u32(&tslot), kL1Cols);
    if (tid == 0)
        tc::mbar_init(bar_s, 1);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    chain_release();
    const uint32_t tbase = *reinterpret_cast<volatile uint32_t *>(&tslot);
    const uint64_t adesc = tc::smem_desc(smem_u32(&A[0][0]), kL1Threads * 16, 128);
    const uint64_t bdesc = tc::smem_desc(smem_u32(&B[0][0]), kCh * 16, 128);
    constexpr uint32_t idesc = tc::idesc_bf16_f32(128, kCh);
    const uint32_t total = (uint32_t)n * L * L, tiles = (total + kL1Threads - 1) / kL1Threads;
    const uint32_t step = gridDim.x * kL1Threads, step_y = step / L % L, step_x = step % L;
    bf16 *const win = Win[warp];
    uint32_t p = blockIdx.x * kL1Threads + tid; // this thread's position, its row and column
    int y = (int)(p / L % L), x = (int)(p % L);
    // the spins around the warp's positions, rows y - 2, y - 1, y: 36 each, from two left of the first
    int raw[3][2];
    auto fetch = [&](uint32_t first) {
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t i = first + lane + 32 * h - 2 - (2 - r) * L; // wraps below 0: out of range
                raw[r][h] = (h == 0 || lane < 4) && i < total ? spins[i] : 0;
            }
    };
    fetch(p - lane);
    int ok = 1;
    uint32_t uses = 0;
    for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x, ++uses) {
        const bool live = p < total;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (h == 0 || lane < 4)
                    win[r * 40 + lane + 32 * h] = __float2bfloat16((float)(negate ? -raw[r][h] : raw[r][h]));
        __syncwarp();
        p += step;
        fetch(p - lane);
        // neighbours e = 0..4 (dx = e - 2) of a row as pairs, zero outside the lattice
        const uint32_t m01 = (x >= 2 ? 0xFFFFu : 0u) | (x >= 1 ? 0xFFFF0000u : 0u),
                       m3 = x + 1 < L ? 0xFFFF0000u : 0u, m4 = x + 2 < L ? 0xFFFFu : 0u;
        uint32_t e01[3], e23[2], e4[2];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(win + r * 40) + (lane >> 1);
            const uint32_t w0 = w[0], w1 = w[1], in = y - 2 + r >= 0 ? 0xFFFFFFFFu : 0u;
            e01[r] = (lane & 1 ? __byte_perm(w0, w1, 0x5432) : w0) & m01 & in;
            if (r < 2) {
                const uint32_t w2 = w[2];
                e23[r] = (lane & 1 ? __byte_perm(w1, w2, 0x5432) : w1) & (0xFFFFu | m3) & in;
                e4[r] = (lane & 1 ? w2 >> 16 : w2) & m4 & in;
            }
        }
        // taps 0..4 of row y - 2, 5..9 of row y - 1, 10 and 11 of row y
        A[0][tid] = make_uint4(e01[0], e23[0], e4[0] | e01[1] << 16, __byte_perm(e01[1], e23[1], 0x5432));
        A[1][tid] = make_uint4(e23[1] >> 16 | e4[1] << 16, e01[2], 0u, 0u);
        x += step_x;
        y += step_y;
        if (x >= L) {
            x -= L;
            ++y;
        }
        if (y >= L)
            y -= L;
        tc::fence_smem_for_async();
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {
            tc::mma_bf16(tbase, adesc, bdesc, idesc, 0u);
            tc::commit(bar_s);
        }
        if (!__syncthreads_and(tc::mbar_wait(bar_s, uses & 1u, kTcMaxPolls))) { // block-uniform
            ok = 0;
            break;
        }
        tc::fence_after_sync();
        float v[kCh];
        tc::ld_32x32b_x32(tbase + ((uint32_t)(32 * warp) << 16), v);
        uint32_t u[kCh / 2];
#pragma unroll
        for (int c = 0; c < kCh; c += 2) {
            const float2 s = add2(make_float2(v[c], v[c + 1]), *reinterpret_cast<const float2 *>(&Bias[c]));
            u[c / 2] = relu_pack(s.x, s.y);
        }
        if (live) {
            bf16 *dst = h1 + (size_t)(p - step) * kCh;
            store32(dst, make_uint4(u[0], u[1], u[2], u[3]), make_uint4(u[4], u[5], u[6], u[7]));
            store32(dst + 16, make_uint4(u[8], u[9], u[10], u[11]), make_uint4(u[12], u[13], u[14], u[15]));
            if (bits)
                bits[p - step] = positive_bits(u);
        }
        tc::fence_before_sync(); // this tile's tensor-memory reads precede the next MMA
    }
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0)
        atomicExch(err, 1);
    tc::fence_after_sync();
    if (warp == 0)
        tc::tmem_free(tbase, kL1Cols);
}

// Gradients travel between the backward kernels as a BF16 hi + lo pair
// (hi = bf16(v), lo = bf16(v - hi), ~16 mantissa bits): two [n][L][L][32] BF16
// arrays in the space of one FP32 array, which the tensor cores read directly.
__device__ __forceinline__ void split8(const float *v, uint4 &hi, uint4 &lo)
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        h[k] = pack_bf16x2(v[2 * k], v[2 * k + 1]);
        l[k] = pack_bf16x2(v[2 * k] - bf16_lo(h[k]), v[2 * k + 1] - bf16_hi(h[k]));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// ---------------------------------------------------------------- masked 32-channel convolutions
// The hidden layers' forward and data-gradient convolutions and the last layer's
// forward, on the fifth-generation tensor cores (tcgen05.mma, BF16 in, FP32
// accumulator in tensor memory), as implicit GEMMs over runs of G = 4 (L % 4 == 0)
// or 2 neighbouring positions: row q of the operand A is the run x .. x + G - 1, 64 G
// bytes, and the accumulator of 128 rows holds the outputs of all its positions, G x
// 32 columns.  An MMA of one input position and 16 channels (K = 16) feeds all
// outputs of the run whose window it is in (N = 32 .. 32 G).  What bounds these kernels
// is the shared-memory read of the operands, 128 bytes per clock and SM: an MMA
// reads 4 KB of A and N x 32 bytes of B, so that 128 positions cost 1040 cycles with
// one-position rows (26 MMAs), 740 with G = 2 and 560 with G = 4.  Measured at L = 64,
// batch 4096, per hidden layer: forward 643 us with one-position rows, 463 with G = 2,
// 430 with G = 4 (its MMAs alone 370; 2.15 GB of activations, 5.0 TB/s), the data
// gradient 2600 with one-position rows staged by the CTA's threads, 1070 now (5.4 GB,
// 5.0 TB/s).
//
// Runs are indexed on a padded grid, q = (smp (R + 2) + r) P + pp with P = L / G + 1:
// pp = 0 is the zero run left of the row, and the run right of it is the next row's
// pp = 0.  A tap is a shifted view of the staged rows, which lie in G / 2 slabs of
// 128-byte rows (two positions each; 128-byte swizzle, which follows the absolute
// shared-memory address): the descriptor's start moves by whole rows, by 64 bytes for
// the second position of a slab.  Rows of A on the padding are computed and
// dropped.  B holds each tap's weights once, the taps of a kernel row in the order in
// which the next position of a run meets them one step later, so that the operand of
// N = 32 c columns is c consecutive taps.
//
//   FWD  : out(p)[o] = ReLU(b[o] + sum_t sum_c W[t][o][c] in(p + d_t)[c]), BF16.
//   LAST : the 32 -> 1 layer, 16 columns per position (the smallest N) of which
//          the first holds the logit f; the epilogue forms log sigmoid(s f) and
//          (training) dF = -(1/n) s sigmoid(-s f).
//   BWD  : out(p)[c] = [mask(p)[c] > 0] sum_t sum_o W[t][o][c] dz(p - d_t)[o], dz and
//          out as BF16 hi + lo pairs (two MMAs per K step).
//
// Warp-specialised: a producer warp streams an item's rows (R + 2 rows of P runs of
// S samples, a box per slab, everything outside the lattice zero-filled) by TMA into
// the second of two stage buffers, one thread of another warp issues the MMAs of the
// current item, the first EW warps drain tensor memory, 64 columns each (two slots
// per accumulator buffer: two tiles for G = 2, the halves of a tile for G = 4).  They hand over through mbarriers: stage
// full (TMA bytes), stage free (MMA commit), accumulator full (MMA commit) and
// accumulator free (epilogue arrivals); every wait is bounded and a timeout
// latches MC_ETIMEOUT.  Two CTAs per SM (4 epilogue warps each) where that costs at
// most 15% more tiles than one, to fill each other's pipeline gaps; else one, with 8
// epilogue warps for the data gradient.
constexpr int kFwd = 0, kLast = 1, kBwd = 2;
constexpr int kRunGuard = 8;                   // rows ahead of staged row 0 (8 x 128 bytes: a box lands 1024-byte aligned)
constexpr uint32_t kRunMaxSmem1 = 200u * 1024; // two stages + weights + barriers + scratch, one CTA per SM
constexpr uint32_t kRunMaxSmem2 = 113u * 1024; // the same, two CTAs per SM
constexpr uint32_t kRunBarBytes = 128;         // 9 mbarriers, tensor-memory slot
constexpr int kMaxItemRows = 32, kMaxItemSamples = 16, kMaxPackedTiles = 4;

__host__ __device__ constexpr int conv_cols(int mode) { return mode == kLast ? 16 : kCh; } // per position
__host__ __device__ constexpr uint32_t conv_weight_bytes(int mode) { return kTapsB * 4u * (uint32_t)conv_cols(mode) * 16u; }
__host__ __device__ constexpr int epilogue_warps(int mode, int ctas) { return mode == kBwd && ctas == 1 ? 8 : 4; }

struct RunGeom {
    int L, G, P, R, S, YB, tiles, ctas_per_sm; // S samples per item (1 unless an item holds whole lattices)
    uint32_t inv_p, inv_rows;                  // ceil(2^32 / P), ceil(2^32 / (R + 2)): exact quotients below 2^16
    uint32_t plane_bytes, stage_bytes, smem_bytes;
};

RunGeom run_geom_of(int L, int G, int R, int S, int mode, int ctas)
{
    RunGeom g{};
    g.L = L;
    g.G = G;
    g.P = L / g.G + 1;
    g.R = R;
    g.S = S;
    g.YB = (L + R - 1) / R;
    g.ctas_per_sm = ctas;
    const int q = (S * (R + 2) - 2) * g.P, qpad = (q + 127) / 128 * 128;
    g.tiles = qpad / 128;
    // the staged rows and the zero row past them; the views of the last tile's padding rows run on into what
    // follows (the other planes, the weights), whose products are dropped
    g.plane_bytes = (uint32_t)((kRunGuard + S * (R + 2) * g.P + 1 + 7) / 8 * 8) * 128u;
    g.stage_bytes = (mode == kBwd ? 2u : 1u) * (uint32_t)(g.G / 2) * g.plane_bytes;
    const uint32_t used = 2 * g.stage_bytes + conv_weight_bytes(mode) + kRunBarBytes;
    const uint32_t read = 2 * g.stage_bytes - g.plane_bytes + (uint32_t)(kRunGuard + qpad + 2 * g.P + 2) * 128u;
    g.smem_bytes = std::max(used, read) + 1024; // + alignment slack
    g.inv_p = (uint32_t)(((1ull << 32) + g.P - 1) / g.P);
    g.inv_rows = (uint32_t)(((1ull << 32) + R + 1) / (R + 2));
    return g;
}

// Shared-memory cycles of a tile's MMAs: 4 KB of A and 32 bytes per column of B each,
// at 128 bytes per clock (two channel halves; BWD hi and lo alike for every G).
int tile_cycles(int mode, int G)
{
    int cycles = 0;
    for (int d = 0; d < 3; ++d)
        for (int j = -2; j <= G + 1; ++j) {
            const int ulo = d == 2 && mode != kBwd ? 2 : 0, uhi = d == 2 && mode == kBwd ? 2 : 4;
            const int n = std::min(uhi - 1 + j, G) - std::max(ulo - 2 + j, 0);
            cycles += n > 0 ? 2 * (32 + n * conv_cols(mode) / 4) : 0;
        }
    return cycles;
}

// Run length, rows and (for lattices that fit an item whole) samples per item: the
// fewest cycles per sample among those whose two stages fit `max_smem`.
RunGeom run_geom_cap(int L, int mode, int ctas, uint32_t max_smem, double &cost)
{
    RunGeom best{};
    cost = 1e300;
    for (int G = 2; G <= 4 && L % G == 0; G += 2) {
        const int cycles = tile_cycles(mode, G);
        for (int R = 1; R <= kMaxItemRows && R <= L; ++R)
            for (int S = 1; S == 1 || (R == L && S <= kMaxItemSamples); ++S) {
                const RunGeom g = run_geom_of(L, G, R, S, mode, ctas);
                if (g.smem_bytes > max_smem || (S > 1 && g.tiles > kMaxPackedTiles))
                    continue;
                const double c = (double)g.YB * g.tiles / S * cycles;
                if (c < cost || (c == cost && S == 1 && R > best.R)) {
                    best = g;
                    cost = c;
                }
            }
    }
    return best;
}

RunGeom run_geom(int L, int mode)
{
    double c1, c2;
    const RunGeom one = run_geom_cap(L, mode, 1, kRunMaxSmem1, c1), two = run_geom_cap(L, mode, 2, kRunMaxSmem2, c2);
    return two.R > 0 && c2 <= 1.15 * c1 ? two : one;
}

struct LastLayerArgs {
    const float *wD; // [t][c], BF16-representable
    const float *bD; // the layer's bias (one value)
    const int8_t *spins;
    int negate;
    float *f, *ll, *dF; // dF may be null
    float inv_n;
};

struct ConvArgs {
    const bf16 *W;     // [t][o][c] (FWD, BWD)
    const float *bias; // FWD
    const uint32_t *mask; // BWD: positive_bits of the layer's input activations
    uint32_t *bits;    // FWD: positive_bits of the output, or null
    bf16 *out, *out_lo;
    LastLayerArgs la;
    int n;
    int *err;
};

template <int MODE, int G, int MINB>
__global__ void __launch_bounds__(32 * (epilogue_warps(MODE, MINB) + 2), MINB)
    k_conv_runs(const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
                const __grid_constant__ ConvArgs a, const __grid_constant__ RunGeom g)
{
    constexpr int EW = epilogue_warps(MODE, MINB);
    constexpr int NB = conv_cols(MODE);             // accumulator columns per position
    constexpr uint32_t kSlot = 2 * NB;              // columns of a slot: two positions
    constexpr uint32_t kCols = 4 * kSlot;           // two buffers of two slots
    constexpr int kGroup = G == 2 ? 2 : 1;          // tiles per commit
    constexpr int SLABS = G / 2;
    constexpr uint32_t kTap = NB * 16;              // bytes of one tap in one chunk plane
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the stages hold 128-byte-swizzled rows: round the base up to 1024 bytes
    // (the launch reserves 1024 extra bytes)
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sb = smem_u32(smem);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t boff = 2 * g.stage_bytes, bars = boff + conv_weight_bytes(MODE);
    const uint32_t full0 = sb + bars, empty0 = full0 + 16, tfull0 = full0 + 32, tempty0 = full0 + 48,
                   drain = full0 + 64, tslot_off = bars + 80;
    // the run right of the box's last row is zero (BWD reads it); whatever else lies outside the boxes is met only by
    // rows of A that are dropped
    for (uint32_t i = tid; i < 8u * 2u * g.stage_bytes / g.plane_bytes; i += blockDim.x)
        *reinterpret_cast<uint4 *>(smem + (i >> 3) * g.plane_bytes +
                                   (uint32_t)(kRunGuard + g.S * (g.R + 2) * g.P) * 128u + (i & 7u) * 16u) =
            make_uint4(0u, 0u, 0u, 0u);
    // Weights: [kernel row d][chunk of 8 K values][tap u'][row] x 16 bytes.  Tap order: FWD and LAST dx = 2 .. -2
    // (row dy = 0: 0, -1, -2), BWD dx = -2 .. 2 (-2, -1, 0).
    for (int i = tid; i < kTapsB * 4 * NB; i += blockDim.x) {
        const int d = i < 20 * NB ? 0 : i < 40 * NB ? 1 : 2, nt = d == 2 ? 3 : 5;
        const int r0 = i - d * 20 * NB, c8 = r0 / (nt * NB), u = (r0 / NB) % nt, o = r0 % NB;
        const int dx = MODE == kBwd ? u - 2 : (d == 2 ? -u : 2 - u), t = d == 2 ? 12 + dx : 5 * d + dx + 2;
        bf16 v[8];
        if (MODE == kFwd) {
            *reinterpret_cast<uint4 *>(v) =
                *reinterpret_cast<const uint4 *>(a.W + ((size_t)(t * kCh + o) * kCh + c8 * 8));
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                v[k] = MODE == kBwd ? a.W[((size_t)t * kCh + c8 * 8 + k) * kCh + o]
                                    : __float2bfloat16(o == 0 ? a.la.wD[t * kCh + c8 * 8 + k] : 0.f);
        }
        *reinterpret_cast<uint4 *>(smem + boff + (uint32_t)i * 16u) = *reinterpret_cast<uint4 *>(v);
    }
    if (warp == 0)
        tc::tmem_alloc(sb + tslot_off, kCols);
    if (tid == 0) {
        for (int k = 0; k < 2; ++k) {
            tc::mbar_init(full0 + 8 * k, 1);
            tc::mbar_init(empty0 + 8 * k, 1);
            tc::mbar_init(tfull0 + 8 * k, 1);
            tc::mbar_init(tempty0 + 8 * k, EW);
        }
        tc::mbar_init(drain, 1);
    }
    tc::fence_smem_for_async();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    chain_wait(true); // only the weights, final before the first kernel of the pass, were read so far
    const uint32_t tbase = __shfl_sync(0xffffffffu, *reinterpret_cast<volatile uint32_t *>(smem + tslot_off), 0);
    const int total = (a.n + g.S - 1) / g.S * g.YB, rounds = (g.tiles + kGroup - 1) / kGroup;
    int ok = 1;
    if (warp == EW) {
        if (lane == 0) { // producer
            const uint32_t bytes = (uint32_t)(g.S * (g.R + 2) * g.P) * 128u * SLABS * (MODE == kBwd ? 2u : 1u);
            int k = 0, armed[2] = {-1, -1};
            for (int it = blockIdx.x; it < total; it += gridDim.x, ++k) {
                const int s = k & 1;
                if (k >= 2 && !tc::mbar_wait(empty0 + 8 * s, ((k >> 1) - 1) & 1, kTcMaxPolls)) {
                    ok = 0;
                    break;
                }
                const int bi = it / g.YB, y0 = (it - bi * g.YB) * g.R, ys = MODE == kBwd ? y0 : y0 - 2;
                tc::mbar_arrive_expect_tx(full0 + 8 * s, bytes);
                const uint32_t st = sb + (uint32_t)s * g.stage_bytes + kRunGuard * 128u;
                // rows ys .. ys + R + 1 of P runs from x = -G, S samples: one box per slab of two positions
#pragma unroll
                for (int sl = 0; sl < SLABS; ++sl) {
                    tc::tma_load_5d(st + (uint32_t)sl * g.plane_bytes, &map_hi, 0, sl, -1, ys, bi * g.S, full0 + 8 * s);
                    if (MODE == kBwd)
                        tc::tma_load_5d(st + (uint32_t)(SLABS + sl) * g.plane_bytes, &map_lo, 0, sl, -1, ys, bi * g.S,
                                        full0 + 8 * s);
                }
                armed[s] = k;
            }
            for (int s = 0; s < 2; ++s) // the last loads of each stage have landed before the CTA ends
                if (armed[s] >= 0 && !tc::mbar_wait(full0 + 8 * s, (armed[s] >> 1) & 1, kTcMaxPolls))
                    ok = 0;
        }
    } else if (warp == EW + 1) { // MMA issuer: the whole warp, uniform; an elected lane issues
        {
            const uint64_t a0 = tc::smem_desc_sw128(sb + kRunGuard * 128u);
            uint64_t bd[3]; // kernel row d: its chunk planes are nt kTap bytes apart
#pragma unroll
            for (int d = 0; d < 3; ++d)
                bd[d] = tc::smem_desc(sb + boff + (uint32_t)d * 20u * kTap, (d == 2 ? 3u : 5u) * kTap, 128);
            const uint64_t slab = (uint64_t)(g.plane_bytes >> 4), lo_off = SLABS * slab;
            uint32_t tcount = 0;
            int k = 0;
            for (int it = blockIdx.x; ok && it < total; it += gridDim.x, ++k) {
                const int s = k & 1;
                if (!__all_sync(0xffffffffu, tc::mbar_wait(full0 + 8 * s, (k >> 1) & 1, kTcMaxPolls))) {
                    ok = 0;
                    break;
                }
                tc::fence_after_sync();
                for (int rd = 0; rd < rounds; ++rd, ++tcount) {
                    const uint32_t bb = tcount & 1u;
                    if (tcount >= 2 &&
                        !__all_sync(0xffffffffu,
                                    tc::mbar_wait(tempty0 + 8 * bb, ((tcount >> 1) - 1) & 1u, kTcMaxPolls))) {
                        ok = 0;
                        break;
                    }
                    tc::fence_after_sync();
                    const int m0 = rd * kGroup, m1 = m0 + kGroup < g.tiles ? m0 + kGroup : g.tiles;
                    for (int m = m0; m < m1; ++m) {
                        const uint32_t dt = tbase + (2 * bb + (uint32_t)(m - m0)) * kSlot;
                        const uint64_t at = a0 + (uint64_t)(((uint32_t)s * g.stage_bytes) >> 4) +
                                            (uint64_t)((uint32_t)m * 128u * 8u); // 128 rows x 128 B
                        // kernel row d, input position x + j of the run x .. x + G - 1, channel half h: tap u = 2 - j + k
                        // of the run's position k, for the positions k0 <= k < k1 whose window holds it
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            const int ulo = d == 2 && MODE != kBwd ? 2 : 0, uhi = d == 2 && MODE == kBwd ? 2 : 4;
                            const uint64_t ar = at + (uint64_t)((uint32_t)(MODE == kBwd ? 2 - d : d) * (uint32_t)g.P * 8u);
                            const uint64_t bplane = (uint64_t)(((d == 2 ? 3u : 5u) * kTap) >> 4);
#pragma unroll
                            for (int j = -2; j <= G + 1; ++j) {
                                const int k0 = ulo - 2 + j > 0 ? ulo - 2 + j : 0, k1 = uhi - 1 + j < G ? uhi - 1 + j : G;
                                if (k0 >= k1)
                                    continue;
                                const int run = (j + G) / G - 1, pos = (j + G) % G; // the run it lies in, its position there
#pragma unroll
                                for (int h = 0; h < 2; ++h) { // 16 channels at 16 h
                                    const uint64_t A = ar + (uint64_t)(pos >> 1) * slab +
                                                       (uint64_t)(int64_t)(run * 8 + (pos & 1) * 4 + h * 2);
                                    const uint64_t B = bd[d] + (uint64_t)(2 * h) * bplane +
                                                       (uint64_t)((uint32_t)(2 - j + k0 - ulo) * (kTap >> 4));
                                    // position j + 2 meets its first tap here: its columns do not accumulate yet
                                    const bool first = d == 0 && h == 0 && j + 2 < G;
                                    const int ka = first ? k1 - 1 : k1; // accumulating positions k0 .. ka - 1
                                    if (ka > k0) {
                                        tc::mma_bf16_warp<true>(dt + k0 * NB, A, B, tc::idesc_bf16_f32(128, (ka - k0) * NB));
                                        if (MODE == kBwd)
                                            tc::mma_bf16_warp<true>(dt + k0 * NB, A + lo_off, B,
                                                                    tc::idesc_bf16_f32(128, (ka - k0) * NB));
                                    }
                                    if (first) {
                                        const uint64_t B1 = B + (uint64_t)((uint32_t)(ka - k0) * (kTap >> 4));
                                        tc::mma_bf16_warp<false>(dt + ka * NB, A, B1, tc::idesc_bf16_f32(128, NB));
                                        if (MODE == kBwd)
                                            tc::mma_bf16_warp<true>(dt + ka * NB, A + lo_off, B1, tc::idesc_bf16_f32(128, NB));
                                    }
                                }
                            }
                        }
                    }
                    tc::commit_warp(tfull0 + 8 * bb);
                }
                if (!ok)
                    break;
                tc::commit_warp(empty0 + 8 * s); // stage s is free once this item's MMAs have read it
            }
            tc::commit_warp(drain); // every MMA issued above has completed before the CTA ends
            if (!__all_sync(0xffffffffu, tc::mbar_wait(drain, 0u, kTcMaxPolls)))
                ok = 0;
        }
    } else { // epilogue, tensor-memory lanes 32 (warp % 4) .. + 31; 8 warps: slot warp / 4, 4 warps: both slots
        float bv[kCh];
#pragma unroll
        for (int c = 0; c < kCh; ++c)
            bv[c] = MODE == kFwd ? __ldg(&a.bias[c]) : 0.f;
        const float b0 = MODE == kLast ? __ldg(a.la.bD) : 0.f;
        uint32_t tcount = 0;
        for (int it = blockIdx.x; ok && it < total; it += gridDim.x) {
            const int bi = it / g.YB, y0 = (it - bi * g.YB) * g.R;
            for (int rd = 0; rd < rounds; ++rd, ++tcount) {
                const uint32_t bb = tcount & 1u;
                const int m0 = rd * kGroup;
                const int slot0 = EW == 8 ? warp >> 2 : 0;
                const int slot1 = EW == 8 ? slot0 + 1 : (G == 4 || m0 + 1 < g.tiles ? 2 : 1);
                bool waited = false;
#pragma unroll 1
                for (int slot = slot0; slot < slot1; ++slot) {
                    const uint32_t col = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (2 * bb + (uint32_t)slot) * kSlot;
                    const int m = G == 2 ? m0 + slot : m0;
                    const uint32_t q = (uint32_t)(m * 128 + 32 * (warp & 3) + lane), row = __umulhi(q, g.inv_p),
                                   pp = q - row * (uint32_t)g.P;
                    const uint32_t smp = g.S == 1 ? 0u : __umulhi(row, g.inv_rows), r = row - smp * (uint32_t)(g.R + 2);
                    const int b = bi * g.S + (int)smp, y = y0 + (int)r;
                    const bool live = pp >= 1 && (int)r < g.R && y < g.L && (int)smp < g.S && b < a.n && m < g.tiles;
                    // first position of the slot's pair: this lane's row of 2 x 32 channels
                    const size_t p = ((size_t)b * g.L + y) * g.L + G * (pp - 1) + (G == 4 ? 2 * slot : 0);
                    uint2 mk = make_uint2(0u, 0u);
                    if (MODE == kBwd && live) // the masks, in flight during the wait
                        mk = __ldg(reinterpret_cast<const uint2 *>(a.mask + p));
                    if (!waited) {
                        waited = true;
                        ok = __any_sync(0xffffffffu, tc::mbar_wait(tfull0 + 8 * bb, (tcount >> 1) & 1u, kTcMaxPolls));
                        tc::fence_after_sync();
                        if (!ok)
                            break;
                    }
                    auto taken = [&] { // the accumulator is in registers: the next MMAs may have it
                        if (slot + 1 == slot1) {
                            tc::fence_before_sync();
                            __syncwarp();
                            if (lane == 0)
                                tc::mbar_arrive(tempty0 + 8 * bb);
                        }
                    };
                    if (MODE == kLast) {
                        const float acc[2] = {tc::ld_32x32b_x1(col), tc::ld_32x32b_x1(col + NB)};
                        taken();
                        if (live) {
                            const char2 s2 = *reinterpret_cast<const char2 *>(a.la.spins + p);
                            const float sv[2] = {a.la.negate ? -(float)s2.x : (float)s2.x,
                                                 a.la.negate ? -(float)s2.y : (float)s2.y};
                            const float f0 = b0 + acc[0], f1 = b0 + acc[1];
                            *reinterpret_cast<float2 *>(a.la.f + p) = make_float2(f0, f1);
                            *reinterpret_cast<float2 *>(a.la.ll + p) =
                                make_float2(log_sigmoid(sv[0] * f0), log_sigmoid(sv[1] * f1));
                            if (a.la.dF)
                                *reinterpret_cast<float2 *>(a.la.dF + p) =
                                    make_float2(-a.la.inv_n * sv[0] * sigmoid(-sv[0] * f0),
                                                -a.la.inv_n * sv[1] * sigmoid(-sv[1] * f1));
                        }
                    } else if (MODE == kFwd) {
                        float v[2 * kCh];
                        tc::ld_32x32b_x64(col, v);
                        taken();
                        uint4 pk[8];
                        uint32_t *pw = reinterpret_cast<uint32_t *>(pk);
#pragma unroll
                        for (int c = 0; c < 2 * kCh; c += 2) {
                            const float2 s = add2(make_float2(v[c], v[c + 1]), make_float2(bv[c % kCh], bv[c % kCh + 1]));
                            pw[c / 2] = relu_pack(s.x, s.y);
                        }
                        if (live) {
                            store_row(a.out + p * kCh, pk);
                            if (a.bits)
                                *reinterpret_cast<uint2 *>(a.bits + p) = make_uint2(positive_bits(pw), positive_bits(pw + 16));
                        }
                    } else { // one position after the other, for the registers
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            float v[kCh];
                            tc::ld_32x32b_x32(col + h * NB, v);
                            if (h == 1)
                                taken();
                            uint4 hi[4], lo[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                split8(v + 8 * k, hi[k], lo[k]);
                            const uint32_t on = h ? mk.y : mk.x;
                            mask8<0>(on, hi[0], lo[0]);
                            mask8<1>(on, hi[1], lo[1]);
                            mask8<2>(on, hi[2], lo[2]);
                            mask8<3>(on, hi[3], lo[3]);
                            if (live) {
                                bf16 *d = a.out + (p + h) * kCh, *e = a.out_lo + (p + h) * kCh;
                                store32(d, hi[0], hi[1]);
                                store32(d + 16, hi[2], hi[3]);
                                store32(e, lo[0], lo[1]);
                                store32(e + 16, lo[2], lo[3]);
                            }
                        }
                    }
                }
                if (!ok)
                    break;
            }
        }
    }
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0)
        atomicExch(a.err, 1);
    tc::fence_after_sync();
    if (warp == 0)
        tc::tmem_free(tbase, kCols);
}

template <int MODE>
using ConvKernel = void (*)(const CUtensorMap, const CUtensorMap, const ConvArgs, const RunGeom);
template <int MODE>
ConvKernel<MODE> conv_kernel(const RunGeom &g)
{
    if (g.G == 4)
        return g.ctas_per_sm == 2 ? k_conv_runs<MODE, 4, 2> : k_conv_runs<MODE, 4, 1>;
    return g.ctas_per_sm == 2 ? k_conv_runs<MODE, 2, 2> : k_conv_runs<MODE, 2, 1>;
}

// Launch one convolution; map_lo only for BWD.
template <int MODE>
void launch_conv(const RunGeom &g, const CUtensorMap &hi, const CUtensorMap &lo, const ConvArgs &a, int sms,
                 cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<size_t>((size_t)((a.n + g.S - 1) / g.S) * g.YB, (size_t)sms * g.ctas_per_sm);
    launch_chained_on(st, true, conv_kernel<MODE>(g), grid, 32u * (epilogue_warps(MODE, g.ctas_per_sm) + 2), g.smem_bytes,
                      hi, lo, a, g);
}

// Encoder of tensor maps, from the driver through the runtime (no link
// dependency on the driver library).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// Activations [n][L][L][32] BF16 as a 5-D tensor (32 channels, 1, x, y,
// sample); one box is R + 2 rows of P positions from x = -2, all channels: it
// lands in shared memory as 64-byte rows in the 64-byte swizzle, the columns
// outside the lattice zero-filled.
cudaError_t activation_map(CUtensorMap *m, const bf16 *base, int n, int L, int P, int rows)
{
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc)
        return cudaErrorNotSupported;
    const cuuint64_t dims[5] = {32, 1, (cuuint64_t)L, (cuuint64_t)L, (cuuint64_t)n};
    const cuuint64_t strides[4] = {64, 64, (cuuint64_t)64 * L, (cuuint64_t)64 * L * L};
    const cuuint32_t box[5] = {32, 1, (cuuint32_t)P, (cuuint32_t)rows, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// The same tensor as runs of G positions (64 values = two positions, slab, x / G, y,
// sample); one box is R + 2 rows of P runs of S samples of one slab, landing as
// 128-byte rows in the 128-byte swizzle.
cudaError_t run_map(CUtensorMap *m, const bf16 *base, int n, const RunGeom &g)
{
    const PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc)
        return cudaErrorNotSupported;
    const cuuint64_t L = (cuuint64_t)g.L, G = (cuuint64_t)g.G;
    const cuuint64_t dims[5] = {64, G / 2, L / G, L, (cuuint64_t)n};
    const cuuint64_t strides[4] = {128, 64 * G, 64 * L, 64 * L * L};
    const cuuint32_t box[5] = {64, 1, (cuuint32_t)g.P, (cuuint32_t)(g.R + 2), (cuuint32_t)g.S};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<bf16 *>(base), dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// log q per sample: fixed-order FP64 sum of its L^2 log-probabilities.
__global__ void k_logq(const float *ll, double *logq, int L)
{
    __shared__ double part[32];
    const int b = blockIdx.x, n = L * L;
    double acc = 0.0;
    chain_wait(true);
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        acc += (double)ll[(size_t)b * n + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0)
        part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
            s += part[w];
        logq[b] = s;
    }
}

// ------------------------------------------------------------------ backward
// Asynchronous copies into shared memory (non-bulk: any warp lane, 4 or 16 bytes,
// the rest of the destination zeroed when fewer source bytes are given).
__device__ __forceinline__ void cp16(void *dst, const void *src, int bytes = 16)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp4(void *dst, const void *src, int bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT>
__device__ __forceinline__ void cp_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// A warp's work in the edge kernels: pieces of at most 32 positions of the rows item,
// item + step, ..., in order.
struct Piece {
    int item, x; // row b * L + y, first position
    __device__ void next(int L, int step)
    {
        x += 32;
        if (x >= L) {
            x = 0;
            item += step;
        }
    }
};

// Backward of the last layer, data and weights at once, since both need dF at the
// 13 positions p - d_t of every p:
//   dZ_{D-1}(p)[c] = [h(p)[c] > 0] sum_t wD[t][c] dF(p - d_t),
//   gW[t][c] = sum_p h(p)[c] dF(p - d_t),  gb = sum_p dF(p), h = h_{D-1}.
// A warp takes a row, four positions at a time with 8 lanes of 4 channels each; a lane
// keeps its 52 weights and 52 gradient sums in registers, so that a position costs 13
// shared-memory reads (dF) and 104 multiply-adds per lane, and h is read once.  The
// lanes of a channel, then the warps are added in a fixed order into the CTA's partial
// sums part[output][CTA] (reduced in a fixed order by k_edge_grad_reduce: the gradient
// does not depend on the order the CTAs finish in).  L = 64, batch 512: 105 us for the
// 146 + 190 us of separate kernels that read weights and activations per tap from shared
// memory (193 with h prefetched one position ahead in registers: latency-bound); bound
// by the multiply-adds (47 us) and 400 MB of activations and gradients (60 us).
constexpr int kEdgeOutD = kTapsB * kCh + 1;  // last layer: 13 x 32 weights + bias
constexpr int kEdgeOut1 = kCh * (kTapsA + 1); // first layer: 32 x (12 weights + bias)
constexpr int kEdgeThreads = 128, kEdgeCtas = 3;
constexpr int kStagesD = 4, kStages1 = 3; // pieces a warp has staged or in flight
constexpr int kPieceBytes = 32 * kCh * 2; // 32 positions of one BF16 tensor
// Shared memory of a warp: the stages of h (or dZ1 hi and lo), and per stage the rows
// of dF (or the bytes of the spins and, once, their rows as floats).
__host__ __device__ inline int edge_row(int L) { return (3 * (L + 4) * 4 + 15) & ~15; }
__host__ __device__ inline int edge_bytes_d(int L) { return kStagesD * (kPieceBytes + edge_row(L)); }
constexpr int kSpinBytes = 3 * kMaxL + 16;
__host__ __device__ inline int edge_bytes_1(int L) { return kStages1 * (2 * kPieceBytes + kSpinBytes) + edge_row(L); }
__global__ void __launch_bounds__(kEdgeThreads, kEdgeCtas)
    k_layerD_bwd(const float *dF, const float *wD, const bf16 *hD, bf16 *dzh, bf16 *dzl, float *part, int n, int L)
{
    constexpr int NW = kEdgeThreads / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float R[NW][kEdgeOutD];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, c0 = (lane & 7) * 4;
    unsigned char *const H = smem + warp * edge_bytes_d(L);
    float *const G = reinterpret_cast<float *>(H + kStagesD * kPieceBytes);
    const int row = edge_row(L) / 4, rows = n * L, step = gridDim.x * NW;
    float W[kTapsB][4], acc[kTapsB][4], accb = 0.f;
#pragma unroll
    for (int t = 0; t < kTapsB; ++t) {
        const float4 w = *reinterpret_cast<const float4 *>(wD + t * kCh + c0);
        W[t][0] = w.x, W[t][1] = w.y, W[t][2] = w.z, W[t][3] = w.w;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            acc[t][q] = 0.f;
    }
    chain_wait(true);
    Piece next{(int)blockIdx.x * NW + warp, 0}, cur = next;
    int next_stage = 0, next_win = kStagesD - 1, stage = 0, win = kStagesD - 1;
    auto fetch = [&] { // stage the next piece, with the rows y .. y + 2 of dF at the start of a row
        if (next.item < rows) {
            const unsigned char *src = reinterpret_cast<const unsigned char *>(hD + ((size_t)next.item * L + next.x) * kCh);
            const int units = min(32, L - next.x) * 4;
            for (int i = lane; i < units; i += 32)
                cp16(H + next_stage * kPieceBytes + 16 * i, src + 16 * i);
            if (next.x == 0) {
                next_win = next_win + 1 == kStagesD ? 0 : next_win + 1;
                const int y = next.item % L;
                const float *f = dF + (size_t)next.item * L;
                for (int r = 0; r < 3; ++r)
                    for (int x = lane - 2; x < L + 2; x += 32) {
                        const bool in = y + r < L && x >= 0 && x < L;
                        cp4(G + next_win * row + r * (L + 4) + x + 2, in ? f + r * L + x : f, in ? 4 : 0);
                    }
            }
            next.next(L, step);
            next_stage = next_stage + 1 == kStagesD ? 0 : next_stage + 1;
        }
        cp_commit();
    };
    for (int k = 0; k < kStagesD - 1; ++k)
        fetch();
    while (cur.item < rows) {
        cp_wait<kStagesD - 2>();
        __syncwarp(); // the piece is there for every lane, and the stage before it is read
        fetch();
        if (cur.x == 0)
            win = win + 1 == kStagesD ? 0 : win + 1;
        const float *g = G + win * row + cur.x + 2;
        const unsigned char *hs = H + stage * kPieceBytes + c0 * 2;
        const size_t out = ((size_t)cur.item * L + cur.x) * kCh + c0;
        const int len = min(32, L - cur.x);
#pragma unroll 1
        for (int x = lane >> 3; x < len; x += 4) {
            const uint2 hx = *reinterpret_cast<const uint2 *>(hs + x * (kCh * 2));
            const float hv[4] = {__uint_as_float(hx.x << 16), __uint_as_float(hx.x & 0xFFFF0000u),
                                 __uint_as_float(hx.y << 16), __uint_as_float(hx.y & 0xFFFF0000u)};
            float o[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int t = 0; t < kTapsB; ++t) {
                const float gv = g[-tap_dy(t) * (L + 4) + x - tap_dx(t)];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    o[q] += W[t][q] * gv;
                    acc[t][q] += gv * hv[q];
                }
                if (t == kTapsB - 1)
                    accb += gv;
            }
            bf16 hi[4], lo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float v = hv[q] > 0.f ? o[q] : 0.f;
                hi[q] = __float2bfloat16(v);
                lo[q] = __float2bfloat16(v - bf(hi[q]));
            }
            *reinterpret_cast<uint2 *>(dzh + out + x * kCh) = *reinterpret_cast<uint2 *>(hi);
            *reinterpret_cast<uint2 *>(dzl + out + x * kCh) = *reinterpret_cast<uint2 *>(lo);
        }
        cur.next(L, step);
        stage = stage + 1 == kStagesD ? 0 : stage + 1;
    }
#pragma unroll
    for (int t = 0; t < kTapsB; ++t)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float v = acc[t][q];
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (lane < 8)
                R[warp][t * kCh + c0 + q] = v;
        }
    accb += __shfl_xor_sync(0xffffffffu, accb, 8);
    accb += __shfl_xor_sync(0xffffffffu, accb, 16);
    if (lane == 0)
        R[warp][kTapsB * kCh] = accb;
    __syncthreads();
    for (int o = tid; o < kEdgeOutD; o += blockDim.x) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w)
            v += R[w][o];
        part[(size_t)o * gridDim.x + blockIdx.x] = v;
    }
}

// Gradient of the first (FIRST) or last layer: one CTA per output adds its
// nb per-CTA partial sums (part[output][CTA]) in a fixed order -- strided
// per-thread sums, then a fixed shuffle and shared-memory tree -- and writes
// the canonical parameter.
template <bool FIRST>
__global__ void __launch_bounds__(256) k_edge_grad_reduce(const float *part, int nb, float *g, DevParams P)
{
    __shared__ float ws[8];
    const int o = blockIdx.x, tid = threadIdx.x;
    float v = 0.f;
    chain_wait(true);
    for (int b = tid; b < nb; b += blockDim.x)
        v += part[(size_t)o * nb + b];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, d);
    if ((tid & 31) == 0)
        ws[tid >> 5] = v;
    __syncthreads();
    if (tid != 0)
        return;
    v = ((ws[0] + ws[1]) + (ws[2] + ws[3])) + ((ws[4] + ws[5]) + (ws[6] + ws[7]));
    if (FIRST) {
        const int oc = o / (kTapsA + 1), t = o - oc * (kTapsA + 1);
        g[t < kTapsA ? canon_w(P, 0, oc, 0, tap_dy(t), tap_dx(t)) : P.b_off[0] + oc] = v;
    } else {
        const int t = o / kCh, c = o - t * kCh;
        g[t < kTapsB ? canon_w(P, P.D - 1, 0, c, tap_dy(t), tap_dx(t)) : P.b_off[P.D - 1]] = v;
    }
}

// Weight gradient of a 32 -> 32 layer on the fifth-generation tensor cores:
//   dW[t][o][c] = sum_(b, y, x) dz(b, y, x)[o] X(b, y + dy_t, x + dx_t)[c],
//   db[o] = sum_(b, y, x) dz(b, y, x)[o],
// dz as its BF16 hi + lo pair.  One item is one row (b, y): its dz hi and lo
// rows and the input rows y-2 .. y (columns -2 .. PX-3, zero outside the
// lattice) arrive by TMA in the 64-byte swizzle, and the positions of the row
// are the reduction dimension K.  Both operands are read MN-major.  A = the
// input rows, whose M dimension takes four taps at once: the taps (dy, dx ..
// dx+3) of one kernel row are the same staged row shifted by one position,
// i.e. 32-channel atoms 64 bytes apart (the descriptor's leading offset), and
// taps (-2, 2), (-1, 2) are one staged row apart (M = 64).  B = dz (N = 64: 32
// columns of hi, then 32 of lo, the lo plane one descriptor stride away).  The
// 13 taps are four MMAs per 16 positions (M = 128, 128, 128 with one unused
// tap, 64), accumulated in 256 tensor-memory columns over all items of the
// CTA; tensor-memory lane (tap, c) then holds the hi and the lo sums of
// channel c, added in the drain.  Roles: warp 4 loads (ring of NS stages),
// warp 5 issues, warps 0-3 sum the bias gradient from the staged dz rows and
// drain the accumulator.  Per-CTA partial sums [t][o][c] then the 32 biases,
// reduced in CTA order by k_dw_reduce.  Two CTAs per SM, so that one's MMAs
// fill the other's gaps.  Every wait is bounded; a timeout latches *err.
struct DwTcGeom {
    int L, PZ, PX, KS, NS;
    uint32_t zbytes, xbytes, stage_bytes, smem_bytes;
};
constexpr uint32_t kDwTcAlloc = 256;       // tensor-memory columns: 4 tap groups x (32 hi + 32 lo)
constexpr uint32_t kDwTcMaxSmem = 110u * 1024;
constexpr int kDwTcMaxStages = 6;

DwTcGeom dw_tc_geom(int L)
{
    DwTcGeom g{};
    g.L = L;
    g.PZ = (L + 15) / 16 * 16;
    g.PX = (g.PZ + 4 + 7) / 8 * 8;
    g.KS = g.PZ / 16;
    g.zbytes = (uint32_t)g.PZ * 64u;
    g.xbytes = ((uint32_t)(3 * g.PX) * 64u + 1023u) / 1024u * 1024u;
    g.stage_bytes = 2 * g.zbytes + g.xbytes;
    const uint32_t extra = 256 + 512 + 1024; // barriers and tensor-memory slot, bias sums, alignment slack
    g.NS = (int)std::min<uint32_t>(kDwTcMaxStages, (kDwTcMaxSmem - extra) / g.stage_bytes);
    g.smem_bytes = (uint32_t)g.NS * g.stage_bytes + extra;
    return g;
}

__global__ void __launch_bounds__(192, 2) k_dw32_tc(const __grid_constant__ CUtensorMap zh_map,
                                                    const __grid_constant__ CUtensorMap zl_map,
                                                    const __grid_constant__ CUtensorMap x_map, float *__restrict__ part,
                                                    int n, DwTcGeom g, int *err)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const uint32_t sb = smem_u32(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, NS = g.NS;
    const uint32_t ring = (uint32_t)NS * g.stage_bytes;
    const uint32_t full0 = sb + ring, empty0 = full0 + 8 * kDwTcMaxStages, done = empty0 + 8 * kDwTcMaxStages,
                   tslot_off = ring + 16 * kDwTcMaxStages + 8;
    float *bsum_s = reinterpret_cast<float *>(smem + ring + 256); // [4][32]
    if (warp == 0)
        tc::tmem_alloc(sb + tslot_off, kDwTcAlloc);
    if (tid == 0) {
        for (int s = 0; s < NS; ++s) {
            tc::mbar_init(full0 + 8 * s, 1);
            tc::mbar_init(empty0 + 8 * s, 5); // the MMA commit and the four bias warps
        }
        tc::mbar_init(done, 1);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    chain_wait(true);
    const uint32_t tbase = *reinterpret_cast<volatile uint32_t *>(smem + tslot_off);
    const int total = n * g.L;
    int ok = 1;
    if (warp == 4) {
        if (lane == 0) { // producer
            const uint32_t bytes = 2 * g.zbytes + (uint32_t)(3 * g.PX) * 64u;
            int k = 0, armed[kDwTcMaxStages];
            for (int s = 0; s < kDwTcMaxStages; ++s)
                armed[s] = -1;
            for (int it = blockIdx.x; it < total; it += gridDim.x, ++k) {
                const int s = k % NS, use = k / NS;
                if (use >= 1 && !tc::mbar_wait(empty0 + 8 * s, (use - 1) & 1, kTcMaxPolls)) {
                    ok = 0;
                    break;
                }
                const int b = it / g.L, y = it - b * g.L;
                const uint32_t st = sb + (uint32_t)s * g.stage_bytes;
                tc::mbar_arrive_expect_tx(full0 + 8 * s, bytes);
                tc::tma_load_5d(st, &zh_map, 0, 0, 0, y, b, full0 + 8 * s);
                tc::tma_load_5d(st + g.zbytes, &zl_map, 0, 0, 0, y, b, full0 + 8 * s);
                tc::tma_load_5d(st + 2 * g.zbytes, &x_map, 0, 0, -2, y - 2, b, full0 + 8 * s);
                armed[s] = use;
            }
            for (int s = 0; s < NS; ++s) // the last loads of each stage have landed before the CTA ends
                if (armed[s] >= 0 && !tc::mbar_wait(full0 + 8 * s, armed[s] & 1, kTcMaxPolls))
                    ok = 0;
        }
    } else if (warp == 5) {
        if (lane == 0) { // MMA issuer
            // tap group q: first tap (dy, dx), atom stride, M; descriptors of stage 0 at
            // position 0, advanced by 16-byte units (1024 bytes per 16 positions)
            const int cdy[4] = {-2, -1, 0, -2}, cdx[4] = {-2, -2, -2, 2};
            const uint32_t clbo[4] = {64u, 64u, 64u, (uint32_t)g.PX * 64u};
            uint64_t abase[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                abase[q] = tc::smem_desc_mn_sw64(sb + 2 * g.zbytes + (uint32_t)((cdy[q] + 2) * g.PX + cdx[q] + 2) * 64u,
                                                 clbo[q]);
            const uint64_t bbase = tc::smem_desc_mn_sw64(sb, g.zbytes);
            constexpr uint32_t id128 = tc::idesc_bf16_f32_mn(128, 64), id64 = tc::idesc_bf16_f32_mn(64, 64);
            int k = 0;
            for (int it = blockIdx.x; ok && it < total; it += gridDim.x, ++k) {
                const int s = k % NS, use = k / NS;
                if (!tc::mbar_wait(full0 + 8 * s, use & 1, kTcMaxPolls)) {
                    ok = 0;
                    break;
                }
                tc::fence_after_sync();
                const uint64_t soff = (uint64_t)(((uint32_t)s * g.stage_bytes) >> 4);
                for (int j = 0; j < g.KS; ++j) {
                    const uint64_t jo = soff + (uint64_t)(64 * j);
                    const uint32_t acc = (k > 0 || j > 0) ? 1u : 0u;
                    const uint64_t bd = bbase + jo;
                    tc::mma_bf16(tbase, abase[0] + jo, bd, id128, acc);
                    tc::mma_bf16(tbase + 64u, abase[1] + jo, bd, id128, acc);
                    tc::mma_bf16(tbase + 128u, abase[2] + jo, bd, id128, acc);
                    tc::mma_bf16(tbase + 192u, abase[3] + jo, bd, id64, acc);
                }
                tc::commit(empty0 + 8 * s); // stage s is free once this item's MMAs have read it
            }
            tc::commit(done); // every MMA issued above has completed before the drain
        }
    } else { // warps 0-3: bias gradient per item, then the drain
        // a lane sums 8 channels of every 32nd position (16-byte reads: two bytes a lane, one position a warp
        // at a time, cost as much shared-memory bandwidth as the MMAs' operands)
        float bsum[8] = {};
        int k = 0;
        for (int it = blockIdx.x; ok && it < total; it += gridDim.x, ++k) {
            const int s = k % NS, use = k / NS;
            const bool got = __any_sync(0xffffffffu, tc::mbar_wait(full0 + 8 * s, use & 1, kTcMaxPolls));
            if (!got) {
                ok = 0;
                break;
            }
            const unsigned char *zh = smem + (size_t)s * g.stage_bytes, *zl = zh + g.zbytes;
            for (int x = 8 * warp + (lane >> 2); x < g.L; x += 32) { // 64-byte swizzle
                const uint32_t off = (uint32_t)x * 64u + ((((uint32_t)lane & 3u) ^ (((uint32_t)x >> 1) & 3u)) << 4);
                const uint4 h = *reinterpret_cast<const uint4 *>(zh + off), l = *reinterpret_cast<const uint4 *>(zl + off);
                const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    bsum[2 * e] += bf16_lo(hw[e]) + bf16_lo(lw[e]);
                    bsum[2 * e + 1] += bf16_hi(hw[e]) + bf16_hi(lw[e]);
                }
            }
            __syncwarp();
            if (lane == 0)
                tc::mbar_arrive(empty0 + 8 * s);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            bsum[e] += __shfl_xor_sync(0xffffffffu, bsum[e], 4);
            bsum[e] += __shfl_xor_sync(0xffffffffu, bsum[e], 8);
            bsum[e] += __shfl_xor_sync(0xffffffffu, bsum[e], 16);
            if (lane < 4)
                bsum_s[warp * 32 + 8 * lane + e] = bsum[e];
        }
        const bool got = __any_sync(0xffffffffu, tc::mbar_wait(done, 0u, kTcMaxPolls));
        tc::fence_after_sync();
        if (!got)
            ok = 0;
        float *mine = part + (size_t)blockIdx.x * kDwPart;
        const bool any = blockIdx.x < total;
        // tap groups 0-2 (M = 128): lane 32 w + c holds tap w of the group, channel c;
        // group 3 (M = 64): lanes 0-15 of warp w hold tap (w < 2 ? 4 : 9), channel 16 (w & 1) + lane
        for (int q = 0; q < 4; ++q) {
            float v[32], u[32];
            const uint32_t col = tbase + ((uint32_t)(32 * warp) << 16) + (uint32_t)(64 * q);
            tc::ld_32x32b_x32(col, v);
            tc::ld_32x32b_x32(col + 32u, u);
            int t, c;
            if (q < 3) {
                t = 5 * q + warp; // (dy, dx) = (q - 2, warp - 2): raster index 5 (dy + 2) + dx + 2
                c = lane;
                if (q == 2 && warp == 3)
                    continue; // (0, 1) is not a tap of the mask
            } else {
                if (lane >= 16)
                    continue;
                t = warp < 2 ? 4 : 9;
                c = 16 * (warp & 1) + lane;
            }
#pragma unroll
            for (int o = 0; o < kCh; ++o)
                mine[(t * kCh + o) * kCh + c] = any ? v[o] + u[o] : 0.f;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (tid < kCh)
            mine[kTapsB * kCh * kCh + tid] = bsum_s[tid] + bsum_s[32 + tid] + bsum_s[64 + tid] + bsum_s[96 + tid];
    }
    ok = __syncthreads_and(ok);
    if (!ok && tid == 0)
        atomicExch(err, 1);
    tc::fence_after_sync();
    if (warp == 0)
        tc::tmem_free(tbase, kDwTcAlloc);
}

// Sum the per-CTA partials of k_dw32_tc in a fixed order (deterministic) into the
// canonical gradient of hidden layer `layer`: 32 outputs per CTA, warp w adds the
// parts w, w + 8, ..., then the warps in order (a thread per output over all ~300
// parts, on 53 CTAs, took 18 us).
__global__ void __launch_bounds__(256) k_dw_reduce(const float *__restrict__ part, int nparts, float *g, DevParams P,
                                                   int layer)
{
    __shared__ float ws[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    chain_wait(true);
    float v = 0.f;
    if (i < kDwPart)
        for (int k = w; k < nparts; k += 8)
            v += part[(size_t)k * kDwPart + i];
    ws[w][lane] = v;
    __syncthreads();
    if (w != 0 || i >= kDwPart)
        return;
    v = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k)
        v += ws[k][lane];
    if (i < kTapsB * kCh * kCh) {
        const int t = i / (kCh * kCh), o = (i / kCh) % kCh, c = i % kCh;
        g[canon_w(P, layer, o, c, tap_dy(t), tap_dx(t))] = v;
    } else {
        g[P.b_off[layer] + (i - kTapsB * kCh * kCh)] = v;
    }
}

// Layer-1 weight and bias gradients: gW1[o][t] = sum_p dZ1(p)[o] s(p + d_t),
// gb1[o] = sum_p dZ1(p)[o].  As k_layerD_bwd: a warp takes a row, eight positions at a
// time with 4 lanes of 8 channels each, a lane keeps its 104 sums in registers and the spins of rows y-2 .. y in the warp's shared rows.  L = 64, batch
// 512: 70 us against 125 for one lane per channel with the row's dZ1 staged in
// shared memory between CTA barriers; 268 MB of dZ1 take 40 us.
__global__ void __launch_bounds__(kEdgeThreads, kEdgeCtas)
    k_layer1_bwd_w(const bf16 *dzh, const bf16 *dzl, const int8_t *spins, float *part, int n, int L)
{
    constexpr int NW = kEdgeThreads / 32;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float R[NW][kEdgeOut1];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, o0 = (lane & 3) * 8;
    unsigned char *const Z = smem + warp * edge_bytes_1(L), *const B = Z + kStages1 * 2 * kPieceBytes;
    float *const S = reinterpret_cast<float *>(B + kStages1 * kSpinBytes);
    const int rows = n * L, step = gridDim.x * NW;
    float acc[kTapsA + 1][8];
#pragma unroll
    for (int t = 0; t <= kTapsA; ++t)
#pragma unroll
        for (int q = 0; q < 8; ++q)
            acc[t][q] = 0.f;
    chain_wait(true);
    Piece next{(int)blockIdx.x * NW + warp, 0}, cur = next;
    int next_stage = 0, next_win = kStages1 - 1, stage = 0, win = kStages1 - 1;
    // The spins of rows max(y - 2, 0) .. y are one run of bytes, copied from the 16-byte
    // boundary before it (the spins start on one) and no further than their end.
    auto spin_run = [&](int item, const int8_t *&from, int &off) {
        const size_t first = (size_t)(item - min(item % L, 2)) * L;
        off = (int)(first & 15);
        from = spins + (first - off);
        return (int)((size_t)(item + 1) * L - (first - off)); // bytes from `from` to the end of row y
    };
    auto fetch = [&] {
        if (next.item < rows) {
            const size_t at = ((size_t)next.item * L + next.x) * kCh;
            const unsigned char *h = reinterpret_cast<const unsigned char *>(dzh + at),
                                *l = reinterpret_cast<const unsigned char *>(dzl + at);
            unsigned char *dst = Z + next_stage * 2 * kPieceBytes;
            const int units = min(32, L - next.x) * 4;
            for (int i = lane; i < units; i += 32) {
                cp16(dst + 16 * i, h + 16 * i);
                cp16(dst + kPieceBytes + 16 * i, l + 16 * i);
            }
            if (next.x == 0) {
                next_win = next_win + 1 == kStages1 ? 0 : next_win + 1;
                const int8_t *from;
                int off;
                const int bytes = spin_run(next.item, from, off);
                if (16 * lane < bytes)
                    cp16(B + next_win * kSpinBytes + 16 * lane, from + 16 * lane, min(16, bytes - 16 * lane));
            }
            next.next(L, step);
            next_stage = next_stage + 1 == kStages1 ? 0 : next_stage + 1;
        }
        cp_commit();
    };
    for (int k = 0; k < kStages1 - 1; ++k)
        fetch();
    while (cur.item < rows) {
        cp_wait<kStages1 - 2>();
        __syncwarp();
        fetch();
        if (cur.x == 0) { // the row's spins as floats, zero outside the lattice
            win = win + 1 == kStages1 ? 0 : win + 1;
            const int8_t *from;
            int off;
            spin_run(cur.item, from, off);
            const int up = min(cur.item % L, 2); // rows above y inside the lattice
            const signed char *src = reinterpret_cast<const signed char *>(B + win * kSpinBytes + off);
            for (int r = 0; r < 3; ++r)
                for (int x = lane - 2; x < L + 2; x += 32)
                    S[r * (L + 4) + x + 2] =
                        r + up >= 2 && x >= 0 && x < L ? (float)src[(r + up - 2) * L + x] : 0.f;
            __syncwarp();
        }
        const float *s0 = S + 2 * (L + 4) + cur.x + 2;
        const unsigned char *zs = Z + stage * 2 * kPieceBytes + o0 * 2;
        const int len = min(32, L - cur.x);
#pragma unroll 1
        for (int x = lane >> 2; x < len; x += 8) {
            const uint4 h = *reinterpret_cast<const uint4 *>(zs + x * (kCh * 2));
            const uint4 l = *reinterpret_cast<const uint4 *>(zs + kPieceBytes + x * (kCh * 2));
            const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
            float z[8]; // value = hi + lo
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                z[2 * k] = __uint_as_float(hw[k] << 16) + __uint_as_float(lw[k] << 16);
                z[2 * k + 1] = __uint_as_float(hw[k] & 0xFFFF0000u) + __uint_as_float(lw[k] & 0xFFFF0000u);
            }
#pragma unroll
            for (int t = 0; t < kTapsA; ++t) {
                const float s = s0[tap_dy(t) * (L + 4) + x + tap_dx(t)];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    acc[t][q] += z[q] * s;
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                acc[kTapsA][q] += z[q];
        }
        cur.next(L, step);
        stage = stage + 1 == kStages1 ? 0 : stage + 1;
    }
#pragma unroll
    for (int t = 0; t <= kTapsA; ++t)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            float v = acc[t][q];
            v += __shfl_xor_sync(0xffffffffu, v, 4);
            v += __shfl_xor_sync(0xffffffffu, v, 8);
            v += __shfl_xor_sync(0xffffffffu, v, 16);
            if (lane < 4)
                R[warp][(o0 + q) * (kTapsA + 1) + t] = v;
        }
    __syncthreads();
    for (int i = tid; i < kEdgeOut1; i += blockDim.x) {
        float v = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w)
            v += R[w][i];
        part[(size_t)i * gridDim.x + blockIdx.x] = v;
    }
}

__global__ void k_adam(float *p, float *m, float *v, const float *g, size_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    chain_wait(true);
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

}  // namespace
}  // namespace van
}  // namespace mc

namespace mc {
namespace van {
namespace {

constexpr uint32_t kTagVanSample = 0x21000000u; // sampler uniforms
constexpr uint32_t kTagVanMH = 0x22000000u;     // accept uniform and global flip
constexpr int kSampleTile = 32;                 // samples per sampler CTA (two m16 tiles)
constexpr int kTapBytes = kSampleTile * kCh * 2; // one tap of the 32 samples of a CTA: 2 KB
constexpr int kTileBytes = kTapsA * kTapBytes;      // a gathered tile [12 taps][32 samples][32 ch]
constexpr int kSampleMaxBufs = 3;                   // gathered hidden-layer tiles in flight
constexpr size_t kSampleSmemLimit = 232448;         // 227 KB, the opt-in maximum per block
constexpr int kGroupThreads = 128;                  // main warps 0-3, side warps 4-7
constexpr int kSampleThreads = 2 * kGroupThreads + 32; // + the producer warp (gathers)

// Ring arrays of the sampler, per layer [32-sample block][row % 3][x][32 samples]
// [32 ch]: a block's five taps of one row are one contiguous run (one bulk
// copy), and the 16-byte channel chunks of sample s are stored in the order
// c ^ ((s >> 1) & 3), so that eight consecutive samples' rows of one chunk fall
// on distinct shared-memory banks when a tile is read by ldmatrix.  The same
// layout holds the layer values of the current position (Hc) and, per tap, the
// weights (row = output channel).
__device__ __forceinline__ int ring_elem(int s, int o) { return s * kCh + ((((o >> 3) ^ (s >> 1)) & 3) << 3) + (o & 7); }

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

// Named barriers of the sampler's warp groups (0 is __syncthreads).
constexpr int kBarMain = 1, kBarSide = 2;
__device__ __forceinline__ void group_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Wait for an mbarrier phase.  A wait that gives up latches *err and sets the
// CTA's abort flag; once the flag is set every wait returns at once, so that
// all threads run to the end (no barrier is left short of threads) and the
// sampled values are garbage, reported through *err.
__device__ __forceinline__ void wait_phase(uint32_t bar, uint32_t parity, volatile int *abort, int *err)
{
    for (int it = 0; it < kTcMaxPolls; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (done || *abort)
            return;
    }
    *abort = 1;
    atomicExch(err, 1);
}

// The tap of position k = y L + x whose position is k - 1 (the one just sampled),
// or -1: tap 11 (dx = -1) for x > 0; for x = 0 the position k - 1 is (y - 1,
// L - 1), a tap only when L = 2 (tap 8).  In either case no later tap of 0..11
// is inside the lattice.
__device__ __forceinline__ int newest_tap(int L, int y, int x) { return x > 0 ? 11 : (L == 2 && y > 0 ? 8 : -1); }

// One 16 x 16 output tile of a 32 -> 32 layer for this warp (m-tile w >> 1,
// n-tiles 2 (w & 1) + 0, 1): accumulate one tap (K = 32) from the [32][32]
// operand at shared address `a` with the tap's weights at `wt`.
__device__ __forceinline__ void mma_tap(float (&c0)[4], float (&c1)[4], uint32_t a, uint32_t wt, uint32_t ao0,
                                        uint32_t ao1, uint32_t bo0, uint32_t bo1)
{
    uint32_t a0, a1, a2, a3, b0, b1, b2, b3;
    ldsm_x4(a + ao0, a0, a1, a2, a3);
    ldsm_x4(wt + bo0, b0, b1, b2, b3);
    mma_bf16(c0, a0, a1, a2, a3, b0, b1);
    mma_bf16(c1, a0, a1, a2, a3, b2, b3);
    ldsm_x4(a + ao1, a0, a1, a2, a3);
    ldsm_x4(wt + bo1, b0, b1, b2, b3);
    mma_bf16(c0, a0, a1, a2, a3, b0, b1);
    mma_bf16(c1, a0, a1, a2, a3, b2, b3);
}

// Autoregressive sampling, one position k = y L + x at a time in raster order,
// 32 samples per CTA.  Layer l at position k sums its taps over the 12 earlier
// positions (values of layer l - 1 from earlier steps, gathered from that
// layer's ring array) and tap 12, the value of layer l - 1 at k itself; s_k =
// +1 iff u < sigmoid(f_k), u from Philox (k >> 2, round, TAG_SAMPLE, id) word
// k & 3, and log q accumulates log sigmoid(s_k f_k) in FP64.  Warp roles:
//   * main warps 0-3 run the chain of dependent layers of step k: the first
//     layer (its partial plus w s_{k-1}), the hidden layers on the tensor cores
//     (a 16 x 16 output tile per warp, 26 MMA k-steps), the output layer (its
//     partial plus tap 12) and the draw; they write each hidden value to the
//     layer's ring array (followed by a proxy fence, for the bulk copies);
//   * side warps 4-7 compute, off that chain, the output layer's partial sum
//     over its 12 earlier taps for step k and the first layer's partial over
//     its taps other than s_{k-1} for step k + 1, and accumulate log q -- in
//     the order of one pass over all taps, so that the result is that of the
//     plain evaluation;
//   * a producer warp gathers, per (position, consuming layer g = 1..G, G = D -
//     1), the 12 earlier taps of the CTA's samples from the ring array by bulk
//     copies into one of `nbuf` tiles (taps outside the lattice copy a zero
//     page), in the sequence q = k G + g - 1.  Main releases a hidden layer's
//     tile after the layer; side releases the output layer's tile of step k
//     once main has finished step k, so that every release comes after the ring
//     stores that the gather nbuf later may read (nbuf <= G).
// Signals between main and side are mbarriers with one completion per step:
// E0 (first layer of step k done: its partial consumed), E1 (step k done:
// output partial consumed, s_k drawn), R0 (first-layer partial of step k
// written), R1 (output partial of step k written).  Every wait is bounded; one
// that gives up latches *err and sets an abort flag after which all waits return
// at once, so that every thread still reaches every barrier.
__global__ void __launch_bounds__(kSampleThreads, 1) k_sample(const bf16 *__restrict__ wh, const float *__restrict__ w1,
                                                   const float *__restrict__ wD, const float *__restrict__ bias, int D,
                                                   int L, int n, int nbuf, bf16 *hist, const bf16 *zero, int8_t *out,
                                                   double *logq, PhiloxKey key, uint32_t round, const uint32_t *ids,
                                                   int *err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int nh = D - 2, G = nh + 1;
    bf16 *Ws = reinterpret_cast<bf16 *>(smem);                      // [nh][13][32 o][32 c] (ring_elem)
    bf16 *Ts = Ws + (size_t)nh * kTapsB * kCh * kCh;                // nbuf + 1 x [12][32][32] gathered taps
    bf16 *Hc = Ts + (size_t)(nbuf + 1) * kTapsA * kSampleTile * kCh; // [2 (layer & 1)][32][32] values at k
    float *P0 = reinterpret_cast<float *>(Hc + (size_t)2 * kSampleTile * kCh); // [32 s][32 o] first-layer partial
    float *Po = P0 + kSampleTile * kCh;                             // [32 s][8 parts] output partial
    float *W1 = Po + kSampleTile * 8;                               // [12][32] (tap-major)
    float *WD = W1 + kCh * kTapsA;                                  // [13][32]
    float *Bs = WD + kTapsB * kCh;                                  // [(D-1) 32 + 1]
    float *LT = Bs + (D - 1) * kCh + 1;                             // [32] s_k f_k of the last draw
    int8_t *Sr = reinterpret_cast<int8_t *>(LT + kSampleTile);      // [32][3][L] spins of rows y-2..y
    const uint32_t bar0 = (smem_u32(Sr + kSampleTile * 3 * L) + 7u) & ~7u;
    const uint32_t full0 = bar0, empty0 = bar0 + 8u * (kSampleMaxBufs + 1), E0 = empty0 + 8u * (kSampleMaxBufs + 1),
                   E1 = E0 + 8u, R0 = E0 + 16u, R1 = E0 + 24u;
    __shared__ int abort_flag;
    volatile int *abort = &abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s0 = blockIdx.x * kSampleTile;
    for (int i = tid; i < nh * kTapsB * kCh * kCh; i += blockDim.x) {
        const int row = i / kCh, c = i % kCh, o = row % kCh; // row = (l, t, o)
        Ws[(size_t)(row - o) * kCh + ring_elem(o, c)] = wh[i];
    }
    for (int i = tid; i < kCh * kTapsA; i += blockDim.x)
        W1[(i % kTapsA) * kCh + i / kTapsA] = w1[i]; // w1 is [o][t]
    for (int i = tid; i < kTapsB * kCh; i += blockDim.x)
        WD[i] = wD[i];
    for (int i = tid; i < (D - 1) * kCh + 1; i += blockDim.x)
        Bs[i] = bias[i];
    if (tid == 0) {
        abort_flag = 0;
        for (int b = 0; b <= nbuf; ++b) {
            tc::mbar_init(full0 + 8u * b, 1);
            tc::mbar_init(empty0 + 8u * b, 1);
        }
        for (int j = 0; j < 4; ++j)
            tc::mbar_init(E0 + 8u * j, 1);
    }
    const int nsb = (n + kSampleTile - 1) / kSampleTile;
    const size_t pblk = (size_t)kSampleTile * kCh;                  // ring elements per position of a block
    const size_t lstride = (size_t)nsb * 3 * L * pblk;             // ring elements per layer
    bf16 *ring = hist + (size_t)blockIdx.x * 3 * L * pblk;         // this CTA's block of layer 0
    const int P = L * L, Q = P * G;
    const uint32_t ts0 = smem_u32(Ts), ws0 = smem_u32(Ws);
    __syncthreads();

    if (warp == 8) { // ---------------------------------------------------------------- producer
        int issued = 0;
        for (int q = 0; q < Q; ++q) {
            const int kq = q / G, g = q - kq * G + 1, yq = kq / L, xq = kq - yq * L;
            // hidden-layer gathers cycle through slots 0..nbuf-1, output-layer gathers use slot nbuf
            const int hq = kq * nh + g - 1, slot = g < G ? hq % nbuf : nbuf, use = g < G ? hq / nbuf : kq;
            if (use > 0)
                wait_phase(empty0 + 8u * (uint32_t)slot, (uint32_t)(use - 1) & 1u, abort, err);
            if (*abort)
                break;
            const uint32_t bar = full0 + 8u * (uint32_t)slot;
            if (lane == 0)
                tc::mbar_arrive_expect_tx(bar, kTileBytes);
            __syncwarp();
            // lane 3 r + p copies part p (0 zeros left of the lattice, 1 the positions inside, 2 zeros right
            // of it) of tap row r: rows y-2 and y-1 (taps 5 r .. 5 r + 4, dx = -2..2), row y (taps 10, 11)
            const int r = lane / 3, part = lane - 3 * r;
            if (r < 3) {
                const int ntap = r < 2 ? 5 : 2, yy = yq - 2 + r, xlo = xq - 2;
                int zl = ntap, nd = 0;
                if (yy >= 0) {
                    zl = xlo < 0 ? -xlo : 0;
                    nd = ntap - zl - max(0, xlo + ntap - L);
                }
                const int first = part == 0 ? 0 : part == 1 ? zl : zl + nd;
                const int cnt = part == 0 ? zl : part == 1 ? nd : ntap - zl - nd;
                if (cnt > 0) {
                    const bf16 *src = part == 1 ? ring + (size_t)(g - 1) * lstride + ((size_t)(yy % 3) * L + xlo + zl) * pblk
                                                : zero;
                    bulk_g2s(ts0 + (uint32_t)(slot * kTileBytes + (5 * r + first) * kTapBytes), src,
                             (uint32_t)cnt * kTapBytes, bar);
                }
            }
            issued = q + 1;
        }
        // copies still in flight (the consumers stopped early): let them land before the CTA ends
        if (lane == 0 && *abort) {
            uint32_t seen = 0; // the last fill of each slot
            for (int q = issued - 1; q >= 0 && seen != (2u << nbuf) - 1u; --q) {
                const int kq = q / G, g = q - kq * G + 1, hq = kq * nh + g - 1;
                const int slot = g < G ? hq % nbuf : nbuf, use = g < G ? hq / nbuf : kq;
                if (!(seen >> slot & 1u)) {
                    seen |= 1u << slot;
                    tc::mbar_wait(full0 + 8u * (uint32_t)slot, (uint32_t)use & 1u, kTcMaxPolls);
                }
            }
        }
        return;
    }

    if (warp >= 4) { // ---------------------------------------------------------------------- side
        const int h = tid - 128, s = h >> 2, sub = h & 3;
        double lq = 0.0; // owned by side thread s < 32
        // the first-layer partial of position k: bias + taps 0..11 inside, except the one at k - 1
        auto first_partial = [&](int k) {
            const int y = k / L, x = k % L, tn = newest_tap(L, y, x), o0 = sub * 8;
            float acc[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                acc[j] = Bs[o0 + j];
#pragma unroll
            for (int t = 0; t < kTapsA; ++t) {
                const int yy = y + tap_dy(t), xx = x + tap_dx(t);
                if (t != tn && yy >= 0 && xx >= 0 && xx < L) {
                    const float v = (float)Sr[(s * 3 + yy % 3) * L + xx];
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        acc[j] = __fmaf_rn(W1[t * kCh + o0 + j], v, acc[j]);
                }
            }
            *reinterpret_cast<float4 *>(P0 + s * kCh + o0) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            *reinterpret_cast<float4 *>(P0 + s * kCh + o0 + 4) = make_float4(acc[4], acc[5], acc[6], acc[7]);
        };
        first_partial(0);
        group_sync(kBarSide, kGroupThreads);
        if (h == 0)
            tc::mbar_arrive(R0);
        for (int k = 0; k < P; ++k) {
            const int y = k / L, x = k % L;
            if (k > 0) {
                wait_phase(E1, (uint32_t)(k - 1) & 1u, abort, err); // step k - 1 done
                if (h == 0) // its output tile: every ring store of step k - 1 is in
                    tc::mbar_arrive(empty0 + 8u * (uint32_t)nbuf);
                if (h < kSampleTile && s0 + h < n)
                    lq += (double)log_sigmoid(LT[h]);
            }
            // ---- output partial of step k: taps 0..11 inside, 8 parts of 4 channels per sample
            wait_phase(full0 + 8u * (uint32_t)nbuf, (uint32_t)k & 1u, abort, err);
            {
                const bf16 *tl = Ts + (size_t)nbuf * kTapsA * kSampleTile * kCh;
                float po0 = 0.f, po1 = 0.f;
                for (int t = 0; t < kTapsA; ++t) {
                    const int yy = y + tap_dy(t), xx = x + tap_dx(t);
                    if (yy < 0 || xx < 0 || xx >= L)
                        continue;
                    const bf16 *src = tl + t * kSampleTile * kCh;
                    const uint2 hv0 = *reinterpret_cast<const uint2 *>(src + ring_elem(s, sub * 8));
                    const uint2 hv1 = *reinterpret_cast<const uint2 *>(src + ring_elem(s, sub * 8 + 4));
                    const float4 w0 = *reinterpret_cast<const float4 *>(WD + t * kCh + sub * 8);
                    const float4 wv1 = *reinterpret_cast<const float4 *>(WD + t * kCh + sub * 8 + 4);
                    po0 = __fmaf_rn(w0.x, bf16_lo(hv0.x), po0);
                    po0 = __fmaf_rn(w0.y, bf16_hi(hv0.x), po0);
                    po0 = __fmaf_rn(w0.z, bf16_lo(hv0.y), po0);
                    po0 = __fmaf_rn(w0.w, bf16_hi(hv0.y), po0);
                    po1 = __fmaf_rn(wv1.x, bf16_lo(hv1.x), po1);
                    po1 = __fmaf_rn(wv1.y, bf16_hi(hv1.x), po1);
                    po1 = __fmaf_rn(wv1.z, bf16_lo(hv1.y), po1);
                    po1 = __fmaf_rn(wv1.w, bf16_hi(hv1.y), po1);
                }
                *reinterpret_cast<float2 *>(Po + s * 8 + sub * 2) = make_float2(po0, po1);
            }
            group_sync(kBarSide, kGroupThreads);
            if (h == 0)
                tc::mbar_arrive(R1);
            // ---- first-layer partial of step k + 1 (its spins at positions <= k - 1 are drawn)
            if (k + 1 < P) {
                wait_phase(E0, (uint32_t)k & 1u, abort, err); // the partial of step k consumed
                first_partial(k + 1);
                group_sync(kBarSide, kGroupThreads);
                if (h == 0)
                    tc::mbar_arrive(R0);
            }
        }
        wait_phase(E1, (uint32_t)(P - 1) & 1u, abort, err); // the last draw
        if (h < kSampleTile && s0 + h < n)
            logq[s0 + h] = lq + (double)log_sigmoid(LT[h]);
        return;
    }

    // ----------------------------------------------------------------------------------------- main
    const int c = tid, s = c >> 2, sub = c & 3, gs = s0 + s;
    const int mt = warp >> 1, np = warp & 1; // this warp's 16 x 16 output tile of a hidden layer
    const int ar = mt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8, br = (2 * np + (lane >> 4)) * 8 + (lane & 7);
    const uint32_t ao0 = 2u * ring_elem(ar, (lane >> 4) * 8), ao1 = 2u * ring_elem(ar, 16 + (lane >> 4) * 8);
    const uint32_t bo0 = 2u * ring_elem(br, ((lane >> 3) & 1) * 8), bo1 = 2u * ring_elem(br, 16 + ((lane >> 3) & 1) * 8);
    const int fg = lane >> 2, ft = lane & 3; // accumulator fragment: rows fg, fg + 8; columns 2 ft, 2 ft + 1
    uint32_t my_id = 0;
    if (sub == 0 && gs < n)
        my_id = ids ? ids[gs] : (uint32_t)gs;
    for (int k = 0; k < P; ++k) {
        const int y = k / L, x = k % L, tn = newest_tap(L, y, x);
        bf16 *hpos = ring + ((size_t)(y % 3) * L + x) * pblk; // position k in the ring of layer 0
        // ---- first layer: partial + w s_{k-1}
        wait_phase(R0, (uint32_t)k & 1u, abort, err);
        {
            const int o0 = sub * 8;
            float v = 0.f;
            if (tn >= 0)
                v = (float)Sr[(s * 3 + (y + tap_dy(tn)) % 3) * L + x + tap_dx(tn)];
            float a[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                a[j] = P0[s * kCh + o0 + j];
                if (tn >= 0)
                    a[j] = __fmaf_rn(W1[tn * kCh + o0 + j], v, a[j]);
            }
            const uint4 pk =
                make_uint4(pack_bf16x2(fmaxf(a[0], 0.f), fmaxf(a[1], 0.f)), pack_bf16x2(fmaxf(a[2], 0.f), fmaxf(a[3], 0.f)),
                           pack_bf16x2(fmaxf(a[4], 0.f), fmaxf(a[5], 0.f)), pack_bf16x2(fmaxf(a[6], 0.f), fmaxf(a[7], 0.f)));
            *reinterpret_cast<uint4 *>(Hc + ring_elem(s, o0)) = pk;
            *reinterpret_cast<uint4 *>(hpos + ring_elem(s, o0)) = pk;
            asm volatile("fence.proxy.async.global;" ::: "memory");
        }
        group_sync(kBarMain, kGroupThreads);
        if (c == 0)
            tc::mbar_arrive(E0);
        // ---- hidden layers (tensor cores): M = 32 samples, N = 32, K = 13 x 32
        for (int l = 1; l <= nh; ++l) {
            const int hq = k * nh + l - 1, slot = hq % nbuf;
            const uint32_t tile = ts0 + (uint32_t)(slot * kTileBytes);
            const uint32_t wl = ws0 + (uint32_t)((l - 1) * kTapsB * kCh * kCh * 2);
            wait_phase(full0 + 8u * (uint32_t)slot, (uint32_t)(hq / nbuf) & 1u, abort, err);
            float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
            for (int t = 0; t < kTapsA; ++t)
                mma_tap(c0, c1, tile + (uint32_t)t * kTapBytes, wl + (uint32_t)t * kCh * kCh * 2, ao0, ao1, bo0, bo1);
            mma_tap(c0, c1, smem_u32(Hc + (size_t)((l - 1) & 1) * kSampleTile * kCh), wl + (uint32_t)kTapsA * kCh * kCh * 2,
                    ao0, ao1, bo0, bo1);
            bf16 *hn = Hc + (size_t)(l & 1) * kSampleTile * kCh;
            bf16 *hr = hpos + (size_t)l * lstride;
            // bias, ReLU, BF16 of n-tile j's fragment (rows fg, fg + 8), to Hc and the ring
            auto store = [&](const float(&acc)[4], int j) {
                const int o = (2 * np + j) * 8 + 2 * ft;
                const float bo = Bs[l * kCh + o], b1v = Bs[l * kCh + o + 1];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) {
                    const int sr = mt * 16 + fg + 8 * hh;
                    const uint32_t v = pack_bf16x2(fmaxf(acc[2 * hh] + bo, 0.f), fmaxf(acc[2 * hh + 1] + b1v, 0.f));
                    *reinterpret_cast<uint32_t *>(hn + ring_elem(sr, o)) = v;
                    *reinterpret_cast<uint32_t *>(hr + ring_elem(sr, o)) = v;
                }
            };
            store(c0, 0);
            store(c1, 1);
            asm volatile("fence.proxy.async.global;" ::: "memory");
            group_sync(kBarMain, kGroupThreads);
            if (c == 0)
                tc::mbar_arrive(empty0 + 8u * (uint32_t)slot);
        }
        // ---- output layer: partial + tap 12, then the draw
        wait_phase(R1, (uint32_t)k & 1u, abort, err);
        {
            const bf16 *hp = Hc + (size_t)(nh & 1) * kSampleTile * kCh;
            float a2[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int part = sub * 2 + j;
                float acc = Po[s * 8 + part];
                const uint2 hv = *reinterpret_cast<const uint2 *>(hp + ring_elem(s, part * 4));
                const float4 w = *reinterpret_cast<const float4 *>(WD + kTapsA * kCh + part * 4);
                acc = __fmaf_rn(w.x, bf16_lo(hv.x), acc);
                acc = __fmaf_rn(w.y, bf16_hi(hv.x), acc);
                acc = __fmaf_rn(w.z, bf16_lo(hv.y), acc);
                acc = __fmaf_rn(w.w, bf16_hi(hv.y), acc);
                a2[j] = acc;
            }
            float f = a2[0] + a2[1];
            f += __shfl_xor_sync(0xffffffffu, f, 1);
            f += __shfl_xor_sync(0xffffffffu, f, 2);
            f += Bs[(D - 1) * kCh];
            if (sub == 0 && gs < n) {
                const uint4 r = philox4x32_10(make_uint4((uint32_t)k >> 2, round, kTagVanSample, my_id), key);
                const uint32_t rk = (k & 2) ? ((k & 1) ? r.w : r.z) : ((k & 1) ? r.y : r.x);
                const float sp = uniform_open0(rk) < sigmoid(f) ? 1.f : -1.f;
                Sr[(s * 3 + y % 3) * L + x] = (int8_t)sp;
                out[((size_t)gs * L + y) * L + x] = (int8_t)sp;
                LT[s] = sp * f;
            }
        }
        group_sync(kBarMain, kGroupThreads);
        if (c == 0)
            tc::mbar_arrive(E1);
    }
}

// ------------------------------------------------- sampler, columns streamed
// The same sampling as k_sample (bit for bit: every hidden value adds its taps in raster
// order, 16 channels at a time), arranged so that the chain of a step holds nothing that
// could be computed before it.  The latency of a step is what bounds the sampler: L^2
// of them follow one another whatever the batch.
//
//   * A chain warp owns 16 samples and runs first layer, hidden layers, output layer and
//     draw in its registers: a layer's accumulator fragment, packed to BF16, is the next
//     layer's operand fragment (m16n8k16), so that a layer costs 8 matrix instructions
//     (tap 12) and an epilogue, with no shared-memory round trip between layers.
//   * For each hidden layer and 16 samples a helper warp prepares the accumulators over
//     taps 0..11.  Taps 0..9 are of the two rows above, known for a whole row: the helper
//     computes them for the next block of 4 positions while the chain works on the
//     current one, a quarter of the block's taps per step, so that a weight fragment
//     serves 4 positions and a column of activations up to 5 taps.  Taps 10 and 11 (the
//     two positions just before) are added step by step.
//   * For each 16 samples a warp prepares the first layer's sum over the spins other than
//     the last one and the uniforms, and two warps the output layer's sum over taps 0..11
//     and log q: after a step the terms of its own values first, since the chain waits for
//     them, then the upper rows' terms of the position after.
//
// Activations of earlier rows stay in the ring arrays in global memory, written and read
// back by the same lane in its own order (an asynchronous 16-byte copy per lane and half
// a column: nothing crosses lanes).  A helper publishes position k's accumulators, the
// chain loads them, then publishes the layer's input at k, from which the helper finishes
// position k + 1: each slot is read before the next value is written.  No register
// spills and loops short enough to share the instruction cache are what the roles'
// registers and code are cut for: 12 bytes of spills cost 8%, 56 missed lines a step 15%.
//
// us per position at L = 64, depth 6, 4096 samples: 1.64 against 4.45 for k_sample (depth 5:
// 1.46 / 3.63, depth 4: 1.11 / 2.94, depth 3: 1.10 / 2.18; depth 6 on L = 8 to 50: 1.65 to 2.0
// / 4.5 to 4.9).  Tensor throughput would allow 0.87 (832 matrix instructions per step and SM,
// 208 per sub-core at 8 cycles); the chain's latency is ~3100 cycles, of them ~1300 in its
// matrix instructions, which share the tensor cores with the helpers', and the shared-memory
// pipe is 85% busy with weights, columns and hand-overs.
constexpr int kHalf = 16;                     // samples of a chain warp
constexpr int kColBytes = kHalf * kCh * 2;    // 16 samples of one position: 1 KB
constexpr int kPipeTiles = 7;                 // columns a helper has staged or in flight
constexpr int kPipeSide = 6;                  // columns (of two rows) of a side warp
constexpr int kPipeHidden = 4;                // hidden layers: 8 helper warps
constexpr int kPipeMinL = 8;                  // a block's columns are known a block ahead
constexpr int kPipeThreads = 32 * (2 * kPipeHidden + 8); // helpers; chains and first-layer warps; output warps
constexpr int kPipeRegs = 128; // at launch, a thread; then by warp group: helpers, chains, output warps
constexpr int kHelperRegs = 184, kChainRegs = 88, kOutRegs = 56;
static_assert(2 * kHelperRegs + kChainRegs + kOutRegs == 4 * kPipeRegs, "the split is the launch's total");
// words of a row's spins as bits, from bit 2 on (read two at a time)
__host__ __device__ inline int spin_words(int L) { return (L - 1) / 32 + 2; }

struct PipeSmem { // byte offsets
    int w, fifo, p, h, p0, win, hn, po, w1, wd, bias, draw, u, bits, bar, total;
};
__host__ __device__ inline PipeSmem pipe_smem(int D, int L)
{
    const int nh = D - 2;
    PipeSmem o{};
    int at = 0;
    auto take = [&](int bytes) {
        const int r = at;
        at += (bytes + 15) & ~15;
        return r;
    };
    o.w = take(nh * kTapsB * kCh * kCh * 2);       // fragments [l][t][k-step][n-tile pair][lane]
    o.fifo = take(nh * 2 * kPipeTiles * kColBytes); // per helper
    o.p = take(nh * 2 * kHalf * kCh * 4);          // accumulators of position k, fragments
    o.h = take(nh * 2 * kColBytes);                // input of hidden layer l at k, fragments
    o.p0 = take(2 * 2 * kHalf * kCh * 4);          // first-layer sums, two steps, fragments
    o.win = take(2 * kPipeSide * 2 * kColBytes);   // the output layer's window of two rows
    o.hn = take(2 * kColBytes);                    // last hidden layer at k, ring_elem order
    o.po = take(2 * 32 * 16);                      // output-layer sums, by the chain's lanes
    o.w1 = take(kTapsA * kCh * 4);
    o.wd = take(kTapsB * kCh * 4);
    o.bias = take(((D - 1) * kCh + 1) * 4);
    o.draw = take(2 * kHalf * 8);                  // s_k, s_k f_k
    o.u = take(2 * 2 * kHalf * 4);                 // uniforms, two steps
    o.bits = take(2 * kHalf * 3 * spin_words(L) * 4);
    o.bar = take((2 * nh + 2) * 8);
    o.total = at;
    return o;
}

// D(16 x 8) += A(16 x 16) B(16 x 8), A as one uint4 fragment.
__device__ __forceinline__ void mma16(float (&c)[4], const uint4 &a, uint32_t b0, uint32_t b1)
{
    mma_bf16(c, a.x, a.y, a.z, a.w, b0, b1);
}
// c += A B over one 16-channel step and all four n-tiles; w: the lane's two weight quads.
__device__ __forceinline__ void mma_step(float (&c)[4][4], const uint4 &a, const uint4 &w0, const uint4 &w1)
{
    mma16(c[0], a, w0.x, w0.y);
    mma16(c[1], a, w0.z, w0.w);
    mma16(c[2], a, w1.x, w1.y);
    mma16(c[3], a, w1.z, w1.w);
}

// The channel of accumulator column i (n-tile i / 8).  The last hidden layer's columns are
// ordered so that a lane of the fragment holds four channels of a part of the output layer's
// sum one after the other (4 t + 0..3 and 16 + 4 t + 0..3 for lane t of a row).
__host__ __device__ inline int pipe_channel(bool last, int i)
{
    return last ? (i >> 4) * 16 + ((i >> 1) & 3) * 4 + ((i >> 3) & 1) * 2 + (i & 1) : i;
}

// wait_phase for whole warps: the lanes agree before the branch, which is then uniform (a
// loop that lanes may leave one by one costs ~100 cycles more, and the chain waits
// six times a step).
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int *abort, int *err)
{
#pragma unroll 1
    for (int it = 0; it < kTcMaxPolls; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (__all_sync(0xffffffffu, done))
            return true;
        if (__any_sync(0xffffffffu, *abort))
            return false;
    }
    *abort = 1;
    atomicExch(err, 1);
    return false;
}

// What the chain waits for (nh + 2 times a step) is handed over by named barriers, at which
// the preparing warps arrive and only the chain warp waits: a completed mbarrier wait took
// it ~200 cycles.  The next arrival always follows from a signal the chain gives after its
// wait.  The warps that wait for the chain do so by mbarriers, several on the same one.
constexpr int kReadyHidden = 1, kReadyFirst = kReadyHidden + 2 * kPipeHidden, kReadyOut = kReadyFirst + 2;
__device__ __forceinline__ void ready(int id, int threads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
// After a wait that gave up: arrive until the chain, which stops at its next step, has left.
__device__ __forceinline__ void release_chain(int id, int threads, volatile int *done)
{
#pragma unroll 1
    for (int it = 0; it < kTcMaxPolls && !__any_sync(0xffffffffu, *done); ++it)
        ready(id, threads);
}

// Registers of a warp group, out of what the block was launched with.
template <int REGS>
__device__ __forceinline__ void regs_grow()
{
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS));
}
template <int REGS>
__device__ __forceinline__ void regs_shrink()
{
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS));
}

__global__ void __launch_bounds__(kPipeThreads, 1)
    k_sample_pipe(const bf16 *__restrict__ wh, const float *__restrict__ w1, const float *__restrict__ wD,
                  const float *__restrict__ bias, int D, int L, int n, bf16 *hist, int8_t *out, double *logq, PhiloxKey key,
                  uint32_t round, const uint32_t *ids, int *err)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int abort_flag, chain_done[2];
    volatile int *abort = &abort_flag;
    const int nh = D - 2, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s0 = blockIdx.x * kSampleTile, P = L * L;
    bool ok = true; // no wait has given up
    const PipeSmem o = pipe_smem(D, L);
    const int words = spin_words(L);
    // ---- weights (fragment order), biases, cleared spins, barriers
    for (int i = tid; i < nh * kTapsB * 512; i += kPipeThreads) { // 32-bit words
        const int q = i & 3, ln = (i >> 2) & 31, pair = (i >> 7) & 1, ks = (i >> 8) & 1, lt = i >> 9;
        const int oc = pipe_channel(lt / kTapsB == nh - 1, (2 * pair + (q >> 1)) * 8 + (ln >> 2)),
                  c = ks * 16 + (q & 1) * 8 + (ln & 3) * 2;
        reinterpret_cast<uint32_t *>(smem + o.w)[i] =
            *reinterpret_cast<const uint32_t *>(wh + ((size_t)lt * kCh + oc) * kCh + c);
    }
    float *W1 = reinterpret_cast<float *>(smem + o.w1), *WD = reinterpret_cast<float *>(smem + o.wd),
          *Bs = reinterpret_cast<float *>(smem + o.bias);
    for (int i = tid; i < kCh * kTapsA; i += kPipeThreads) { // w1 is [o][t]; in the order of a lane's fragment columns
        const int oc = i / kTapsA;
        W1[(i % kTapsA) * kCh + ((oc >> 1) & 3) * 8 + (oc >> 3) * 2 + (oc & 1)] = w1[i];
    }
    for (int i = tid; i < kTapsB * kCh; i += kPipeThreads)
        WD[i] = wD[i];
    for (int i = tid; i < (D - 1) * kCh + 1; i += kPipeThreads)
        Bs[i] = bias[i / kCh == nh ? nh * kCh + pipe_channel(true, i % kCh) : i];
    for (int i = tid; i < 2 * kHalf * 3 * words; i += kPipeThreads)
        reinterpret_cast<uint32_t *>(smem + o.bits)[i] = 0u;
    const uint32_t bars = smem_u32(smem + o.bar);
    if (tid == 0) {
        abort_flag = chain_done[0] = chain_done[1] = 0;
        for (int j = 0; j < 2 * nh + 2; ++j)
            tc::mbar_init(bars + 8u * j, 1);
    }
    __syncthreads();
    auto bar_h = [&](int l, int mt) { return bars + 8u * (uint32_t)((l - 1) * 2 + mt); };
    auto bar_e = [&](int mt) { return bars + 8u * (uint32_t)(2 * nh + mt); };
    auto signal = [&](uint32_t bar) { // after every lane's shared accesses before it
        __syncwarp();
        if (lane == 0)
            tc::mbar_arrive(bar);
    };
    const size_t row_bytes = (size_t)L * kColBytes, ring_bytes = 3 * row_bytes; // of 16 samples and one layer
    const size_t lstride = (size_t)gridDim.x * 2 * ring_bytes;

    if (warp < 2 * kPipeHidden) { // ------------------------------------------------------------ helpers
        regs_grow<kHelperRegs>();
        const int l = 1 + (warp >> 1), mt = warp & 1;
        if (l > nh)
            return;
        unsigned char *ring = reinterpret_cast<unsigned char *>(hist) + (l - 1) * lstride +
                              ((size_t)blockIdx.x * 2 + mt) * ring_bytes + lane * 16;
        unsigned char *fifo = smem + o.fifo + warp * kPipeTiles * kColBytes;
        const uint4 *w = reinterpret_cast<const uint4 *>(smem + o.w) + (l - 1) * kTapsB * 128;
        float4 *slotP = reinterpret_cast<float4 *>(smem + o.p + warp * (kHalf * kCh * 4)) + lane;
        const uint4 *slotH = reinterpret_cast<const uint4 *>(smem + o.h + warp * kColBytes) + lane;
        const uint32_t H = bar_h(l, mt);
        // The columns of a block: rows y - 2 and y - 1, each x0 - 2 .. x0 + 5, column c of a row in
        // slot c, the last in slot 0.  Taps dx = -2 .. 0 use columns 0..5 and are the last to use 0..2;
        // taps dx = 1, 2 use 3..7.  What is free then is filled with the row's column 7 and the next row's.
        int fy = 0, fx = 0, fr = 0, fm = 1; // the row whose columns are fetched: block, which row, (fy + 1) % 3
        const unsigned char *rsrc = ring, *psrc = ring;
        int rx = -2, px = 0; // its first column's x (a row outside the lattice: far outside), and the row's before
        auto fetch = [&](const unsigned char *src, int x, int c, int s) {
            const bool in = (unsigned)(x + c) < (unsigned)L;
            const unsigned char *from = in ? src + c * kColBytes : ring;
            cp16(fifo + s * kColBytes + lane * 16, from, in ? 16 : 0);
            cp16(fifo + s * kColBytes + lane * 16 + 512, from + 512, in ? 16 : 0);
        };
        auto place = [&] { // where the row's columns are
            const int m = fm + fr >= 3 ? fm + fr - 3 : fm + fr;
            rx = fy < L && fy - 2 + fr >= 0 ? fx - 2 : -(1 << 20);
            rsrc = ring + m * row_bytes + (ptrdiff_t)(fx - 2) * kColBytes;
        };
        auto next_row = [&] {
            psrc = rsrc;
            px = rx;
            fr ^= 1;
            if (fr == 0) {
                fx += 4;
                if (fx >= L) {
                    fx = 0;
                    ++fy;
                    fm = fm == 2 ? 0 : fm + 1;
                }
            }
            place();
        };
        auto column = [&](uint4(&a)[2], int c) {
            const uint4 *p = reinterpret_cast<const uint4 *>(fifo + (c == 7 ? 0 : c) * kColBytes) + lane;
            a[0] = p[0];
            a[1] = p[32];
        };
        float cur[4][4][4], nxt[4][4][4]; // the accumulators of a block's positions; of the next block's
        auto taps = [&](uint4(&a)[4][2], int r, int d) { // a: columns d .. d + 3, column c in a[c & 3]
            const uint4 *wt = w + (5 * r + d) * 128 + lane;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {
                const uint4 w0 = wt[ks * 64], w1 = wt[ks * 64 + 32];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    mma_step(nxt[q], a[(d + q) & 3][ks], w0, w1);
            }
        };
        auto first_taps = [&](int r) {
            uint4 a[4][2];
            cp_wait<0>();
            column(a[0], 0);
            column(a[1], 1);
            column(a[2], 2);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                column(a[(d + 3) & 3], d + 3);
                taps(a, r, d);
            }
            next_row();
            fetch(psrc, px, 7, 0);
            fetch(rsrc, rx, 1, 1);
            fetch(rsrc, rx, 2, 2);
            cp_commit();
        };
        auto last_taps = [&](int r) {
            uint4 a[4][2];
            cp_wait<0>();
            column(a[3], 3);
            column(a[0], 4);
            column(a[1], 5);
#pragma unroll
            for (int d = 3; d < 5; ++d) {
                column(a[(d + 3) & 3], d + 3);
                taps(a, r, d);
            }
            fetch(rsrc, rx, 0, 0);
#pragma unroll
            for (int c = 3; c < 7; ++c)
                fetch(rsrc, rx, c, c);
            cp_commit();
        };
        uint4 a11[2] = {}; // the layer's input at the position before, in this row
        int k = 0, stored = 0;
        unsigned char *dst = ring; // of position k - 1 in the ring (position modulo 3 L)
        // position k, at x: taps 10, 11, hand over
        auto finish = [&](float(&c)[4][4], int x) {
            if ((unsigned)x >= (unsigned)L)
                return;
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            const uint4 *wt = w + 10 * 128 + lane;
            if (x == 0)
                a11[0] = a11[1] = zero;
            mma_step(c, a11[0], wt[0], wt[32]);
            mma_step(c, a11[1], wt[64], wt[96]);
            if (k > 0) {
                ok = wait_warp(H, (uint32_t)(k - 1) & 1u, abort, err);
                a11[0] = slotH[0];
                a11[1] = slotH[32];
                *reinterpret_cast<uint4 *>(dst) = a11[0];
                *reinterpret_cast<uint4 *>(dst + 512) = a11[1];
                dst += kColBytes;
                if (++stored == 3 * L) {
                    stored = 0;
                    dst = ring;
                }
                if (x == 0)
                    a11[0] = a11[1] = zero;
            }
            wt += 128;
            mma_step(c, a11[0], wt[0], wt[32]);
            mma_step(c, a11[1], wt[64], wt[96]);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                slotP[q * 32] = make_float4(c[q][0], c[q][1], c[q][2], c[q][3]);
            ready(kReadyHidden + warp, 64);
            ++k;
        };
        place();
#pragma unroll
        for (int c = 0; c < 7; ++c)
            fetch(rsrc, rx, c, c);
        cp_commit();
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    nxt[q][j][e] = 0.f;
        // Two positions of a block at a time, between them the taps of one row above the next block; the block
        // before the first has no positions.  (The loop's body stays one row long: the roles' loops have to share
        // the instruction cache.  With all four positions written out, 56 lines a step missed it.)
        int x0 = -4, r = 0;
#pragma unroll 1
        for (int y = 0; y < L && ok;) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (r == 0) {
                            cur[q][j][e] = nxt[q][j][e];
                            nxt[q][j][e] = 0.f;
                        } else if (q < 2) {
                            cur[q][j][e] = cur[q + 2][j][e];
                        }
                    }
            finish(cur[0], x0 + 2 * r);
            first_taps(r);
            finish(cur[1], x0 + 2 * r + 1);
            last_taps(r);
            r ^= 1;
            if (r == 0) {
                x0 += 4;
                if (x0 >= L) {
                    x0 = 0;
                    ++y;
                }
            }
        }
        cp_wait<0>();
        if (!ok)
            release_chain(kReadyHidden + warp, 64, chain_done + mt);
        return;
    }
    if (warp >= 2 * kPipeHidden + 4) { // -------------------------------------------------- output layer
        regs_shrink<kOutRegs>();
        // Two warps per half, 8 samples each: a lane has 4 channels (one of the sum's 8 parts) of two samples, so that
        // a tap is one 16-byte read of weights and one of activations (with 8 channels of one sample, three;
        // the shared-memory pipe is 88% busy).
        const int mt = warp & 1, sub = (warp >> 1) & 1, part = lane & 7, ls = 8 * sub + (lane >> 3); // samples ls, ls + 4
        const int s = mt * kHalf + ls + 4 * (part & 1), mine = part < 2; // the sample whose log q this lane keeps
        unsigned char *ring = reinterpret_cast<unsigned char *>(hist) + nh * lstride +
                              ((size_t)blockIdx.x * 2 + mt) * ring_bytes + sub * 512 + lane * 16;
        unsigned char *win = smem + o.win + mt * kPipeSide * 2 * kColBytes + sub * 512 + lane * 16;
        const bf16 *Hn = reinterpret_cast<const bf16 *>(smem + o.hn + mt * kColBytes);
        const uint2 *Ha = reinterpret_cast<const uint2 *>(Hn + ring_elem(ls, part * 4)),
                    *Hb = reinterpret_cast<const uint2 *>(Hn + ring_elem(ls + 4, part * 4));
        const float2 *draw = reinterpret_cast<const float2 *>(smem + o.draw) + s;
        // part p of the sum goes to the chain's lane 4 (s % 8) + p % 4: float (s / 8) 2 + p / 4 of its four
        float *Po = reinterpret_cast<float *>(smem + o.po) + mt * 128 + (lane >> 3) * 16 + (part & 3) * 4 + 2 * sub + (part >> 2);
        const float4 *wdl = reinterpret_cast<const float4 *>(WD) + part;
        double lq = 0.0;
        float po[2]; // of the two samples
        auto tap = [&](const uint4 &h, int t) {
            const float4 w = wdl[t * 8];
            const uint32_t lo[2] = {h.x, h.z}, hi[2] = {h.y, h.w};
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                po[p] = __fmaf_rn(w.x, bf16_lo(lo[p]), po[p]);
                po[p] = __fmaf_rn(w.y, bf16_hi(lo[p]), po[p]);
                po[p] = __fmaf_rn(w.z, bf16_lo(hi[p]), po[p]);
                po[p] = __fmaf_rn(w.w, bf16_hi(hi[p]), po[p]);
            }
        };
        int slot = 0; // of column x - 2 of the position `rows_above` works on
        auto rows_above = [&](int y, int x) { // taps 0..9 at (y, x)
            po[0] = po[1] = 0.f;
            const unsigned char *col[5];
#pragma unroll
            for (int d = 0; d < 5; ++d)
                col[d] = win + (slot + d >= kPipeSide ? slot + d - kPipeSide : slot + d) * 2 * kColBytes;
            slot = slot + 1 == kPipeSide ? 0 : slot + 1;
            if (y >= 2 && x >= 2 && x + 2 < L) {
#pragma unroll 1
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int d = 0; d < 5; ++d)
                        tap(*reinterpret_cast<const uint4 *>(col[d] + r * kColBytes), 5 * r + d);
                return;
            }
            int s = slot == 0 ? kPipeSide - 1 : slot - 1; // slot of column x - 2
#pragma unroll 1
            for (int t = 0, d = 0; t < 10; ++t) {
                const int r = t >= 5;
                if (y - 2 + r >= 0 && x - 2 + d >= 0 && x - 2 + d < L)
                    tap(*reinterpret_cast<const uint4 *>(win + (s * 2 + r) * kColBytes), t);
                s = s + 1 == kPipeSide ? 0 : s + 1;
                if (++d == 5) {
                    d = 0;
                    s = s + 1 == kPipeSide ? 0 : s + 1; // five on in a ring of six: back to column x - 2
                }
            }
        };
        int cy = 0, cx = 3, cslot = 5, at = 3; // next column to fetch, its slot, its position modulo 3 L
        auto fetch = [&] {                     // the next column, rows y - 2 and y - 1 there
            if (cy < L) {
#pragma unroll
                for (int r = 0; r < 2; ++r)
                    if (cy - 2 + r >= 0) {
                        int from = at + (1 + r) * L;
                        from = from >= 3 * L ? from - 3 * L : from;
                        cp16(win + (cslot * 2 + r) * kColBytes, ring + (size_t)from * kColBytes);
                    }
            }
            cp_commit();
            cslot = cslot + 1 == kPipeSide ? 0 : cslot + 1;
            at = at + 1 == 3 * L ? 0 : at + 1;
            if (++cx == L) {
                cx = 0;
                ++cy;
            }
        };
        // after step k - 1: taps 10, 11 at k, which the chain waits for (R1), then the upper rows' taps at k + 1
        uint4 h10 = make_uint4(0u, 0u, 0u, 0u), h11 = h10;
        unsigned char *dst = ring; // of position k - 1
        int stored = 0;
        rows_above(0, 0);
        fetch(); // position 3
        int y = 0, x = 0;
#pragma unroll 1
        for (int k = 0; k < P && ok; ++k) {
            float lt = 0.f;
            if (k > 0) {
                ok = wait_warp(bar_e(mt), (uint32_t)(k - 1) & 1u, abort, err);
                h10 = h11;
                const uint2 ha = *Ha, hb = *Hb;
                h11 = make_uint4(ha.x, ha.y, hb.x, hb.y);
                lt = draw->y;
            }
            if (x >= 2)
                tap(h10, 10);
            if (x >= 1)
                tap(h11, 11);
            Po[0] = po[0];
            Po[64] = po[1];
            ready(kReadyOut + mt, 96);
            if (k > 0) {
                *reinterpret_cast<uint4 *>(dst) = h11;
                dst += kColBytes;
                if (++stored == 3 * L) {
                    stored = 0;
                    dst = ring;
                }
            }
            cp_wait<0>(); // columns up to position k + 3
            fetch();      // and k + 4
            if (++x == L) {
                x = 0;
                ++y;
            }
            rows_above(y, x);
            if (k > 0 && mine)
                lq += (double)log_sigmoid(lt);
        }
        if (ok)
            wait_warp(bar_e(mt), (uint32_t)(P - 1) & 1u, abort, err);
        if (mine && s0 + s < n)
            logq[s0 + s] = lq + (double)log_sigmoid(draw->y);
        cp_wait<0>();
        if (!ok)
            release_chain(kReadyOut + mt, 96, chain_done + mt);
        return;
    }
    regs_shrink<kChainRegs>();

    if (warp >= 2 * kPipeHidden + 2) { // --------------------------------------------- first layer, uniforms
        const int mt = warp & 1, g = lane >> 2, qt = lane & 3; // samples g, g + 8; the fragment's columns
        const int sb = mt * kHalf + g + 8 * (qt & 1), mine = qt < 2; // the sample whose spins and uniforms this lane keeps
        const int gs = s0 + sb, live = mine && gs < n;
        const uint32_t *bits = reinterpret_cast<const uint32_t *>(smem + o.bits) + mt * kHalf * 3 * words;
        uint32_t *my_bits = reinterpret_cast<uint32_t *>(smem + o.bits) + sb * 3 * words;
        const float2 *draw = reinterpret_cast<const float2 *>(smem + o.draw) + sb;
        float *u = reinterpret_cast<float *>(smem + o.u) + sb;
        const float4 *w1l = reinterpret_cast<const float4 *>(W1) + 2 * qt;
        int8_t *out_g = out + (size_t)gs * P;
        const uint32_t my_id = live ? (ids ? ids[gs] : (uint32_t)gs) : 0u;
        uint4 rnd = make_uint4(0u, 0u, 0u, 0u);
        float a[2][8];
        auto spins_of = [&](int h, int row, int x) { // bit d: the spin of sample g + 8 h at (row, x - 2 + d)
            const uint32_t *b = bits + ((g + 8 * h) * 3 + row % 3) * words + (x >> 5);
            return __funnelshift_r(b[0], b[1], x & 31);
        };
        auto tap = [&](int t, uint32_t m0, uint32_t m1) { // bit 0 of m: the tap's spin
            const float4 wa = w1l[t * 8], wb = w1l[t * 8 + 1];
            const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
            const float v[2] = {m0 & 1u ? 1.f : -1.f, m1 & 1u ? 1.f : -1.f};
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    a[h][e] = __fmaf_rn(w[e], v[h], a[h][e]);
        };
        auto rows_above = [&](int y, int x) { // bias and taps 0..9 at (y, x)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float2 b = *reinterpret_cast<const float2 *>(Bs + 8 * j + 2 * qt);
                a[0][2 * j] = a[1][2 * j] = b.x;
                a[0][2 * j + 1] = a[1][2 * j + 1] = b.y;
            }
            if (y >= 2 && x >= 2 && x + 2 < L) {
#pragma unroll 1
                for (int r = 0; r < 2; ++r) {
                    const uint32_t m0 = spins_of(0, y + 1 + r, x), m1 = spins_of(1, y + 1 + r, x);
#pragma unroll
                    for (int d = 0; d < 5; ++d)
                        tap(5 * r + d, m0 >> d, m1 >> d);
                }
                return;
            }
#pragma unroll 1
            for (int t = 0; t < 10; ++t) {
                const int r = t / 5, d = t - 5 * r;
                if (y - 2 + r >= 0 && x - 2 + d >= 0 && x - 2 + d < L)
                    tap(t, spins_of(0, y + 1 + r, x) >> d, spins_of(1, y + 1 + r, x) >> d);
            }
        };
        auto uniforms = [&](int k) {
            if ((k & 3) == 0 && mine)
                rnd = philox4x32_10(make_uint4((uint32_t)k >> 2, round, kTagVanSample, my_id), key);
        };
        auto done = [&](int k, int y, int x) { // tap 10 at k = (y, x) (tap 11 is the last spin, left to the chain)
            if (x >= 2)
                tap(10, spins_of(0, y, x), spins_of(1, y, x));
            float4 *dst = reinterpret_cast<float4 *>(smem + o.p0 + ((k & 1) * 2 + mt) * (kHalf * kCh * 4)) + lane;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    dst[(2 * h + q) * 32] = make_float4(a[h][4 * q], a[h][4 * q + 1], a[h][4 * q + 2], a[h][4 * q + 3]);
            const uint32_t rk = (k & 2) ? ((k & 1) ? rnd.w : rnd.z) : ((k & 1) ? rnd.y : rnd.x);
            if (mine)
                u[(k & 1) * 2 * kHalf] = uniform_open0(rk);
            ready(kReadyFirst + mt, 64);
        };
        // after step k - 1: tap 10 at k + 1, which the chain waits for (R0), then the upper rows' taps at k + 2
        uniforms(0);
        rows_above(0, 0);
        done(0, 0, 0);
        rows_above(0, 1);
        int y = 0, x = 1, py = 0, px = 0; // positions k + 1, k - 1
#pragma unroll 1
        for (int k = 0; k + 1 < P && ok; ++k) {
            if (k > 0) {
                ok = wait_warp(bar_e(mt), (uint32_t)(k - 1) & 1u, abort, err);
                __syncwarp();
                if (mine) {
                    const float sp = draw->x;
                    uint32_t *b = my_bits + (py % 3) * words + ((px + 2) >> 5);
                    const uint32_t bit = 1u << ((px + 2) & 31);
                    *b = sp > 0.f ? *b | bit : *b & ~bit;
                    if (live)
                        out_g[k - 1] = (int8_t)sp;
                }
                if (++px == L) {
                    px = 0;
                    ++py;
                }
                __syncwarp();
            } else { // once the chain has taken the sum of step 0
                ok = wait_warp(bar_h(1, mt), 0u, abort, err);
            }
            done(k + 1, y, x);
            if (++x == L) {
                x = 0;
                ++y;
            }
            rows_above(y, x);
            uniforms(k + 2);
        }
        for (int k = P - 2; k < P && ok; ++k) { // the last two draws
            ok = wait_warp(bar_e(mt), (uint32_t)k & 1u, abort, err);
            if (live)
                out_g[k] = (int8_t)draw->x;
            if (k == P - 2)
                ready(kReadyFirst + mt, 64); // the chain may write its last draw
        }
        if (!ok)
            release_chain(kReadyFirst + mt, 64, chain_done + mt);
        return;
    }

    // ------------------------------------------------------------------------------------------- chain
    // Lane 4 g + t of a fragment holds rows (samples) g and g + 8.  After the output layer's first exchange even
    // lanes have row g, odd lanes row g + 8; lanes t = 0 and 1 publish the draw.
    const int mt = warp & 1, g = lane >> 2, t = lane & 3, odd = t & 1;
    const int sd = mt * kHalf + g + odd * 8;
    float2 *draw = reinterpret_cast<float2 *>(smem + o.draw) + sd;
    const float *u = reinterpret_cast<const float *>(smem + o.u) + sd;
    const float4 *Po = reinterpret_cast<const float4 *>(smem + o.po) + mt * 32 + lane;
    bf16 *Hn = reinterpret_cast<bf16 *>(smem + o.hn + mt * kColBytes);
    const uint4 *w12 = reinterpret_cast<const uint4 *>(smem + o.w) + 12 * 128 + lane;
    const float4 *Pf = reinterpret_cast<const float4 *>(smem + o.p + mt * (kHalf * kCh * 4)) + lane;
    uint4 *slotH = reinterpret_cast<uint4 *>(smem + o.h + mt * kColBytes) + lane;
    float v[2] = {0.f, 0.f}; // the last spin of rows g, g + 8
    uint32_t pk[4][2] = {};  // a layer's values, packed: [n-tile][row]
    auto load = [&](float(&c)[4][4], int l) { // accumulators of hidden layer l over taps 0..11
        group_sync(kReadyHidden + (l - 1) * 2 + mt, 64);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 x = Pf[(l - 1) * 256 + q * 32];
            c[q][0] = x.x, c[q][1] = x.y, c[q][2] = x.z, c[q][3] = x.w;
        }
    };
    // Hidden layer l of the values pk; the next layer's accumulators are fetched meanwhile.
    auto layer = [&](float(&c)[4][4], float(&cn)[4][4], int l) {
        const uint4 a0 = make_uint4(pk[0][0], pk[0][1], pk[1][0], pk[1][1]), a1 = make_uint4(pk[2][0], pk[2][1], pk[3][0], pk[3][1]);
        const uint4 *w = w12 + (l - 1) * kTapsB * 128;
        mma_step(c, a0, w[0], w[32]);
        mma_step(c, a1, w[64], w[96]);
        float2 b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            b[j] = *reinterpret_cast<const float2 *>(Bs + l * kCh + 2 * t + 8 * j);
        slotH[(l - 1) * 128] = a0;
        slotH[(l - 1) * 128 + 32] = a1;
        signal(bar_h(l, mt));
        if (l < nh)
            load(cn, l + 1);
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 s = add2(make_float2(c[j][2 * h], c[j][2 * h + 1]), b[j]);
                pk[j][h] = relu_pack(s.x, s.y);
            }
    };
    float ca[4][4], cb[4][4], f0[2][8], uk = 0.f;
    // What the first layer at k needs besides the last spin: its sum, and the uniform of the draw
    auto first = [&](int k) {
        const float4 *src = reinterpret_cast<const float4 *>(smem + o.p0 + ((k & 1) * 2 + mt) * (kHalf * kCh * 4)) + lane;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 s4 = src[(2 * h + q) * 32];
                f0[h][4 * q] = s4.x, f0[h][4 * q + 1] = s4.y, f0[h][4 * q + 2] = s4.z, f0[h][4 * q + 3] = s4.w;
            }
        uk = u[(k & 1) * 2 * kHalf];
    };
    int x = 0;
    group_sync(kReadyFirst + mt, 64);
    first(0);
    load(ca, 1);
#pragma unroll 1
    for (int k = 0; k < P; ++k) {
        // ---- first layer: sum + w s_{k-1}
        if (x > 0) {
            const float4 *w11 = reinterpret_cast<const float4 *>(W1 + 11 * kCh + 8 * t);
            const float4 wa = w11[0], wb = w11[1];
            const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    f0[h][e] = __fmaf_rn(w[e], v[h], f0[h][e]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int j = 0; j < 4; ++j)
                pk[j][h] = relu_pack(f0[h][2 * j], f0[h][2 * j + 1]);
        // ---- hidden layers
#pragma unroll 1
        for (int l = 1; l <= nh; l += 2) {
            layer(ca, cb, l);
            if (l < nh)
                layer(cb, ca, l + 1);
        }
        // The next step's sums, on the way while this one's output is computed.  With the first layer's sum at k + 1
        // there, the warps that keep the draw of step k - 1 have read it.
        group_sync(kReadyFirst + mt, 64);
        if (k + 1 < P)
            load(ca, 1);
        // ---- output layer: sum + tap 12, parts t and 4 + t of both rows; then the parts in pairs
        const float4 wd0 = *reinterpret_cast<const float4 *>(WD + 12 * kCh + 4 * t),
                     wd1 = *reinterpret_cast<const float4 *>(WD + 12 * kCh + 16 + 4 * t);
        const float bD = Bs[(D - 1) * kCh];
        group_sync(kReadyOut + mt, 96);
        const float4 p4 = *Po;
        float part[2][2] = {{p4.x, p4.y}, {p4.z, p4.w}}; // [row][part t, part 4 + t]
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint32_t lo = pk[2 * q][h], hi = pk[2 * q + 1][h];
                const float4 wd = q == 0 ? wd0 : wd1;
                *reinterpret_cast<uint2 *>(Hn + ring_elem(g + 8 * h, 16 * q + 4 * t)) = make_uint2(lo, hi);
                part[h][q] = __fmaf_rn(wd.x, bf16_lo(lo), part[h][q]);
                part[h][q] = __fmaf_rn(wd.y, bf16_hi(lo), part[h][q]);
                part[h][q] = __fmaf_rn(wd.z, bf16_lo(hi), part[h][q]);
                part[h][q] = __fmaf_rn(wd.w, bf16_hi(hi), part[h][q]);
            }
        float f2[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float other = __shfl_xor_sync(0xffffffffu, odd ? part[0][q] : part[1][q], 1);
            f2[q] = (odd ? part[1][q] : part[0][q]) + other; // parts 2 s + 2 s + 1
            f2[q] += __shfl_xor_sync(0xffffffffu, f2[q], 2);
        }
        float f = f2[0] + f2[1];
        f += bD;
        const int stop = *abort;
        // ---- draw
        const float sp = uk < sigmoid(f) ? 1.f : -1.f; // lanes t < 2
        first(k + 1);
        v[0] = __shfl_sync(0xffffffffu, sp, lane & ~3);
        v[1] = __shfl_sync(0xffffffffu, sp, (lane & ~3) | 1);
        if (t < 2)
            *draw = make_float2(sp, sp * f);
        signal(bar_e(mt));
        if (++x == L)
            x = 0;
        if (__any_sync(0xffffffffu, stop))
            break;
    }
    if (lane == 0)
        *(volatile int *)(chain_done + mt) = 1;
}

// Copy the int8 lattices of every chain of an int8-layout Ising context into
// one contiguous [n][L][L] buffer (or back, when `back`).
__global__ void k_gather(const IsingChain *chains, char *lattice, int8_t *buf, int L, int n, int back)
{
    const size_t per = (size_t)L * L;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < per * n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t k = i / per, j = i % per;
        int8_t *lat = reinterpret_cast<int8_t *>(lattice + chains[k].spin_off);
        if (back)
            lat[j] = buf[i];
        else
            buf[i] = lat[j];
    }
}

// H of Eq. (1) per configuration (exact).
__global__ void k_energy(const int8_t *s, long long *E, int L)
{
    __shared__ long long part[32];
    const size_t base = (size_t)blockIdx.x * L * L;
    long long acc = 0;
    for (int i = threadIdx.x; i < L * L; i += blockDim.x) {
        const int y = i / L, x = i % L;
        const int v = s[base + i];
        acc -= v * (s[base + y * L + (x + 1) % L] + s[base + ((y + 1) % L) * L + x]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0)
        part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
            t += part[w];
        E[blockIdx.x] = t;
    }
}

__device__ __forceinline__ double log_add_exp(double a, double b)
{
    const double m = fmax(a, b);
    return m + log1p(exp(-fabs(a - b)));
}

// Metropolis-Hastings for an independence proposal from q_sym(s) = (q(s) +
// q(-s)) / 2: accept s' with probability min(1, e^{-beta (E' - E)} q_sym(s) /
// q_sym(s')).  The proposal is the sample s'' or its global flip -s'' (one bit
// of the chain's MH Philox block), and q_sym, E are flip-invariant.  Accepted
// proposals are written into the chain's lattice.
__global__ void k_mh_accept(const IsingChain *chains, char *lattice, const int8_t *prop, const double *lq_p,
                            const double *lq_pn, const double *lq_s, const double *lq_sn, const long long *E_s,
                            const long long *E_p, int L, int n, PhiloxKey key, uint32_t round, int *accepted,
                            double *log_ratio)
{
    const int k = blockIdx.x;
    __shared__ int take, flip;
    if (threadIdx.x == 0) {
        const IsingChain &ch = chains[k];
        const uint4 r = philox4x32_10(make_uint4(0u, round, kTagVanMH, ch.chain_id), key);
        const double u = (double)((r.x >> 8) + 1u) * (1.0 / 16777216.0);
        flip = (int)(r.y >> 31);
        const double lr = -ch.beta * (double)(E_p[k] - E_s[k]) + log_add_exp(lq_s[k], lq_sn[k]) -
                          log_add_exp(lq_p[k], lq_pn[k]);
        take = log(u) < lr;
        if (log_ratio)
            log_ratio[k] = lr;
        if (take)
            atomicAdd(accepted, 1);
    }
    __syncthreads();
    if (!take)
        return;
    int8_t *lat = reinterpret_cast<int8_t *>(lattice + chains[k].spin_off);
    const int8_t *p = prop + (size_t)k * L * L;
    for (int i = threadIdx.x; i < L * L; i += blockDim.x)
        lat[i] = flip ? (int8_t)(-p[i]) : p[i];
}

size_t a256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace
}  // namespace van
}  // namespace mc

using namespace mc;
using namespace mc::van;

struct mc_van {
    int L = 0, D = 0, nmax = 0;
    PhiloxKey key{};
    uint32_t round = 0;
    int adam_t = 0;
    cudaStream_t stream = nullptr;
    char *ws = nullptr;
    ParamLayout P{};
    DevParams dp{};
    float *p = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
    bf16 *wh = nullptr;
    float *w1 = nullptr, *wD = nullptr, *bias = nullptr;
    bf16 *H = nullptr;
    float *dZa = nullptr, *dZb = nullptr;
    float *f = nullptr, *ll = nullptr, *dF = nullptr;
    uint32_t *bits = nullptr; // positive_bits of hidden layers 0 .. D - 3 of a training step
    int8_t *spins = nullptr, *prop = nullptr;
    double *lq = nullptr, *lq2 = nullptr, *lq3 = nullptr, *lq4 = nullptr, *mh_lr = nullptr;
    long long *E1 = nullptr, *E2 = nullptr;
    int *acc = nullptr;
    bf16 *hist = nullptr;
    const bf16 *zero = nullptr; // 5 kTapBytes of zeros
    float *dwpart = nullptr; // per-CTA partial gradients of k_dw32_tc
    int *err = nullptr;      // device fault latch (a bounded completion wait gave up)
    RunGeom conv[3];         // geometries of the convolutions (kFwd, kLast, kBwd)
    int sms = 0;
    bool pipe = false;       // the sampler with streamed columns (k_sample_pipe)
    bool weights_ready = false;
};

namespace {

mc_status vfail(mc_status s, const std::string &m)
{
    mc::set_last_error(m);
    return s;
}

// Synchronise the stream, then report (and clear) a fault a kernel latched --
// a bounded wait for a tensor-core or bulk-copy completion that gave up.
mc_status check_err(mc_van *w, const char *where)
{
    int v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, w->err, sizeof v, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
    if (v != 0) {
        cudaMemsetAsync(w->err, 0, sizeof v, w->stream);
        return vfail(MC_ETIMEOUT, std::string(where) + ": a tensor-core or bulk-copy completion wait timed out");
    }
    return MC_OK;
}

struct VanLayout {
    size_t p, m, v, g, wh, w1, wD, bias, H, dZa, dZb, f, ll, dF, bits, spins, prop, lq, lq2, lq3, lq4, lr, E1, E2, acc, zero,
        hist, dwpart, err, total;
};

VanLayout van_layout(int L, int nmax, int D)
{
    VanLayout o{};
    const ParamLayout P = param_layout(D);
    size_t off = 0;
    auto take = [&](size_t b) {
        const size_t r = off;
        off = a256(off + std::max<size_t>(b, 1));
        return r;
    };
    const size_t pos = (size_t)nmax * L * L;
    o.p = take(P.total * 4);
    o.m = take(P.total * 4);
    o.v = take(P.total * 4);
    o.g = take(P.total * 4);
    o.wh = take((size_t)(D - 2) * kTapsB * kCh * kCh * 2);
    o.dwpart = take((size_t)kMaxDwBlocks * kDwPart * 4);
    o.err = take(16);
    o.w1 = take((size_t)kCh * kTapsA * 4);
    o.wD = take((size_t)kTapsB * kCh * 4);
    o.bias = take((size_t)((D - 1) * kCh + 1) * 4);
    o.H = take((size_t)(D - 1) * pos * kCh * 2);
    o.dZa = take(pos * kCh * 4);
    o.dZb = take(pos * kCh * 4);
    o.f = take(pos * 4);
    o.ll = take(pos * 4);
    o.dF = take(pos * 4);
    o.bits = take((size_t)(D - 2) * pos * 4);
    o.spins = take(pos);
    o.prop = take(pos);
    o.lq = take((size_t)nmax * 8);
    o.lq2 = take((size_t)nmax * 8);
    o.lq3 = take((size_t)nmax * 8);
    o.lq4 = take((size_t)nmax * 8);
    o.lr = take((size_t)nmax * 8);
    o.E1 = take((size_t)nmax * 8);
    o.E2 = take((size_t)nmax * 8);
    o.acc = take(64);
    o.zero = take((size_t)5 * kTapBytes); // zeros: the sampler's taps outside the lattice
    o.hist = take((size_t)(D - 1) * ((nmax + kSampleTile - 1) / kSampleTile) * kSampleTile * 3 * L * kCh * 2);
    o.total = off;
    return o;
}

unsigned grid_for(size_t n, int threads, int sms) { return (unsigned)std::min<size_t>((n + threads - 1) / threads, (size_t)sms * 16); }

size_t sample_smem(int D, int L, int nbuf)
{
    const size_t nh = (size_t)D - 2, tt = (size_t)kSampleTile * kCh;
    return nh * kTapsB * tt * 2 + (size_t)(nbuf + 1) * kTileBytes + 2 * tt * 2 + tt * 4 + (size_t)kSampleTile * 8 * 4 +
           (size_t)(kCh * kTapsA + kTapsB * kCh + (D - 1) * kCh + 1 + kSampleTile) * 4 + (size_t)kSampleTile * 3 * L +
           8 * (2 * (kSampleMaxBufs + 1) + 4) + 8;
}

// Hidden-layer tiles the sampler keeps in flight (besides the output layer's
// one): as many as fit, at most 3 and at most the D - 2 hidden layers (the
// release of the tile nbuf gathers back must come after the ring stores that
// a gather reads).
int sample_bufs(int D, int L)
{
    for (int b = std::min(kSampleMaxBufs, D - 2); b > 1; --b)
        if (sample_smem(D, L, b) <= kSampleSmemLimit)
            return b;
    return 1;
}

// Dynamic shared memory a kernel may use: raised to what this network needs,
// never lowered, so that creating a smaller network leaves larger ones usable.
cudaError_t raise_smem_limit(const void *kernel, size_t bytes)
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess || (int)bytes <= a.maxDynamicSharedSizeBytes)
        return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int MODE>
cudaError_t raise_conv_limit(const RunGeom &g)
{
    return raise_smem_limit((const void *)conv_kernel<MODE>(g), g.smem_bytes);
}

// Which sampler: k_sample_pipe wherever its 8 helper warps and its shared memory do
// (up to 4 hidden layers) and a block's columns are known a block ahead (L >= 8);
// k_sample otherwise.  The register split of k_sample_pipe needs exactly the registers
// it was written for.
cudaError_t sampler_rule(mc_van *w)
{
    if (w->D - 2 > kPipeHidden || w->L < kPipeMinL)
        return cudaSuccess;
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, (const void *)k_sample_pipe);
    if (e != cudaSuccess || a.numRegs != kPipeRegs)
        return e;
    w->pipe = true;
    return raise_smem_limit((const void *)k_sample_pipe, pipe_smem(w->D, w->L).total);
}

cudaError_t prep(mc_van *w)
{
    k_prep_weights<<<64, 256, 0, w->stream>>>(w->p, w->dp, w->wh, w->w1, w->wD, w->bias);
    w->weights_ready = true;
    return cudaGetLastError();
}

// Forward over n configurations in w->spins (negated when `negate`); log q
// into `logq`; dF (training) when dF != nullptr.
cudaError_t forward(mc_van *w, int n, int negate, double *logq, float *dF)
{
    if (!w->weights_ready) {
        cudaError_t e = prep(w);
        if (e != cudaSuccess)
            return e;
    }
    const int L = w->L, D = w->D;
    const size_t layer = (size_t)w->nmax * L * L * kCh;
    const unsigned l1g =
        (unsigned)std::min<long long>(((long long)n * L * L + kL1Threads - 1) / kL1Threads, (long long)w->sms * 8);
    k_layer1_tc<<<l1g, kL1Threads, 0, w->stream>>>(w->spins, negate, w->w1, w->bias, w->H, dF ? w->bits : nullptr, n, L,
                                                   w->err);
    const RunGeom &gh = w->conv[kFwd], &gl = w->conv[kLast];
    for (int l = 1; l <= D - 1; ++l) { // hidden layers 1 .. D-2, then the last layer
        CUtensorMap in_map;
        const bool is_last = l == D - 1;
        const cudaError_t e = run_map(&in_map, w->H + (l - 1) * layer, n, is_last ? gl : gh);
        if (e != cudaSuccess)
            return e;
        ConvArgs a{};
        a.n = n;
        a.err = w->err;
        if (is_last) {
            a.la = LastLayerArgs{w->wD, w->bias + (D - 1) * kCh, w->spins, negate, w->f, w->ll, dF, 1.0f / n};
            launch_conv<kLast>(gl, in_map, in_map, a, w->sms, w->stream);
        } else {
            a.W = w->wh + (size_t)(l - 1) * kTapsB * kCh * kCh;
            a.bias = w->bias + l * kCh;
            a.out = w->H + l * layer;
            a.bits = dF && l < D - 2 ? w->bits + l * (layer / kCh) : nullptr;
            launch_conv<kFwd>(gh, in_map, in_map, a, w->sms, w->stream);
        }
    }
    launch_chained_on(w->stream, true, k_logq, (unsigned)n, 256u, 0, (const float *)w->ll, logq, L);
    return cudaGetLastError();
}

// Every kernel of the backward pass writes its own part of the gradient; the masked
// taps' zeros are set before the forward pass, which leaves the kernels chained.
cudaError_t backward(mc_van *w, int n)
{
    const int L = w->L, D = w->D;
    const cudaStream_t st = w->stream;
    const size_t layer = (size_t)w->nmax * L * L * kCh;
    const bf16 *hD = w->H + (D - 2) * layer;
    const unsigned eg = (unsigned)std::min<size_t>(((size_t)n * L + kEdgeThreads / 32 - 1) / (kEdgeThreads / 32),
                                                   std::min<size_t>((size_t)w->sms * kEdgeCtas,
                                                                    (size_t)kMaxDwBlocks * kDwPart / kEdgeOutD));
    // gradients as BF16 hi + lo pairs, each pair in the space of one FP32 buffer
    const size_t cap = (size_t)w->nmax * L * L * kCh;
    bf16 *dzh = reinterpret_cast<bf16 *>(w->dZa), *dzl = dzh + cap;
    bf16 *nxh = reinterpret_cast<bf16 *>(w->dZb), *nxl = nxh + cap;
    // edge-layer partial sums go to the dW partial buffer (free at these points)
    launch_chained_on(st, true, k_layerD_bwd, eg, (unsigned)kEdgeThreads,
                      (size_t)(kEdgeThreads / 32) * edge_bytes_d(L), (const float *)w->dF, (const float *)w->wD, hD,
                      dzh, dzl, w->dwpart, n, L);
    launch_chained_on(st, true, k_edge_grad_reduce<false>, (unsigned)kEdgeOutD, 256u, 0, (const float *)w->dwpart, (int)eg,
                      w->g, w->dp);
    const RunGeom &gb = w->conv[kBwd];
    // k_dw32_tc: two CTAs per SM (256 tensor-memory columns and at most 110 KB of stages each)
    const DwTcGeom dg = dw_tc_geom(L);
    const unsigned dwg = (unsigned)std::min<size_t>(std::min<size_t>((size_t)n * L, (size_t)w->sms * 2), kMaxDwBlocks);
    for (int l = D - 2; l >= 1; --l) { // hidden layer l: input H[l-1], output H[l], grad dz wrt its pre-activation
        CUtensorMap zh_map, zl_map, x_map, hi_map, lo_map;
        cudaError_t e = activation_map(&zh_map, dzh, n, L, dg.PZ, 1);
        if (e == cudaSuccess)
            e = activation_map(&zl_map, dzl, n, L, dg.PZ, 1);
        if (e == cudaSuccess)
            e = activation_map(&x_map, w->H + (l - 1) * layer, n, L, dg.PX, 3);
        if (e == cudaSuccess)
            e = run_map(&hi_map, dzh, n, gb);
        if (e == cudaSuccess)
            e = run_map(&lo_map, dzl, n, gb);
        if (e != cudaSuccess)
            return e;
        launch_chained_on(st, true, k_dw32_tc, dwg, 192u, dg.smem_bytes, zh_map, zl_map, x_map, w->dwpart, n, dg, w->err);
        launch_chained_on(st, true, k_dw_reduce, (unsigned)((kDwPart + 31) / 32), 256u, 0, (const float *)w->dwpart,
                          (int)dwg, w->g, w->dp, l);
        ConvArgs a{};
        a.W = w->wh + (size_t)(l - 1) * kTapsB * kCh * kCh;
        a.mask = w->bits + (l - 1) * (layer / kCh);
        a.out = nxh;
        a.out_lo = nxl;
        a.n = n;
        a.err = w->err;
        launch_conv<kBwd>(gb, hi_map, lo_map, a, w->sms, st);
        std::swap(dzh, nxh);
        std::swap(dzl, nxl);
    }
    launch_chained_on(st, true, k_layer1_bwd_w, eg, (unsigned)kEdgeThreads,
                      (size_t)(kEdgeThreads / 32) * edge_bytes_1(L), (const bf16 *)dzh, (const bf16 *)dzl,
                      (const int8_t *)w->spins, w->dwpart, n, L);
    launch_chained_on(st, true, k_edge_grad_reduce<true>, (unsigned)kEdgeOut1, 256u, 0, (const float *)w->dwpart, (int)eg,
                      w->g, w->dp);
    return cudaGetLastError();
}

}  // namespace

extern "C" {

size_t mc_van_param_count(int32_t depth)
{
    if (depth < 3 || depth > kMaxDepth)
        return 0;
    return param_layout(depth).total;
}

size_t mc_van_workspace_bytes(int32_t L, int32_t batch, int32_t depth)
{
    if (L < 2 || L > kMaxL || (L & 1) || batch < 1 || depth < 3 || depth > kMaxDepth) {
        mc::set_last_error("mc_van_workspace_bytes: need even L in [2, 128], batch >= 1, depth in [3, 7]");
        return 0;
    }
    return van_layout(L, batch, depth).total;
}

mc_status mc_van_create(mc_van **out, int32_t L, int32_t batch, int32_t depth, uint64_t seed, void *workspace,
                        size_t bytes, void *cuda_stream)
{
    if (!out)
        return vfail(MC_EINVAL, "out is NULL");
    *out = nullptr;
    const size_t need = mc_van_workspace_bytes(L, batch, depth);
    if (need == 0)
        return MC_EINVAL;
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u))
        return vfail(MC_EINVAL, "workspace must be a device pointer aligned to 256 bytes");
    if (bytes < need)
        return vfail(MC_ENOMEM, "van workspace too small: need " + std::to_string(need) + " bytes");
    mc_van *w = new (std::nothrow) mc_van();
    if (!w)
        return vfail(MC_ENOMEM, "host allocation failed");
    w->L = L;
    w->D = depth;
    w->nmax = batch;
    w->key = PhiloxKey{(uint32_t)seed, (uint32_t)(seed >> 32)};
    w->stream = static_cast<cudaStream_t>(cuda_stream);
    w->ws = static_cast<char *>(workspace);
    w->P = param_layout(depth);
    w->dp.D = depth;
    for (int l = 0; l < depth; ++l) {
        w->dp.w_off[l] = w->P.w_off[l];
        w->dp.b_off[l] = w->P.b_off[l];
    }
    const VanLayout o = van_layout(L, batch, depth);
    char *b = w->ws;
    w->p = reinterpret_cast<float *>(b + o.p);
    w->m = reinterpret_cast<float *>(b + o.m);
    w->v = reinterpret_cast<float *>(b + o.v);
    w->g = reinterpret_cast<float *>(b + o.g);
    w->wh = reinterpret_cast<bf16 *>(b + o.wh);
    w->dwpart = reinterpret_cast<float *>(b + o.dwpart);
    w->err = reinterpret_cast<int *>(b + o.err);
    w->w1 = reinterpret_cast<float *>(b + o.w1);
    w->wD = reinterpret_cast<float *>(b + o.wD);
    w->bias = reinterpret_cast<float *>(b + o.bias);
    w->H = reinterpret_cast<bf16 *>(b + o.H);
    w->dZa = reinterpret_cast<float *>(b + o.dZa);
    w->dZb = reinterpret_cast<float *>(b + o.dZb);
    w->f = reinterpret_cast<float *>(b + o.f);
    w->ll = reinterpret_cast<float *>(b + o.ll);
    w->dF = reinterpret_cast<float *>(b + o.dF);
    w->bits = reinterpret_cast<uint32_t *>(b + o.bits);
    w->spins = reinterpret_cast<int8_t *>(b + o.spins);
    w->prop = reinterpret_cast<int8_t *>(b + o.prop);
    w->lq = reinterpret_cast<double *>(b + o.lq);
    w->lq2 = reinterpret_cast<double *>(b + o.lq2);
    w->lq3 = reinterpret_cast<double *>(b + o.lq3);
    w->lq4 = reinterpret_cast<double *>(b + o.lq4);
    w->mh_lr = reinterpret_cast<double *>(b + o.lr);
    w->E1 = reinterpret_cast<long long *>(b + o.E1);
    w->E2 = reinterpret_cast<long long *>(b + o.E2);
    w->acc = reinterpret_cast<int *>(b + o.acc);
    w->hist = reinterpret_cast<bf16 *>(b + o.hist);
    w->zero = reinterpret_cast<const bf16 *>(b + o.zero);
    for (int mode = 0; mode < 3; ++mode)
        w->conv[mode] = run_geom(L, mode);
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&w->sms, cudaDevAttrMultiProcessorCount, dev);
    cudaError_t e = cudaMemsetAsync(w->ws, 0, o.hist, w->stream); // params, Adam state, buffers
    if (e == cudaSuccess)
        e = raise_conv_limit<kFwd>(w->conv[kFwd]);
    if (e == cudaSuccess)
        e = raise_conv_limit<kLast>(w->conv[kLast]);
    if (e == cudaSuccess)
        e = raise_conv_limit<kBwd>(w->conv[kBwd]);
    if (e == cudaSuccess)
        e = raise_smem_limit((const void *)k_dw32_tc, dw_tc_geom(L).smem_bytes);
    if (e == cudaSuccess)
        e = raise_smem_limit((const void *)k_layerD_bwd, (size_t)(kEdgeThreads / 32) * edge_bytes_d(L));
    if (e == cudaSuccess)
        e = raise_smem_limit((const void *)k_layer1_bwd_w, (size_t)(kEdgeThreads / 32) * edge_bytes_1(L));
    if (e == cudaSuccess)
        e = raise_smem_limit((const void *)k_sample, sample_smem(depth, L, sample_bufs(depth, L)));
    if (e == cudaSuccess)
        e = sampler_rule(w);
    if (e != cudaSuccess) {
        delete w;
        return vfail(MC_ECUDA, std::string("mc_van_create: ") + cudaGetErrorString(e));
    }
    *out = w;
    return MC_OK;
}

mc_status mc_van_set_params(mc_van *w, const float *host_params, size_t n)
{
    if (!w || !host_params || n != w->P.total)
        return vfail(MC_EINVAL, "mc_van_set_params: need mc_van_param_count(depth) floats");
    cudaError_t e = cudaMemcpyAsync(w->p, host_params, n * 4, cudaMemcpyHostToDevice, w->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(w->m, 0, n * 4, w->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(w->v, 0, n * 4, w->stream);
    if (e == cudaSuccess)
        e = prep(w);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(w->stream);
    w->adam_t = 0;
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_set_params: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_get_params(mc_van *w, float *host_params, size_t n, float *host_grads)
{
    if (!w || !host_params || n != w->P.total)
        return vfail(MC_EINVAL, "mc_van_get_params: need mc_van_param_count(depth) floats");
    cudaError_t e = cudaMemcpyAsync(host_params, w->p, n * 4, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess && host_grads)
        e = cudaMemcpyAsync(host_grads, w->g, n * 4, cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_get_params: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_get_activations(mc_van *w, int32_t layer, int32_t n, uint16_t *host_dst)
{
    if (!w || !host_dst || layer < 0 || layer > w->D - 2 || n < 1 || n > w->nmax)
        return vfail(MC_EINVAL, "mc_van_get_activations: bad argument (0 <= layer <= depth - 2, 1 <= n <= batch)");
    const size_t layer_elems = (size_t)w->nmax * w->L * w->L * kCh;
    cudaError_t e = cudaMemcpyAsync(host_dst, w->H + (size_t)layer * layer_elems, (size_t)n * w->L * w->L * kCh * 2,
                                    cudaMemcpyDeviceToHost, w->stream);
    if (e == cudaSuccess)
        e = cudaStreamSynchronize(w->stream);
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_get_activations: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_log_prob(mc_van *w, const int8_t *dev_spins, int32_t n, int32_t negate, double *dev_logq)
{
    if (!w || !dev_spins || !dev_logq || n < 1 || n > w->nmax)
        return vfail(MC_EINVAL, "mc_van_log_prob: bad argument (1 <= n <= batch)");
    cudaError_t e = cudaMemcpyAsync(w->spins, dev_spins, (size_t)n * w->L * w->L, cudaMemcpyDeviceToDevice, w->stream);
    if (e == cudaSuccess)
        e = forward(w, n, negate, dev_logq, nullptr);
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_log_prob: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_train_step(mc_van *w, const int8_t *dev_spins, int32_t n, float lr, int32_t apply, double *host_loss)
{
    if (!w || !dev_spins || n < 1 || n > w->nmax)
        return vfail(MC_EINVAL, "mc_van_train_step: bad argument (1 <= n <= batch)");
    cudaError_t e = cudaMemcpyAsync(w->spins, dev_spins, (size_t)n * w->L * w->L, cudaMemcpyDeviceToDevice, w->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(w->g, 0, w->P.total * 4, w->stream);
    if (e == cudaSuccess)
        e = forward(w, n, 0, w->lq, w->dF);
    if (e == cudaSuccess)
        e = backward(w, n);
    if (e == cudaSuccess && apply) {
        ++w->adam_t;
        const float b1 = 0.9f, b2 = 0.999f;
        e = launch_chained_on(w->stream, true, k_adam, grid_for(w->P.total, 256, w->sms), 256u, 0, w->p, w->m, w->v,
                              (const float *)w->g, w->P.total, lr, b1, b2, 1e-8f, 1.f - powf(b1, (float)w->adam_t),
                              1.f - powf(b2, (float)w->adam_t));
        if (e == cudaSuccess)
            e = prep(w);
    }
    if (e == cudaSuccess && host_loss) {
        std::vector<double> lq(n);
        e = cudaMemcpyAsync(lq.data(), w->lq, (size_t)n * 8, cudaMemcpyDeviceToHost, w->stream);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(w->stream);
        double s = 0.0;
        for (double v : lq)
            s += v;
        *host_loss = -s / n;
    }
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_train_step: ") + cudaGetErrorString(e));
    return host_loss ? check_err(w, "mc_van_train_step") : MC_OK;
}

mc_status mc_van_sample(mc_van *w, int32_t n, uint32_t round, const uint32_t *dev_ids, int8_t *dev_out,
                        double *dev_logq)
{
    if (!w || n < 1 || n > w->nmax)
        return vfail(MC_EINVAL, "mc_van_sample: 1 <= n <= batch");
    if (!w->weights_ready) {
        cudaError_t e = prep(w);
        if (e != cudaSuccess)
            return vfail(MC_ECUDA, cudaGetErrorString(e));
    }
    int8_t *out = dev_out ? dev_out : w->prop;
    double *lq = dev_logq ? dev_logq : w->lq;
    cudaError_t e = cudaMemsetAsync(out, 0, (size_t)n * w->L * w->L, w->stream);
    if (e == cudaSuccess) {
        const unsigned blocks = (unsigned)((n + kSampleTile - 1) / kSampleTile);
        const int nbuf = sample_bufs(w->D, w->L);
        if (w->pipe)
            k_sample_pipe<<<blocks, kPipeThreads, pipe_smem(w->D, w->L).total, w->stream>>>(
                w->wh, w->w1, w->wD, w->bias, w->D, w->L, n, w->hist, out, lq, w->key, round, dev_ids, w->err);
        else
            k_sample<<<blocks, kSampleThreads, sample_smem(w->D, w->L, nbuf), w->stream>>>(
                w->wh, w->w1, w->wD, w->bias, w->D, w->L, n, nbuf, w->hist, w->zero, out, lq, w->key, round, dev_ids, w->err);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_sample: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_sync(mc_van *w)
{
    if (!w)
        return vfail(MC_EINVAL, "mc_van_sync: NULL network");
    return check_err(w, "mc_van_sync");
}

mc_status mc_ising_gather(mc_ctx *c, int8_t *dev_out, int32_t back)
{
    if (!c || !dev_out || c->kind != MC_KIND_ISING || c->layout != MC_LAYOUT_INT8)
        return vfail(MC_EINVAL, "mc_ising_gather: needs an int8-layout Ising context");
    const int L = (int)c->ising[0].Lx;
    for (const auto &ch : c->ising)
        if ((int)ch.Lx != L || (int)ch.Ly != L)
            return vfail(MC_EINVAL, "mc_ising_gather: every chain must be L x L with the same L");
    const size_t total = (size_t)c->n_chains * L * L;
    k_gather<<<(unsigned)std::min<size_t>((total + 255) / 256, 4096), 256, 0, c->stream>>>(
        static_cast<const IsingChain *>(c->d_chains), c->d_lattice, dev_out, L, c->n_chains, back);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_ising_gather: ") + cudaGetErrorString(e));
    return MC_OK;
}

mc_status mc_van_mh_round(mc_van *w, mc_ctx *c, int32_t *host_accepted)
{
    if (!w || !c || c->kind != MC_KIND_ISING || c->layout != MC_LAYOUT_INT8)
        return vfail(MC_EINVAL, "mc_van_mh_round: needs an int8-layout Ising context");
    const int n = c->n_chains, L = w->L;
    if (n > w->nmax)
        return vfail(MC_EINVAL, "mc_van_mh_round: more chains than the network's batch");
    for (const auto &ch : c->ising)
        if ((int)ch.Lx != L || (int)ch.Ly != L)
            return vfail(MC_EINVAL, "mc_van_mh_round: every chain must be L x L with the network's L");
    if (c->stream != w->stream)
        return vfail(MC_EINVAL, "mc_van_mh_round: context and network must share a stream");
    // ids for the sampler: the chains' own Philox chain ids
    static_assert(sizeof(IsingChain) % 4 == 0, "chain layout");
    const uint32_t round = w->round++;
    mc_status s = mc_van_sample(w, n, round, nullptr, w->prop, w->lq); // q(s'')
    if (s != MC_OK)
        return s;
    cudaError_t e = cudaMemcpyAsync(w->spins, w->prop, (size_t)n * L * L, cudaMemcpyDeviceToDevice, w->stream);
    if (e == cudaSuccess)
        e = forward(w, n, 1, w->lq2, nullptr); // q(-s'')
    if (e == cudaSuccess)
        k_energy<<<n, 256, 0, w->stream>>>(w->prop, w->E2, L);
    if (e == cudaSuccess && mc_ising_gather(c, w->spins, 0) != MC_OK)
        return MC_ECUDA;
    if (e == cudaSuccess)
        e = forward(w, n, 0, w->lq3, nullptr); // q(s)
    if (e == cudaSuccess)
        e = forward(w, n, 1, w->lq4, nullptr); // q(-s)
    if (e == cudaSuccess)
        k_energy<<<n, 256, 0, w->stream>>>(w->spins, w->E1, L);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(w->acc, 0, 4, w->stream);
    if (e == cudaSuccess)
        k_mh_accept<<<n, 256, 0, w->stream>>>(static_cast<const IsingChain *>(c->d_chains), c->d_lattice, w->prop,
                                              w->lq, w->lq2, w->lq3, w->lq4, w->E1, w->E2, L, n, w->key, round, w->acc,
                                              w->mh_lr);
    if (e == cudaSuccess)
        e = cudaGetLastError();
    if (e == cudaSuccess && host_accepted) {
        e = cudaMemcpyAsync(host_accepted, w->acc, 4, cudaMemcpyDeviceToHost, w->stream);
        if (e == cudaSuccess)
            e = cudaStreamSynchronize(w->stream);
    }
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_mh_round: ") + cudaGetErrorString(e));
    return host_accepted ? check_err(w, "mc_van_mh_round") : MC_OK;
}

mc_status mc_van_set_round(mc_van *w, uint32_t round)
{
    if (!w)
        return vfail(MC_EINVAL, "NULL network");
    w->round = round;
    return MC_OK;
}

mc_status mc_van_destroy(mc_van *w)
{
    if (!w)
        return MC_OK;
    cudaError_t e = cudaStreamSynchronize(w->stream);
    delete w;
    if (e != cudaSuccess)
        return vfail(MC_ECUDA, std::string("mc_van_destroy: ") + cudaGetErrorString(e));
    return MC_OK;
}

}  // extern "C"
