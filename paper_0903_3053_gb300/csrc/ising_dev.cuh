// ising_dev.cuh -- per-site and per-word device code of the 2D Ising
// Metropolis update (Eq. (1), Sec. 2.3), shared by the grid-mode and resident
// kernels of ising.cu and the persistent batch kernel of batch.cu.
//
// Random numbers: site i = y*(Lx/2) + j of colour c uses word (i & 3) of the
// Philox block with counter (i >> 2, sweep, TAG_METRO | c, chain_id).  A spin
// flips when dE = 2 s h <= 0, or when its word is below
// T[dE] = floor(e^{-beta dE} 2^32).
#pragma once
#include "mc_internal.cuh"

namespace mc {
namespace {

__device__ __forceinline__ uint32_t inc_wrap(uint32_t v, uint32_t n) { return v + 1 == n ? 0u : v + 1; }
__device__ __forceinline__ uint32_t dec_wrap(uint32_t v, uint32_t n) { return v == 0 ? n - 1 : v - 1; }

// Sum two per-thread counters over the CTA; thread 0 receives the totals.
// Every thread of the CTA must call it.
__device__ __forceinline__ void block_sum2(uint32_t &a, uint32_t &b)
{
    __shared__ uint32_t sa[32], sb[32];
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        sa[warp] = a;
        sb[warp] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t ta = 0, tb = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            ta += sa[w];
            tb += sb[w];
        }
        a = ta;
        b = tb;
    }
}

// ------------------------------------------------------------------ int8 layout
// Two forms of the same update of the (up to four) sites of colour C that share
// a Philox block.
//
// int8_group, any even extents: the sites are consecutive in the colour's
// raster order and may run over the end of a row, so the row and column are
// carried from site to site (one division per group, by a multiplication).  The bytes of
// AHEAD sites are loaded before the first of them is updated: loads that follow a store
// wait for it, and a launch of few blocks is one such chain (us per measured sweep with 1 / 4
// ahead: 620 x 170 5.6 / 4.0, four of them 6.1 / 4.7, 1022 x 512 5.6 / 4.7; in shared memory the
// registers cost more than the wait: 512 lattices of 50^2 6.5 / 7.0).
template <int C, bool MEASURE, int LD = kLdPlain, int AHEAD = 4>
__device__ __forceinline__ void int8_group(int8_t *s, const IsingChain &ch, const PhiloxSchedule &ks, uint32_t g,
                                           uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    const uint32_t Lx = ch.Lx, Ly = ch.Ly, half = Lx >> 1, nc = (Lx * Ly) >> 1;
    const uint32_t live = nc - 4 * g < 4u ? nc - 4 * g : 4u;
    uint32_t y, j, rr[4];
    static_assert(AHEAD == 1 || AHEAD == 4, "the draws are made once");
    const auto draw = [&]() {
        const uint4 r = philox4x32_10(make_uint4(g, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
        rr[0] = r.x, rr[1] = r.y, rr[2] = r.z, rr[3] = r.w;
    };
    if (AHEAD == 1)
        draw();
    fast_divmod(4 * g, ch.div_half, y, j);
#pragma unroll
    for (uint32_t q0 = 0; q0 < 4; q0 += AHEAD) {
        if (q0 >= live)
            break;
        uint32_t at[AHEAD];
        int sv[AHEAD], ne[AHEAD], nw[AHEAD], nn[AHEAD], ns[AHEAD];
#pragma unroll
        for (uint32_t q = 0; q < AHEAD; ++q) {
            const uint32_t x = 2 * j + ((y + C) & 1u), row = y * Lx;
            at[q] = row + x;
            sv[q] = lat_load<LD>(&s[row + x]);
            ne[q] = lat_load<LD>(&s[row + inc_wrap(x, Lx)]);
            nw[q] = lat_load<LD>(&s[row + dec_wrap(x, Lx)]);
            nn[q] = lat_load<LD>(&s[dec_wrap(y, Ly) * Lx + x]);
            ns[q] = lat_load<LD>(&s[inc_wrap(y, Ly) * Lx + x]);
            if (q0 + q + 1 < live && ++j == half) { // the last site of the colour is loaded again
                j = 0;
                ++y;
            }
        }
        if (AHEAD > 1)
            draw();
#pragma unroll
        for (uint32_t q = 0; q < AHEAD; ++q) {
            if (q0 + q >= live)
                break;
            const int local = sv[q] * (ne[q] + nw[q] + nn[q] + ns[q]); // dE / 2
            const bool flip = local <= 0 || rr[q0 + q] < (local == 2 ? ch.T2 : ch.T4);
            const int nv = flip ? -sv[q] : sv[q];
            if (flip)
                s[at[q]] = (int8_t)nv;
            if (MEASURE) {
                anti += (uint32_t)(ne[q] != nv) + (uint32_t)(nw[q] != nv) + (uint32_t)(nn[q] != nv) + (uint32_t)(ns[q] != nv);
                const int partner = (at[q] & 1u) ? nw[q] : ne[q]; // colour-0 site (x ^ 1, y)
                up += (uint32_t)(nv > 0) + (uint32_t)(partner > 0);
            }
        }
    }
}

// Comparison of one random word with a threshold, appended to a bit mask: the
// carry out of r + (2^32 - T) is (r >= T) for T >= 1 and is shifted into `g`
// (g <- 2 g + carry), two integer adds per site and no predicate.  T = 0 (no
// site accepted) is fixed up by the caller.
__device__ __forceinline__ void ge_chain2(uint32_t &g2, uint32_t &g4, uint32_t r, uint32_t nT2, uint32_t nT4)
{
    asm("{\n\t.reg .u32 t;\n\t"
        "add.cc.u32 t, %2, %3;\n\t"
        "addc.u32 %0, %0, %0;\n\t"
        "add.cc.u32 t, %2, %4;\n\t"
        "addc.u32 %1, %1, %1;\n\t}"
        : "+r"(g2), "+r"(g4)
        : "r"(r), "r"(nT2), "r"(nT4));
}

// int8_oct, rows of whole groups (Lx % 8 == 0): the group's four sites are every
// other byte of eight consecutive ones, (y, 8 gx .. 8 gx + 7), so the four sites
// are updated as the four bytes of one word.  Spins are the bytes 0x01 and 0xFF,
// whose xor is 0x00 or 0xFE: the anti-aligned neighbours are counted by
// bitwise adders on all four sites at once, as in the 32-spin words, and the
// accept bits of ge_chain2 are spread to bit 1 of the bytes by a multiplication.
// par: parity of the sites' x; w, wu, wd: the eight bytes in the row and in the rows
// above and below; edge: the in-row neighbour outside the eight bytes.  Returns
// whether a site flipped; w is then the row's new bytes.
template <bool MEASURE>
__device__ __forceinline__ bool int8_oct(uint32_t par, uint2 &w, uint2 wu, uint2 wd, uint32_t edge, const uint4 &r,
                                         const IsingChain &ch, uint32_t &anti, uint32_t &up)
{
    const uint32_t selA = par ? 0x7531u : 0x6420u, selO = par ? 0x6420u : 0x7531u;
    uint32_t g2 = 0, g4 = 0;
    ge_chain2(g2, g4, r.w, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.z, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.y, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.x, 0u - ch.T2, 0u - ch.T4);
    // bit q of the nibble to bit 1 of byte q; T = 0 leaves no carry but means r >= T: all ones
    const uint32_t G2 = g2 * 0x00408102u + (ch.T2 == 0 ? 0x02020202u : 0u);
    const uint32_t G4 = g4 * 0x00408102u + (ch.T4 == 0 ? 0x02020202u : 0u);
    const uint32_t sv = __byte_perm(w.x, w.y, selA), ns = __byte_perm(w.x, w.y, selO);
    const uint32_t side = __byte_perm(ns, edge, par ? 0x4321u : 0x2104u);
    const uint32_t a1 = sv ^ __byte_perm(wu.x, wu.y, selA), a2 = sv ^ __byte_perm(wd.x, wd.y, selA), a3 = sv ^ ns,
                   a4 = sv ^ side;
    const uint32_t x = a1 ^ a2 ^ a3, m = (a1 & a2) | (a3 & (a1 | a2)); // 2 m + x = a1 + a2 + a3
    // two or more anti-aligned, or r < T4, or one anti-aligned and r < T2 (T4 <= T2)
    const uint32_t f = ((x & a4) | m | ~G4 | ((x ^ a4) & ~G2)) & 0x02020202u;
    const uint32_t fe = f * 0x7Fu, nv = sv ^ fe; // 0x02 -> 0xFE per byte
    w.x = __byte_perm(nv, ns, par ? 0x1504u : 0x5140u);
    w.y = __byte_perm(nv, ns, par ? 0x3726u : 0x7362u);
    if (MEASURE) { // 0xFE = -2 per anti-aligned bond, +-1 per spin
        int bonds = __dp4a((int)(a1 ^ fe), 0x01010101, 0);
        bonds = __dp4a((int)(a2 ^ fe), 0x01010101, bonds);
        bonds = __dp4a((int)(a3 ^ fe), 0x01010101, bonds);
        bonds = __dp4a((int)(a4 ^ fe), 0x01010101, bonds);
        anti += (uint32_t)(-bonds) >> 1;
        up += (uint32_t)(8 + __dp4a((int)nv, 0x01010101, __dp4a((int)ns, 0x01010101, 0))) >> 1;
    }
    return f != 0;
}

// One group: column gx of row y.  Three 8-byte loads and one byte replace the 20 byte
// loads of int8_group; the other colour's bytes of the 8-byte store hold the values
// they had.  Bound by the schedulers' dispatch (Philox is 72 of its ~200 cycles per
// warp and group); the byte-wise form took 1.6 times as long.
template <int C, bool MEASURE, int LD = kLdPlain>
__device__ __forceinline__ void int8_row(int8_t *s, const IsingChain &ch, const PhiloxSchedule &ks, uint32_t y,
                                         uint32_t gx, uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    const uint32_t Lx = ch.Lx, Ly = ch.Ly, par = (y + C) & 1u, x0 = 8 * gx;
    int8_t *row = s + y * Lx;
    uint2 w = lat_load<LD>(reinterpret_cast<const uint2 *>(row + x0));
    const uint2 wu = lat_load<LD>(reinterpret_cast<const uint2 *>(s + dec_wrap(y, Ly) * Lx + x0));
    const uint2 wd = lat_load<LD>(reinterpret_cast<const uint2 *>(s + inc_wrap(y, Ly) * Lx + x0));
    const uint32_t xs = par ? (x0 + 8 == Lx ? 0u : x0 + 8) : (x0 == 0 ? Lx - 1 : x0 - 1);
    const uint32_t edge = (uint8_t)lat_load<LD>(row + xs);
    const uint4 r = philox4x32_10(make_uint4(y * (Lx >> 3) + gx, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
    if (int8_oct<MEASURE>(par, w, wu, wd, edge, r, ch, anti, up))
        *reinterpret_cast<uint2 *>(row + x0) = w;
}

// The groups of column gx in the row pairs y = 2 yy, 2 yy + 1, yy0 <= yy < yy1.  A
// pair's rows have fixed parities, so the byte selectors are constants, and each
// row is loaded once; a thread's prologue is spread over several groups.  For
// large grid launches (an 8192^2 chain 141 -> 81 us per measured sweep, 4096^2 37
// -> 25); with fewer threads than the chip holds int8_row is faster (1024 x 512
// 3.5 against 4.0 us).
template <int C, bool MEASURE, int LD = kLdPlain>
__device__ __forceinline__ void int8_row_pairs(int8_t *s, const IsingChain &ch, const PhiloxSchedule &ks, uint32_t yy0,
                                               uint32_t yy1, uint32_t gx, uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    const uint32_t Lx = ch.Lx, Ly = ch.Ly, W8 = Lx >> 3, x0 = 8 * gx;
    const uint32_t xl = x0 == 0 ? Lx - 1 : x0 - 1, xr = x0 + 8 == Lx ? 0u : x0 + 8;
    const uint32_t e0 = C ? xr : xl, e1 = C ? xl : xr; // row 2 yy holds sites x = 2 j + C, row 2 yy + 1 x = 2 j + 1 - C
    uint32_t y0 = 2 * yy0, blk = y0 * W8 + gx;
    int8_t *row = s + y0 * Lx;
    const auto oct = [&](const int8_t *p) { return lat_load<LD>(reinterpret_cast<const uint2 *>(p + x0)); };
    uint2 wu = oct(s + dec_wrap(y0, Ly) * Lx), w0 = oct(row);
#pragma unroll 1
    for (uint32_t yy = yy0; yy < yy1; ++yy) {
        int8_t *row1 = row + Lx, *row2 = y0 + 2 == Ly ? s : row1 + Lx;
        uint2 w1 = oct(row1);
        const uint2 wd = oct(row2);
        const uint32_t b0 = (uint8_t)lat_load<LD>(row + e0), b1 = (uint8_t)lat_load<LD>(row1 + e1);
        const uint4 r0 = philox4x32_10(make_uint4(blk, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
        const uint4 r1 = philox4x32_10(make_uint4(blk + W8, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
        const uint2 v0 = w0; // the other colour's bytes of row 2 yy, neighbours of row 2 yy + 1
        const uint2 v1 = w1;
        if (int8_oct<MEASURE>(C, w0, wu, v1, b0, r0, ch, anti, up))
            *reinterpret_cast<uint2 *>(row + x0) = w0;
        if (int8_oct<MEASURE>(1 - C, w1, v0, wd, b1, r1, ch, anti, up))
            *reinterpret_cast<uint2 *>(row1 + x0) = w1;
        wu = v1;
        w0 = wd;
        y0 += 2;
        blk += 2 * W8;
        row += 2 * Lx;
    }
}

// Nibbles: a resident int8 lattice of whole groups (Lx % 8 == 0), held as one byte per group and colour,
// plane[c][y][g] with the group's four sites x = 8 g + 2 j + ((y + c) & 1) as bits j = 0..3 (1 = up).  A
// group's update is then the 32-spin words' logic on four bits: ~110 dispatch cycles per warp and group, 72 of them
// Philox, against ~200 on bytes.  us per measured sweep: 4096 chains of 64^2 19.9 against 26.4, 1024 of 128^2 18.4 / 25.7, one of
// 64^2 1.25 / 1.66 (0.2 of it the record's slot, counted instead of divided for).
// The bits (1 = up) of the four bytes of v.
__device__ __forceinline__ uint32_t nibble_of(uint32_t v)
{
    return ((~v >> 7 & 0x01010101u) * 0x01020408u >> 24) & 15u;
}
// The spin bytes of a nibble: 1 -> 0x01, 0 -> 0xFF.
__device__ __forceinline__ uint32_t bytes_of(uint32_t nib)
{
    return ~(((nib * 0x00204081u) & 0x01010101u) * 0xFEu);
}
// New nibble s given its neighbours (as msc_word).
template <int C>
__device__ __forceinline__ uint32_t nibble_update(uint32_t s, uint32_t nu, uint32_t nd, uint32_t ns, uint32_t side, uint32_t blk,
                                                  uint32_t sweep, const IsingChain &ch, const PhiloxSchedule &ks)
{
    const uint4 r = philox4x32_10(make_uint4(blk, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
    uint32_t g2 = 0, g4 = 0;
    ge_chain2(g2, g4, r.w, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.z, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.y, 0u - ch.T2, 0u - ch.T4);
    ge_chain2(g2, g4, r.x, 0u - ch.T2, 0u - ch.T4);
    g2 |= ch.T2 == 0 ? 15u : 0u;
    g4 |= ch.T4 == 0 ? 15u : 0u;
    const uint32_t a1 = s ^ nu, a2 = s ^ nd, a3 = s ^ ns, a4 = s ^ side; // 1 = anti-aligned
    const uint32_t x = a1 ^ a2 ^ a3, m = (a1 & a2) | (a3 & (a1 | a2)); // 2 m + x = a1 + a2 + a3
    return s ^ (((x & a4) | m | ~g4 | ((x ^ a4) & ~g2)) & 15u);
}
// Group g of rows 2 yy and 2 yy + 1 of plane C (as msc_row_pairs: the rows' parities are fixed and the pair shares
// the other plane's rows).
template <int C, bool MEASURE>
__device__ __forceinline__ void nibble_row_pair(uint8_t *pc, const uint8_t *po, uint32_t yy, uint32_t g, const IsingChain &ch,
                                                const PhiloxSchedule &ks, uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    const uint32_t G = ch.Lx >> 3, Ly = ch.Ly, y0 = 2 * yy, r0 = y0 * G, r1 = r0 + G;
    const uint32_t gl = dec_wrap(g, G), gr = inc_wrap(g, G);
    const uint32_t om = po[dec_wrap(y0, Ly) * G + g], o0 = po[r0 + g], o1 = po[r1 + g],
                   op = po[(y0 + 2 == Ly ? 0u : r1 + G) + g];
    const uint32_t s0 = pc[r0 + g], s1 = pc[r1 + g];
    // offset C on the even row, 1 - C on the odd one: the neighbour at j - 1 (offset 0) or j + 1
    const uint32_t e0 = po[r0 + (C == 0 ? gl : gr)], e1 = po[r1 + (C == 0 ? gr : gl)];
    const uint32_t left = C == 0 ? o0 : o1, le = C == 0 ? e0 : e1, right = C == 0 ? o1 : o0, re = C == 0 ? e1 : e0;
    const uint32_t from_left = (left << 1 | le >> 3) & 15u, from_right = right >> 1 | (re << 3 & 8u);
    const uint32_t side0 = C == 0 ? from_left : from_right, side1 = C == 0 ? from_right : from_left;
    const uint32_t n0 = nibble_update<C>(s0, om, o1, o0, side0, r0 + g, sweep, ch, ks);
    const uint32_t n1 = nibble_update<C>(s1, o0, op, o1, side1, r1 + g, sweep, ch, ks);
    pc[r0 + g] = (uint8_t)n0;
    pc[r1 + g] = (uint8_t)n1;
    if (MEASURE) {
        const uint32_t u0 = om | o1 << 4 | o0 << 8 | side0 << 12, u1 = o0 | op << 4 | o1 << 8 | side1 << 12;
        anti += __popc((n0 * 0x1111u ^ u0) | (n1 * 0x1111u ^ u1) << 16);
        up += __popc(n0 | o0 << 4 | n1 << 8 | o1 << 12);
    }
}

// First row pair of run q of a column (run `runs`: their number).
__device__ __forceinline__ uint32_t run_start(const IsingChain &ch, uint32_t q)
{
    return q * ch.run + min(q, (ch.Ly >> 1) - ch.runs * ch.run);
}

// Rows of partial groups (Lx no multiple of 8, at least 8): a group that lies inside a row is updated as in
// int8_row, its eight bytes loaded and stored as four pairs (rows start on even bytes).  The groups over a row's end
// take int8_group, in warps of their own: units 0 .. Ly n - 1 are the slots y n + i of at most n = Lx / 8 inner groups of a
// row, then follows the group at each row's end.  For large grid launches: 4094 x 4098 63.7 -> 52.1 us per measured
// sweep, three of 998 x 1050 16.4 -> 14.6, 2046^2 18.3 -> 17.1; smaller launches and resident lattices are
// faster with one form for all (1022 x 512 4.7 against 6.5, resident 50^2 2.3 against 2.9).
template <int C, bool MEASURE, int LD>
__device__ __forceinline__ void int8_inner(int8_t *s, const IsingChain &ch, const PhiloxSchedule &ks, uint32_t y, uint32_t g,
                                           uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    const uint32_t Lx = ch.Lx, Ly = ch.Ly, par = (y + C) & 1u, x0 = 2 * (4 * g - y * (Lx >> 1));
    int8_t *row = s + y * Lx;
    auto eight = [&](const int8_t *p) {
        const uint16_t *h = reinterpret_cast<const uint16_t *>(p + x0);
        const uint32_t a = lat_load<LD>(h), b = lat_load<LD>(h + 1), c = lat_load<LD>(h + 2), d = lat_load<LD>(h + 3);
        return make_uint2(__byte_perm(a, b, 0x5410u), __byte_perm(c, d, 0x5410u));
    };
    uint2 w = eight(row);
    const uint2 wu = eight(s + dec_wrap(y, Ly) * Lx), wd = eight(s + inc_wrap(y, Ly) * Lx);
    const uint32_t xs = par ? (x0 + 8 == Lx ? 0u : x0 + 8) : (x0 == 0 ? Lx - 1 : x0 - 1);
    const uint32_t edge = (uint8_t)lat_load<LD>(row + xs);
    const uint4 r = philox4x32_10(make_uint4(g, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
    if (int8_oct<MEASURE>(par, w, wu, wd, edge, r, ch, anti, up)) {
        uint16_t *h = reinterpret_cast<uint16_t *>(row + x0);
        h[0] = (uint16_t)w.x;
        h[1] = (uint16_t)(w.x >> 16);
        h[2] = (uint16_t)w.y;
        h[3] = (uint16_t)(w.y >> 16);
    }
}

// Work units of a chain's half-sweep: Philox groups, or (PAIRS, large grid launches) runs of
// row pairs of a group column or, rows of partial groups, inner groups and row ends; and unit u of the chain.
template <bool PAIRS>
__host__ __device__ __forceinline__ uint32_t int8_units(const IsingChain &ch)
{
    if (PAIRS && (ch.Lx & 7u) == 0)
        return ch.runs * (ch.Lx >> 3);
    if (PAIRS && ch.Lx > 8)
        return ch.Ly * ((ch.Lx >> 3) + 1);
    return (((ch.Lx * ch.Ly) >> 1) + 3) >> 2;
}
template <int C, bool MEASURE, bool PAIRS = false, int LD = kLdPlain, int AHEAD = 4>
__device__ __forceinline__ void int8_unit(int8_t *s, const IsingChain &ch, const PhiloxSchedule &ks, uint32_t u,
                                          uint32_t sweep, uint32_t &anti, uint32_t &up)
{
    if (AHEAD == 0 || (ch.Lx & 7u) == 0) { // AHEAD 0: known by the launch
        const uint32_t q = fast_div(4 * u, ch.div_half), gx = u - q * (ch.Lx >> 3); // u / (Lx / 8)
        if (PAIRS)
            int8_row_pairs<C, MEASURE, LD>(s, ch, ks, run_start(ch, q), run_start(ch, q + 1), gx, sweep, anti, up);
        else
            int8_row<C, MEASURE, LD>(s, ch, ks, q, gx, sweep, anti, up);
    } else if (PAIRS && ch.Lx > 8) {
        const uint32_t n = ch.Lx >> 3, half = ch.Lx >> 1;
        if (u < ch.Ly * n) {
            const uint32_t y = fast_div(u, ch.div_inner), g = ((y * half + 3) >> 2) + u - y * n;
            if (4 * g + 4 <= (y + 1) * half)
                int8_inner<C, MEASURE, LD>(s, ch, ks, y, g, sweep, anti, up);
        } else {
            const uint32_t end = (u - ch.Ly * n + 1) * half; // the first site of the next row
            if (end & 3u)
                int8_group<C, MEASURE, LD>(s, ch, ks, end >> 2, sweep, anti, up);
        }
    } else {
        int8_group<C, MEASURE, LD, AHEAD ? AHEAD : 4>(s, ch, ks, u, sweep, anti, up);
    }
}

// ------------------------------------------------------------------ MSC layout
// New value of one colour-C word given its four neighbour words.  Every 4-site
// Philox block is drawn (a per-block skip branch costs more than it saves).
// Every site is compared with both thresholds, as two carry chains that build
// the masks g2 = (r >= T2) and g4 = (r >= T4) with site b at bit b (sites are
// visited from 31 down to 0).  A site with two or more anti-aligned neighbours
// flips, one with one (dE = 4) iff r < T2, one with none (dE = 8) iff r < T4;
// since T4 <= T2, r < T4 flips in every case.  (A per-site select of the
// threshold followed by one compare measured 12% slower; predicates in place
// of the carry chains 20% slower: an integer add takes one dispatch cycle of a
// scheduler, a compare, logic or multiply instruction two.)  Bound by that dispatch:
// a 4-site Philox block is 17 wide multiplies and 19 three-input xors, 72 cycles
// per warp, its compares 16 more; 103 cycles measured (110 with a thread per row
// pair and the neighbour count as half adders): 1.365e12 -> 1.47e12 flips/s on a
// 32768^2 chain.
template <int C>
__device__ __forceinline__ uint32_t msc_word(uint32_t s, uint32_t nu, uint32_t nd, uint32_t ns, uint32_t side,
                                             uint32_t blk0, uint32_t sweep, const IsingChain &ch,
                                             const PhiloxSchedule &ks)
{
    const uint32_t a1 = s ^ nu, a2 = s ^ nd, a3 = s ^ ns, a4 = s ^ side; // 1 = anti-aligned
    const uint32_t x = a1 ^ a2 ^ a3, m = (a1 & a2) | (a3 & (a1 | a2)); // 2 m + x = a1 + a2 + a3
    const uint32_t nT2 = 0u - ch.T2, nT4 = 0u - ch.T4;
    uint32_t g2 = 0, g4 = 0;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        const uint4 r = philox4x32_10(make_uint4(blk0 + k, sweep, kTagIsingMetro | (uint32_t)C, ch.chain_id), ks);
        ge_chain2(g2, g4, r.w, nT2, nT4);
        ge_chain2(g2, g4, r.z, nT2, nT4);
        ge_chain2(g2, g4, r.y, nT2, nT4);
        ge_chain2(g2, g4, r.x, nT2, nT4);
    }
    if (ch.T2 == 0)
        g2 = ~0u;
    if (ch.T4 == 0)
        g4 = ~0u;
    return s ^ ((x & a4) | m | ~g4 | ((x ^ a4) & ~g2));
}

// Update words (y, w) of plane C for the row pairs y = 2 yy, 2 yy + 1 with yy0 <=
// yy < yy1.  The two rows of a pair share the other plane's rows 2 yy and 2 yy +
// 1 as neighbours and the next pair shares rows 2 yy + 1 and 2 yy + 2, so each row
// of the other plane is loaded once.  Row y holds sites x = 2 j + ((y + C) & 1):
// offset C on the even row, 1 - C on the odd one, which decides the side (j - 1
// or j + 1) neighbour.
template <int C, bool MEASURE, int LD = kLdPlain>
__device__ __forceinline__ void msc_row_pairs(uint32_t *pc, const uint32_t *po, uint32_t yy0, uint32_t yy1, uint32_t w,
                                              const IsingChain &ch, const PhiloxSchedule &ks, uint32_t sweep,
                                              uint32_t &anti, uint32_t &up)
{
    const uint32_t W = ch.W, Ly = ch.Ly, bpr = ch.Lx >> 3; // bpr: Philox blocks per row of one colour
    const uint32_t wl = dec_wrap(w, W), wr = inc_wrap(w, W);
    uint32_t y0 = 2 * yy0, r0 = y0 * W, blk = y0 * bpr + 8 * w;
    uint32_t om = lat_load<LD>(&po[dec_wrap(y0, Ly) * W + w]), o0 = lat_load<LD>(&po[r0 + w]);
#pragma unroll 1
    for (uint32_t yy = yy0; yy < yy1; ++yy) {
        const uint32_t r1 = r0 + W, r2 = y0 + 2 == Ly ? 0u : r1 + W;
        const uint32_t o1 = lat_load<LD>(&po[r1 + w]), op = lat_load<LD>(&po[r2 + w]);
        uint32_t side0, side1;
        if (C == 0) {
            side0 = (o0 << 1) | (lat_load<LD>(&po[r0 + wl]) >> 31);
            side1 = (o1 >> 1) | (lat_load<LD>(&po[r1 + wr]) << 31);
        } else {
            side0 = (o0 >> 1) | (lat_load<LD>(&po[r0 + wr]) << 31);
            side1 = (o1 << 1) | (lat_load<LD>(&po[r1 + wl]) >> 31);
        }
        const uint32_t s0 = lat_load<LD>(&pc[r0 + w]), s1 = lat_load<LD>(&pc[r1 + w]);
        const uint32_t n0 = msc_word<C>(s0, om, o1, o0, side0, blk, sweep, ch, ks);
        const uint32_t n1 = msc_word<C>(s1, o0, op, o1, side1, blk + bpr, sweep, ch, ks);
        if (n0 != s0)
            pc[r0 + w] = n0;
        if (n1 != s1)
            pc[r1 + w] = n1;
        if (MEASURE) {
            anti += __popc(n0 ^ om) + __popc(n0 ^ o1) + __popc(n0 ^ o0) + __popc(n0 ^ side0) + __popc(n1 ^ o0) +
                    __popc(n1 ^ op) + __popc(n1 ^ o1) + __popc(n1 ^ side1);
            up += __popc(n0) + __popc(o0) + __popc(n1) + __popc(o1);
        }
        om = o1;
        o0 = op;
        y0 += 2;
        r0 += 2 * W;
        blk += 2 * bpr;
    }
}

// One row pair.
template <int C, bool MEASURE, int LD = kLdPlain>
__device__ __forceinline__ void msc_row_pair(uint32_t *pc, const uint32_t *po, uint32_t yy, uint32_t w,
                                             const IsingChain &ch, const PhiloxSchedule &ks, uint32_t sweep,
                                             uint32_t &anti, uint32_t &up)
{
    msc_row_pairs<C, MEASURE, LD>(pc, po, yy, yy + 1, w, ch, ks, sweep, anti, up);
}

// Gather the neighbours of word (y, w) of plane C from the other plane `po`.
template <int C>
__device__ __forceinline__ void msc_neighbours(const uint32_t *po, uint32_t y, uint32_t w, uint32_t W, uint32_t Ly,
                                               uint32_t &nu, uint32_t &nd, uint32_t &ns, uint32_t &side)
{
    const uint32_t row = y * W;
    nu = po[dec_wrap(y, Ly) * W + w];
    nd = po[inc_wrap(y, Ly) * W + w];
    ns = po[row + w];
    if (((y + C) & 1u) == 0) { // x = 2j: other colour at j-1 and j
        const uint32_t prev = po[row + dec_wrap(w, W)];
        side = (ns << 1) | (prev >> 31);
    } else { // x = 2j+1: other colour at j and j+1
        const uint32_t next = po[row + inc_wrap(w, W)];
        side = (ns >> 1) | (next << 31);
    }
}

}  // namespace
}  // namespace mc
