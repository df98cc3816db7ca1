// su2_dev.cuh -- per-link device code of the 4D SU(2) heat-bath (Sec. 2.4,
// Eqs. (2)-(7)), shared by the per-phase kernels of su2.cu, the persistent
// batch kernel of batch.cu and the resident kernel of su2_resident.cu.
// Quaternion links (U0, U1, U2, U3) of Eq. (4) in FP32, stored per chain as
// float4 [parity][mu][site-within-parity].
//
// Every floating-point sum of products on the update path is written with
// explicit rounding intrinsics (__fmaf_rn, __fmul_rn, __fadd_rn, ...), which
// the compiler neither contracts nor reorders: how it would otherwise fuse
// a*b - c*d into an FMA depends on the surrounding code, and the kernels that
// share these functions must produce bit-identical links.
#pragma once
#include "mc_internal.cuh"

namespace mc {
namespace {

// (a0 + i a.sigma)(b0 + i b.sigma) = (a0 b0 - a.b) + i (a0 b + b0 a - a x b).sigma,
// each component one product and three fused multiply-adds in a fixed order.
__device__ __forceinline__ float4 qmul(float4 a, float4 b)
{
    return make_float4(__fmaf_rn(-a.w, b.w, __fmaf_rn(-a.z, b.z, __fmaf_rn(-a.y, b.y, __fmul_rn(a.x, b.x)))),
                       __fmaf_rn(a.w, b.z, __fmaf_rn(-a.z, b.w, __fmaf_rn(b.x, a.y, __fmul_rn(a.x, b.y)))),
                       __fmaf_rn(a.y, b.w, __fmaf_rn(-a.w, b.y, __fmaf_rn(b.x, a.z, __fmul_rn(a.x, b.z)))),
                       __fmaf_rn(a.z, b.y, __fmaf_rn(-a.y, b.z, __fmaf_rn(b.x, a.w, __fmul_rn(a.x, b.w)))));
}
__device__ __forceinline__ float4 qdag(float4 a) { return make_float4(a.x, -a.y, -a.z, -a.w); }
__device__ __forceinline__ float4 qadd(float4 a, float4 b)
{
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}
__device__ __forceinline__ float qdot(float4 a, float4 b)
{
    return __fmaf_rn(a.w, b.w, __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmul_rn(a.x, b.x))));
}
__device__ __forceinline__ float4 qscale(float4 a, float s)
{
    return make_float4(__fmul_rn(a.x, s), __fmul_rn(a.y, s), __fmul_rn(a.z, s), __fmul_rn(a.w, s));
}

// A site and its neighbours, as byte offsets into the (parity, mu) link arrays.
// A step along directions 2, 3 or 0 moves the index within the parity by a constant
// (wrapped at the ends); the index s >> 1 is the same for both sites of an x1
// pair, so a step along direction 1 moves it only when it leaves the pair.  Each
// coordinate's steps are independent of the others', and one offset serves the
// arrays of every direction.  (Canonical indices, neighbour by neighbour, with an
// array index each took 2.4x the integer instructions.)
struct LinkSite {
    uint32_t o;            // offset of the site
    uint32_t fw[4], bw[4]; // what a step forward / backward along each direction adds to it (mod 2^32)
    uint32_t b;            // parity of x1: the canonical index is 2 e + b
    uint32_t par;          // parity of the site
};

// Coordinates of the x1 pair e = x1/2 + (L1/2) (x2 + L2 (x3 + L3 x0)), the
// steps that its two sites share, and the site with x1 parity b or of parity p.
__device__ __forceinline__ LinkSite link_pair(const Su2Chain &ch, uint32_t e, uint32_t &x1h)
{
    uint32_t q1, q2, x2, x0, x3; // magic-number divisions (fastdiv.cuh)
    fast_divmod(e, ch.div1h, q1, x1h);
    fast_divmod(q1, ch.div2, q2, x2);
    fast_divmod(q2, ch.div3, x0, x3);
    LinkSite s;
    s.o = 16u * e;
    s.par = (x0 + x2 + x3) & 1u; // of the pair's even-x1 site
    s.fw[2] = x2 + 1 == ch.div2.d ? ch.step2 - ch.step3 : ch.step2;
    s.bw[2] = x2 == 0 ? ch.step3 - ch.step2 : 0u - ch.step2;
    s.fw[3] = x3 + 1 == ch.div3.d ? ch.step3 - ch.step0 : ch.step3;
    s.bw[3] = x3 == 0 ? ch.step0 - ch.step3 : 0u - ch.step3;
    s.fw[0] = x0 + 1 == (uint32_t)ch.L[0] ? ch.step0 - ch.bytes : ch.step0;
    s.bw[0] = x0 == 0 ? ch.bytes - ch.step0 : 0u - ch.step0;
    return s;
}
__device__ __forceinline__ LinkSite link_of_pair(const Su2Chain &ch, LinkSite s, uint32_t x1h, uint32_t b)
{
    s.b = b;
    s.par ^= b;
    s.fw[1] = b ? (x1h + 1 == ch.div1h.d ? 16u - ch.step2 : 16u) : 0u;
    s.bw[1] = b ? 0u : (x1h == 0 ? ch.step2 - 16u : 0u - 16u);
    return s;
}
__device__ __forceinline__ LinkSite link_site(const Su2Chain &ch, int p, uint32_t e)
{
    uint32_t x1h;
    const LinkSite s = link_pair(ch, e, x1h);
    return link_of_pair(ch, s, x1h, s.par ^ (uint32_t)p);
}

// The link in direction `dir` of the parity-`par` site at byte offset o.
template <int LD>
__device__ __forceinline__ float4 link_at(const float4 *U, const Su2Chain &ch, int par, int dir, uint32_t o)
{
    const char *base = reinterpret_cast<const char *>(U) + (size_t)(par * 4 + dir) * ch.bytes;
    return lat_load<LD>(reinterpret_cast<const float4 *>(base + o));
}

// The two staples of Eq. (6) in the (MU, NU) plane:
//   U_nu(x) U_mu(x+nu) U_nu(x+mu)^+  +  U_nu(x-nu)^+ U_mu(x-nu) U_nu(x-nu+mu).
// x + nu, x + mu and x - nu have parity 1 - P; x - nu + mu has parity P.
template <int MU, int NU, int P, int LD>
__device__ __forceinline__ float4 staple_pair(const float4 *__restrict__ U, const Su2Chain &ch, const LinkSite &x)
{
    constexpr int Q = 1 - P;
    const uint32_t pm = x.o + x.fw[MU], pn = x.o + x.fw[NU], mn = x.o + x.bw[NU], mnpm = mn + x.fw[MU];
    const float4 a = link_at<LD>(U, ch, P, NU, x.o);
    const float4 b = link_at<LD>(U, ch, Q, MU, pn);
    const float4 c = link_at<LD>(U, ch, Q, NU, pm);
    const float4 d = link_at<LD>(U, ch, Q, NU, mn);
    const float4 f = link_at<LD>(U, ch, Q, MU, mn);
    const float4 h = link_at<LD>(U, ch, P, NU, mnpm);
    return qadd(qmul(qmul(a, b), qdag(c)), qmul(qmul(qdag(d), f), h));
}

template <int MU, int P, int LD>
__device__ __forceinline__ float4 staple(const float4 *__restrict__ U, const Su2Chain &ch, const LinkSite &x)
{
    float4 W = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MU != 0) W = qadd(W, staple_pair<MU, 0, P, LD>(U, ch, x));
    if (MU != 1) W = qadd(W, staple_pair<MU, 1, P, LD>(U, ch, x));
    if (MU != 2) W = qadd(W, staple_pair<MU, 2, P, LD>(U, ch, x));
    if (MU != 3) W = qadd(W, staple_pair<MU, 3, P, LD>(U, ch, x));
    return W;
}

// Counts a link update whose every try was rejected.  Out of line on purpose:
// with the atomic inlined, the phase kernel ran 11% slower on 4 x 32^4
// although the branch is essentially never taken.
__device__ __noinline__ void count_heatbath_failure(DevState *state) { atomicAdd(&state->hb_failures, 1ull); }

constexpr int kKpTries = 8;
constexpr int kCreutzTries = 64;
constexpr uint8_t kFailed = 255;

// The part of a Kennedy-Pendleton try that does not depend on alpha:
// q = -(log u1 + cos^2(2 pi u2) log u3), so that lambda^2 = q / (2 alpha), and
// u4^2 for the acceptance test.
struct KpFirstTry {
    float q, u4sq;
};

__device__ __forceinline__ KpFirstTry kp_parts(uint4 r)
{
    const float u1 = uniform_open0(r.x), u2 = uniform_open0(r.y);
    const float u3 = uniform_open0(r.z), u4 = uniform_open0(r.w);
    const float cs = cospif(2.0f * u2);
    return KpFirstTry{-__fmaf_rn(__fmul_rn(cs, cs), logf(u3), logf(u1)), __fmul_rn(u4, u4)};
}

// Acceptance of a Kennedy-Pendleton try at alpha > 0: lambda^2 = q / (2 alpha),
// accepted iff u4^2 <= 1 - lambda^2; a0 = 1 - 2 lambda^2 either way.
__device__ __forceinline__ bool kp_accept(const KpFirstTry &f, float alpha, float &a0)
{
    const float lam2 = __fmul_rn(f.q, __fdividef(0.5f, alpha));
    a0 = __fmaf_rn(-2.0f, lam2, 1.0f);
    return f.u4sq <= __fsub_rn(1.0f, lam2);
}

// One heat-bath try t for a0 ~ sqrt(1-a0^2) exp(alpha a0): Kennedy-Pendleton
// for t < kKpTries (alpha > 0), Creutz after; a0 is set whether or not the try
// is accepted.
__device__ __forceinline__ bool heatbath_try(int t, float alpha, uint32_t e, uint32_t sweep, uint32_t sel,
                                             const Su2Chain &ch, const PhiloxSchedule &ks, float &a0)
{
    const uint4 r = philox4x32_10(make_uint4(e, sweep, kTagSu2Heatbath | sel | (uint32_t)t, ch.chain_id), ks);
    if (t < kKpTries)
        return kp_accept(kp_parts(r), alpha, a0);
    const float cexp = alpha > 0.f ? -expm1f(-2.0f * alpha) : 0.f; // 1 - e^{-2 alpha}
    const float u1 = uniform_open0(r.x), u2 = uniform_open0(r.y);
    const float c = alpha > 0.f ? __fadd_rn(1.0f, log1pf(__fmul_rn(-__fsub_rn(1.0f, u1), cexp)) / alpha)
                                : __fmaf_rn(2.0f, u1, -1.0f);
    a0 = c;
    return __fmul_rn(u2, u2) <= __fmaf_rn(-c, c, 1.0f);
}

// The alpha-free part of Kennedy-Pendleton try t of a link (t = 0 for the
// first try; `sel` carries parity and direction).  The grid kernel computes
// try 0's part before the staple, so that it fills the wait for the staple's
// loads; the resident kernel computes several tries' parts at once.
__device__ __forceinline__ KpFirstTry kp_first_try(uint32_t e, uint32_t sweep, uint32_t sel, const Su2Chain &ch,
                                                   const PhiloxSchedule &ks)
{
    return kp_parts(philox4x32_10(make_uint4(e, sweep, kTagSu2Heatbath | sel, ch.chain_id), ks));
}

// Heat-bath draw of a0: tries 0 .. kKpTries - 1 by Kennedy-Pendleton (skipped
// when alpha = 0; the first AHEAD tries from their precomputed parts f), then Creutz up to
// kKpTries + kCreutzTries - 1; returns the try taken, or kFailed.  One loop
// over both samplers (measured ~2% faster on 4 x 32^4 than a loop per
// sampler); the same draws as heatbath_try for every t.
template <int AHEAD>
__device__ __forceinline__ int draw_a0(float alpha, uint32_t e, uint32_t sweep, uint32_t sel, const Su2Chain &ch,
                                       const PhiloxSchedule &ks, const KpFirstTry (&f)[AHEAD], float &a0)
{
    if (alpha > 0.f) {
#pragma unroll
        for (int t = 0; t < AHEAD; ++t) {
            float a;
            if (kp_accept(f[t], alpha, a)) {
                a0 = a;
                return t;
            }
        }
    }
    for (int t = alpha > 0.f ? AHEAD : kKpTries; t < kKpTries + kCreutzTries; ++t) {
        float a;
        if (heatbath_try(t, alpha, e, sweep, sel, ch, ks, a)) {
            a0 = a;
            return t;
        }
    }
    return kFailed;
}

// V = W / |W| and alpha = beta |W| of a staple W (V = 1 for a vanishing staple);
// one reciprocal square root serves both.
__device__ __forceinline__ void staple_to_heatbath(const float4 &W, float beta, float4 &V, float &alpha)
{
    const float k2 = qdot(W, W);
    V = make_float4(1.f, 0.f, 0.f, 0.f);
    float kn = 0.f;
    if (k2 > 0.f) {
        const float inv = rsqrtf(k2);
        V = qscale(W, inv);
        kn = __fmul_rn(k2, inv);
    }
    alpha = __fmul_rn(beta, kn);
}

// Uniform direction on S^2 for the vector part of X in Eq. (5): cos theta =
// 2 u1 - 1, phi = 2 pi u2 from the link's direction Philox block.
struct S2Direction {
    float ct, st, sphi, cphi;
};

template <int P, int MU>
__device__ __forceinline__ S2Direction su2_direction(const Su2Chain &ch, const PhiloxSchedule &ks, uint32_t e,
                                                     uint32_t sweep)
{
    const uint32_t sel = ((uint32_t)P << 12) | ((uint32_t)MU << 8);
    const uint4 r = philox4x32_10(make_uint4(e, sweep, kTagSu2Direction | sel, ch.chain_id), ks);
    S2Direction d;
    d.ct = __fmaf_rn(2.0f, uniform_open0(r.x), -1.0f);
    // phi = 2 pi u2 reduced to (-pi, pi]: u2 - 1 for u2 > 1/2 (exact in FP32)
    const float u2 = uniform_open0(r.y), v = u2 > 0.5f ? u2 - 1.0f : u2;
    __sincosf(6.2831853f * v, &d.sphi, &d.cphi);
    const float s2 = fmaxf(0.f, __fmaf_rn(-d.ct, d.ct, 1.0f));
    d.st = s2 > 0.f ? __fmul_rn(s2, rsqrtf(s2)) : 0.f;
    return d;
}

// The new link X V of Eq. (5) for the drawn a0 and direction d, X = a0 +
// i sqrt(1 - a0^2) d.sigma, reprojected onto SU(2) (Eq. (7)).
__device__ __forceinline__ float4 heatbath_link(float a0, const float4 &V, const S2Direction &d)
{
    const float r2 = fmaxf(0.f, __fmaf_rn(-a0, a0, 1.0f));
    const float rad = r2 > 0.f ? __fmul_rn(r2, rsqrtf(r2)) : 0.f;
    const float rs = __fmul_rn(rad, d.st);
    const float4 X = make_float4(a0, __fmul_rn(rs, d.cphi), __fmul_rn(rs, d.sphi), __fmul_rn(rad, d.ct));
    const float4 Un = qmul(X, V);
    return qscale(Un, rsqrtf(qdot(Un, Un)));
}

// Heat-bath draw and store for a link whose staple is (V, alpha) and whose
// direction is d: a0 by Kennedy-Pendleton / Creutz, U = X V, reprojection
// (Eqs. (5), (7)).  Returns the try taken (kFailed: link unchanged, counted).
template <int P, int MU, bool INLINE_FAIL, int AHEAD>
__device__ __forceinline__ int su2_link_draw(float4 *U, const Su2Chain &ch, const PhiloxSchedule &ks, uint32_t e,
                                             uint32_t sweep, float4 V, float alpha, const S2Direction &d,
                                             const KpFirstTry (&f)[AHEAD], DevState *state)
{
    const uint32_t sel = ((uint32_t)P << 12) | ((uint32_t)MU << 8);
    float a0 = 0.f;
    const int t = draw_a0(alpha, e, sweep, sel, ch, ks, f, a0);
    if (t == kFailed) {
        if (INLINE_FAIL)
            atomicAdd(&state->hb_failures, 1ull);
        else
            count_heatbath_failure(state);
        return t;
    }
    U[(size_t)(P * 4 + MU) * ch.nh + e] = heatbath_link(a0, V, d);
    return t;
}

// Heat-bath update of the link U_MU(x) at site e of parity P (Eqs. (5)-(7)):
// staple, a0 by Kennedy-Pendleton / Creutz, direction on S^2, U = X V,
// reprojection.  REC: store the try taken at tries[2 e + b][MU] (canonical
// site 2 e + b, b the parity bit of x1); a separate instantiation so that the
// sweeps that do not record keep no extra state live across the heat-bath loop.
// INLINE_FAIL: count a failed update with an inlined atomic (the persistent
// batch kernel, where the out-of-line call costs a stack frame) instead of
// count_heatbath_failure.
// CHAINED: the links are read only after chain_wait (the phase kernels).
template <int P, int MU, int LD, bool REC, bool INLINE_FAIL = false, int EARLY = 2, bool CHAINED = false>
__device__ __forceinline__ void su2_update_link(float4 *U, const Su2Chain &ch, const PhiloxSchedule &ks, uint32_t e,
                                                uint32_t sweep, uint8_t *tries, DevState *state, bool release = false)
{
    // The direction and the alpha-free part of the first heat-bath try do not
    // depend on the staple: computed first (EARLY = 2), their Philox blocks,
    // logarithms and trigonometry fill the wait for the staple's 18 link loads
    // (0.609 against 0.650 ms per sweep of 4 x 32^4, identical links).  EARLY
    // = 1 moves only the direction, 0 neither; the draws are the same.
    const uint32_t sel = ((uint32_t)P << 12) | ((uint32_t)MU << 8);
    constexpr int AHEAD = EARLY >= 3 ? EARLY - 1 : 1;
    S2Direction d;
    KpFirstTry f[AHEAD];
    if (EARLY >= 1)
        d = su2_direction<P, MU>(ch, ks, e, sweep);
    if (EARLY >= 2)
#pragma unroll
        for (int t = 0; t < AHEAD; ++t)
            f[t] = kp_first_try(e, sweep, sel | (uint32_t)t, ch, ks);
    float4 V;
    float alpha;
    const LinkSite x = link_site(ch, P, e);
    if (CHAINED)
        chain_wait(release);
    staple_to_heatbath(staple<MU, P, LD>(U, ch, x), ch.beta, V, alpha);
    if (EARLY < 2)
        f[0] = kp_first_try(e, sweep, sel, ch, ks);
    if (EARLY < 1)
        d = su2_direction<P, MU>(ch, ks, e, sweep);
    const int t = su2_link_draw<P, MU, INLINE_FAIL, AHEAD>(U, ch, ks, e, sweep, V, alpha, d, f, state);
    if (REC)
        tries[ch.tries_off + (size_t)(2 * e + x.b) * 4 + MU] = (uint8_t)t; // canonical site 2 e + b
}

// Overrelaxation of the link U_MU(x) at site e of parity P (the
// "overrelaxation" of Sec. 2.4's heat-bath with overrelaxation): the
// reflection U' = V U^dag V, V = W / |W|, keeps Re Tr(U W^dag) and so the
// action; deterministic, no random numbers.  A vanishing staple leaves the link
// as it is.  The result is reprojected onto SU(2).
template <int P, int MU, int LD, bool CHAINED = false>
__device__ __forceinline__ void su2_overrelax_link(float4 *U, const Su2Chain &ch, uint32_t e, bool release = false)
{
    float4 V;
    {
        const LinkSite x = link_site(ch, P, e);
        if (CHAINED)
            chain_wait(release);
        const float4 W = staple<MU, P, LD>(U, ch, x);
        const float k2 = qdot(W, W);
        if (!(k2 > 0.f))
            return;
        V = qscale(W, 1.0f / sqrtf(k2));
    }
    float4 *dst = &U[(size_t)(P * 4 + MU) * ch.nh + e];
    const float4 u = lat_load<LD>(dst);
    float4 Un = qmul(qmul(V, qdag(u)), V);
    *dst = qscale(Un, rsqrtf(qdot(Un, Un)));
}

template <int LD>
__device__ __forceinline__ void su2_overrelax_link_rt(int phase, float4 *U, const Su2Chain &ch, uint32_t e)
{
    switch (phase) {
    case 0: su2_overrelax_link<1, 0, LD>(U, ch, e); break;
    case 1: su2_overrelax_link<1, 1, LD>(U, ch, e); break;
    case 2: su2_overrelax_link<1, 2, LD>(U, ch, e); break;
    case 3: su2_overrelax_link<1, 3, LD>(U, ch, e); break;
    case 4: su2_overrelax_link<0, 0, LD>(U, ch, e); break;
    case 5: su2_overrelax_link<0, 1, LD>(U, ch, e); break;
    case 6: su2_overrelax_link<0, 2, LD>(U, ch, e); break;
    default: su2_overrelax_link<0, 3, LD>(U, ch, e); break;
    }
}

// How much of the RNG-only work the persistent batch kernel moves ahead of the
// staple (the EARLY argument of su2_update_link).  With its 128-register
// budget the direction alone measured best on the batched workload: 0.459 ms
// per sweep against 0.475-0.491 (direction and first try) and 0.487 (neither).
#ifndef MC_GROUP_EARLY
#define MC_GROUP_EARLY 1
#endif

// Runtime (P, MU) dispatch of su2_update_link for the persistent batch kernel
// (no try record, inlined failure count).
template <int LD>
__device__ __forceinline__ void su2_update_link_rt(int phase, float4 *U, const Su2Chain &ch, const PhiloxSchedule &ks,
                                                   uint32_t e, uint32_t sweep, DevState *state)
{
    switch (phase) { // phase = position in the sweep: (odd, mu = 0..3), then (even, mu = 0..3)
    case 0: su2_update_link<1, 0, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 1: su2_update_link<1, 1, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 2: su2_update_link<1, 2, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 3: su2_update_link<1, 3, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 4: su2_update_link<0, 0, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 5: su2_update_link<0, 1, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    case 6: su2_update_link<0, 2, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    default: su2_update_link<0, 3, LD, false, true, MC_GROUP_EARLY>(U, ch, ks, e, sweep, nullptr, state); break;
    }
}

// Plaquette sums in exact fixed point: each plaquette's FP32 value h (|h| <= 1)
// is rounded to a multiple of 2^-29 (an int32) and summed in int64.  The sum is
// exact, hence independent of the order, of the launch shape and of how the
// plaquettes are shared out among threads, for up to 2.8e9 sites, and it stays
// off the GB300's FP64 pipe, which made an FP64 shuffle reduction the larger
// part of the measurement's cost.
constexpr float kPlaqFix = 536870912.0f; // 2^29 (kPlaqUnfix, its inverse, is in mc_internal.cuh)
__device__ __forceinline__ long long plaq_fixed(float v) { return (long long)__float2int_rn(v * kPlaqFix); }

__device__ __forceinline__ long long warp_sum_ll(long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// (1/2) Tr U_munu(x) of Eq. (3): (1/2) Tr[U_mu(x) U_nu(x+mu) (U_nu(x) U_mu(x+nu))^+]
// = A . B with A = U_mu(x) U_nu(x+mu), B = U_nu(x) U_mu(x+nu).
__device__ __forceinline__ float plaquette_value(float4 umu_x, float4 unu_xmu, float4 unu_x, float4 umu_xnu)
{
    return qdot(qmul(umu_x, unu_xmu), qmul(unu_x, umu_xnu));
}

// The six plaquettes at a site, from its own links Ux[mu] and the forward
// links Uf[mu][nu] = U_nu(x + mu), added in fixed point: spatial planes to ps,
// temporal (mu = 0) to pt.
__device__ __forceinline__ void plaquettes_of(const float4 (&Ux)[4], const float4 (&Uf)[4][4], long long &ps,
                                              long long &pt)
{
#pragma unroll
    for (int mu = 0; mu < 4; ++mu)
#pragma unroll
        for (int nu = mu + 1; nu < 4; ++nu) {
            const long long h = plaq_fixed(plaquette_value(Ux[mu], Uf[mu][nu], Ux[nu], Uf[nu][mu]));
            if (mu == 0)
                pt += h;
            else
                ps += h;
        }
}

// Spatial and temporal fixed-point sums of the plaquettes with corner at the two
// sites of x1 pair j (L1 is even: both lie in one row, have opposite parities and
// index j within them), added to ps and pt; FP32 products.  The second site's own
// links are the first site's forward links along x1, so the pair takes 29 link
// loads instead of 32; the steps along the other directions are shared, and one
// thread carries two independent chains of products.
template <int LD>
__device__ __forceinline__ void su2_pair_plaquettes(const float4 *U, const Su2Chain &ch, uint32_t j, long long &ps,
                                                    long long &pt)
{
    uint32_t x1h;
    const LinkSite x = link_pair(ch, j, x1h);
    const LinkSite y = link_of_pair(ch, x, x1h, 1u);
    const int p0 = (int)x.par, p1 = 1 - p0;
    const uint32_t f0 = x.o + x.fw[0], f1 = x.o + y.fw[1], f2 = x.o + x.fw[2], f3 = x.o + x.fw[3];
    float4 U0[4], U1[4], F0[4][4], F1[4][4]; // F0[mu][nu] = U_nu(x + mu), F1[mu][nu] = U_nu(y + mu)
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
        U0[mu] = link_at<LD>(U, ch, p0, mu, x.o);
        U1[mu] = link_at<LD>(U, ch, p1, mu, x.o);
    }
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
        F0[1][nu] = U1[nu];
        if (nu != 0) F0[0][nu] = link_at<LD>(U, ch, p1, nu, f0);
        if (nu != 2) F0[2][nu] = link_at<LD>(U, ch, p1, nu, f2);
        if (nu != 3) F0[3][nu] = link_at<LD>(U, ch, p1, nu, f3);
        if (nu != 0) F1[0][nu] = link_at<LD>(U, ch, p0, nu, f0);
        if (nu != 1) F1[1][nu] = link_at<LD>(U, ch, p0, nu, f1);
        if (nu != 2) F1[2][nu] = link_at<LD>(U, ch, p0, nu, f2);
        if (nu != 3) F1[3][nu] = link_at<LD>(U, ch, p0, nu, f3);
    }
    plaquettes_of(U0, F0, ps, pt);
    plaquettes_of(U1, F1, ps, pt);
}

}  // namespace
}  // namespace mc
