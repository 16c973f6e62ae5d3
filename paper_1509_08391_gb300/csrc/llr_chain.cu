// llr_chain.cu -- the window-restricted Monte Carlo of 4-D compact U(1) on
// sm_103a: checkerboard staple sums, heat-bath and overrelaxation proposals,
// the sequential window-accept scan, the fresh energy and the Robbins-Monro
// update, for a batch of independent (interval, replica) lattices.
//
// Paper: Langfeld, Lucini, Pellegrini, Rago (arXiv:1509.08391).
//   Sec. 3.1      action E = sum_P cos(theta_P), plaquette angle
//                 theta_munu(x) = theta_mu(x) + theta_nu(x+mu) - theta_mu(x+nu) - theta_nu(x)
//   eqs. (2.13)-(2.16) weight exp(-a E) on the closed window [E_lo, E_lo + dE],
//                 dE_meas = E - E_lo - dE/2
//   Algorithm 1   n_therm + n_meas sweeps, measure after n_therm
//   eq. (2.30)      a <- a + 12 <<dE>> / (dE^2 (n + 1))
//
// Design
//   * Links are float32 angles, SoA by (direction, site parity), sites of a
//     parity in lexicographic order: theta[off + (2 mu + p) * V/2 + s/2].
//   * One persistent kernel, one CTA of 768 threads per SM (80 registers a
//     thread).  Work items are (composite sweep j, group of up to `teams`
//     lattices); a CTA takes the next item from an atomic counter, waits
//     (bounded) until sweep j-1 of that group is done, and owns its lattices for
//     that sweep.  Items run sweep-major, so uneven lattice sizes balance
//     across SMs.  The lattices of an item advance together, phase by phase
//     (heat-bath pass, overrelaxation passes, energy).
//   * Lattices per item (choose_teams, by the time the launch takes): with fewer
//     lattices than SMs, one with all 24 warps; with many, three with 8 warps
//     each or four with 6 in the heat-bath pass, whose deciding warps are serial
//     and need company, while the overrelaxation pass takes up to three together,
//     or one after another where a slab fills the shared memory; six of L <= 6.
//     Lattices of an uneven batch are taken by falling side, so like ones meet.
//   * A heat-bath pass runs class by class over the whole lattice (one
//     pipeline drain per class); an overrelaxation pass is slab-major: for
//     each x3 slab, all 8 checkerboard classes of that slab in order.
//   * In a heat-bath pass the warps of a lattice are specialised: producer warps
//     build the staples of two links per thread from their neighbour angles,
//     draw the von Mises proposals (Best & Fisher 1979), evaluate their dE from
//     the stored new angle exactly as the old local energy is evaluated,
//     convert dE to int64 fixed point (2^-32) and form prefix sums over a warp's
//     64 links; a consumer warp walks the chunks in link order and decides
//     each block of B links with the restricted Metropolis rule
//     dist(E + dE_block) <= dist(E), using a ballot to find the first rejected
//     block among those of 32 speculatively accepted links, and publishes the
//     accepted links; the producers write their angles.  Chunks pass through a ring of
//     1 or 2 stages in shared memory guarded by named barriers, so proposals
//     for later chunks overlap with the scan of earlier ones.
//   * The multicanonical pass (Sec. 2.6) has the same producers at a fixed
//     proposal slope; its consumer replaces the window rule by a
//     Metropolis-Hastings test for the weight 1/rho~ in the same
//     speculative scan.
//   * Overrelaxation (theta' = -theta - 2 alpha) conserves E exactly, so its
//     passes skip the scan: threads reflect links, neighbours read from the
//     slab in shared memory, and write them directly.
//   * Lattices of L <= 10 that fit are held in shared memory for the whole sweep.
//   * Every sum of products on the way to an angle, a dE or a decision has its
//     fused operations written out, so every program (batched sweeps, single
//     passes, the plain form), launch shape and build gives bit-identical chains.
//   * After 1 + n_or passes the 6V plaquettes are summed (float32 angles
//     summed exactly as hi + lo, their unbiased cosine in packed arithmetic,
//     fixed-point accumulation) and the tracked energy is resynchronised.
//
// Measured (GB300, 2070 MHz; one pass of 456 lattices of L = 20, ms, before ->
// now): heat-bath 10.1 -> 7.4 (797 -> 628 instructions per link), overrelaxation
// 2.7 -> 1.9 (184 -> 120), energy 1.3 -> 0.97, against one CTA of 256 threads per
// lattice and one link per thread.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "llr_internal.h"

namespace llr {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// Best & Fisher (1979) von Mises sampler, density ~ exp(kappa cos X).
// tau = 1 + sqrt(1 + 4 k^2), rho = (tau - sqrt(2 tau)) / (2 k) (rewritten
// without cancellation), r = (1 + rho^2) / (2 rho).  Attempt t uses Philox
// call t/2 (counter word 3), words 0-1 (t even) or 2-3 (t odd) as u1, u2,
// and the lowest bit of the first of them as the sign of X:
// z = cos(pi u1), f = (1 + r z) / (r + z), c = k (r - f); accept if
// c (2 - c) > u2 or ln(c / u2) + 1 - c >= 0 (evaluated as
// log2 c - log2 u2 >= (c - 1) / ln 2).  The accept test runs on fast
// hardware approximations (it only decides which attempt is taken); the
// accepted variate is then evaluated without cancellation as (cos X, sin X),
// X = +-acos f: with sh, ch = sin, cos(pi u1 / 2) (hardware sine/cosine,
// absolute error ~5e-7 on [0, pi/2]), z = ch^2 - sh^2 and
//   1 - f = (r - 1) 2 sh^2 / (r + z)   (f >= 0),   1 + f = (r + 1) 2 ch^2 / (r + z)   (f < 0),
// so w = 1 -+ f has no cancellation, cos X = +-(1 - w) and
// |sin X| = sqrt(w (2 - w)) keep the angle's absolute accuracy near X = 0
// and X = pi.
// ---------------------------------------------------------------------------
struct VonMises {
    float k, r, rm1;   // |kappa|, r, r - 1
    __device__ __forceinline__ explicit VonMises(float kappa)
    {
        k = fabsf(kappa);
        const float sq = sqrt_fast(fmaf(4.0f * k, k, 1.0f));
        const float tau = 1.0f + sq;
        const float rho =
            __fdividef(2.0f * k * tau, (sq + 1.0f) * (tau + sqrt_fast(2.0f * tau)));
        r = __fdividef(fmaf(rho, rho, 1.0f), 2.0f * rho);
        const float omr = 1.0f - rho;
        rm1 = __fdividef(omr * omr, 2.0f * rho);
    }
    // the accept test of one attempt (cheap form only, so lanes that accept at
    // different attempts diverge over as little code as possible)
    __device__ __forceinline__ bool accepts(uint32_t wa, uint32_t wb) const
    {
        const float u1 = u01(wa), u2 = u01(wb);
        const float z = __cosf(kPi * u1);
        const float f = __fdividef(fmaf(r, z, 1.0f), r + z);
        const float c = __fmul_rn(k, rm1 + (1.0f - f));
        const bool quick = fmaf(c, 2.0f - c, -u2) > 0.0f;
        // second test ln(c / u2) + 1 - c >= 0, in base 2 (no branch around it: the
        // lanes of a warp rarely agree)
        const bool full =
            __log2f(c) - __log2f(u2) >= __fmul_rn(c - 1.0f, 1.4426950408889634f);
        return quick | full;
    }
    // the two attempts of one Philox call: the first that accepts, its word 0
    __device__ __forceinline__ bool attempts(const U4 &w, uint32_t &w_acc) const
    {
        const bool first = accepts(w.x, w.y), second = accepts(w.z, w.w);
        w_acc = first ? w.x : w.z;
        return first | second;
    }
    // (cos X, sin X) of the accepted attempt, without cancellation
    __device__ __forceinline__ void evaluate(float kappa, uint32_t w_acc, float &cX,
                                             float &sX) const
    {
        const float u1 = u01(w_acc);
        float sh, ch;
        __sincosf(0.5f * kPi * u1, &sh, &ch);
        const float z = __fmul_rn(ch - sh, ch + sh);
        const float den = __fadd_rn(r, z);
        const bool pos = fmaf(r, z, 1.0f) >= 0.0f;               // f >= 0
        const float w = __fdividef(pos ? rm1 * 2.0f * sh * sh : (r + 1.0f) * 2.0f * ch * ch, den);
        const float s = sqrt_fast(w * (2.0f - w));
        const float c = pos ? 1.0f - w : w - 1.0f;
        const bool neg_x = !(w_acc & 1u);                        // X = -acos f
        const bool flip = kappa < 0.0f;                          // X -> X + pi
        cX = flip ? -c : c;
        sX = (neg_x != flip) ? -s : s;
    }
};

constexpr float kKappaFlat = 1e-6f;   // below it X is drawn uniformly

__device__ __forceinline__ void uniform_angle(const U4 &w, float &cX, float &sX)
{
    const float t = 2.0f * u01(w.x) - 1.0f;   // X = pi t
    sincospif(t, &sX, &cX);
}

// The von Mises variates of a thread's two links: one Philox call each, then
// further calls one at a time for a link that has not accepted, the first
// link's before the second's.  A warp's lanes rarely all accept at the first
// call (91 % do), so for two links the later calls, which cost the warp the same
// however many lanes take part, are shared: 3.6 calls for 64 links where one link
// at a time took 2.2 for 32.  ok: found within the attempt limit.
__device__ __forceinline__ void von_mises2(float kappa0, float kappa1, uint32_t link0,
                                           uint32_t link1, uint32_t sweep, uint32_t tag,
                                           uint32_t k0, uint32_t k1, float2 &cX, float2 &sX,
                                           bool &ok0, bool &ok1)
{
    const VonMises v0(kappa0), v1(kappa1);
    const bool flat0 = fabsf(kappa0) < kKappaFlat, flat1 = fabsf(kappa1) < kKappaFlat;
    const U4 w0 = philox4x32_10(link0, sweep, tag, 0u, k0, k1);
    const U4 w1 = philox4x32_10(link1, sweep, tag, 0u, k0, k1);
    uint32_t acc0, acc1;
    ok0 = v0.attempts(w0, acc0) || flat0;
    ok1 = v1.attempts(w1, acc1) || flat1;
    bool done0 = ok0, done1 = ok1;
    for (uint32_t n = 1; !(done0 && done1);) {
        VonMises v = v0;
        uint32_t link = link0;
        if (done0) {
            v = v1;
            link = link1;
        }
        const U4 w = philox4x32_10(link, sweep, tag, n, k0, k1);
        uint32_t acc;
        const bool found = v.attempts(w, acc);
        ++n;
        const bool last = n >= kSamplerMaxAttempts / 2;
        if (!done0) {
            if (found) acc0 = acc;
            ok0 = found;
            done0 = found || last;
            if (done0) n = 1;
        } else {
            if (found) acc1 = acc;
            ok1 = found;
            done1 = found || last;
        }
    }
    v0.evaluate(kappa0, acc0, cX.x, sX.x);
    v1.evaluate(kappa1, acc1, cX.y, sX.y);
    if (flat0) uniform_angle(w0, cX.x, sX.x);
    if (flat1) uniform_angle(w1, cX.y, sX.y);
}

template <bool FAST>
__device__ __forceinline__ void sin_cos(float x, float *s, float *c)
{
    if (FAST)
        __sincosf(x, s, c);
    else
        sincosf(x, s, c);
}

// arg(x + i y): the polynomial arctangent with fast math, the library's
// atan2f without.
template <bool FAST>
__device__ __forceinline__ float arg(float y, float x)
{
    return FAST ? arg_fast(y, x) : atan2f(y, x);
}

// arg of two vectors, each bit for bit as by arg: the polynomial of arg_fast in
// packed arithmetic.
template <bool FAST>
__device__ __forceinline__ float2 arg2(float2 y, float2 x)
{
    if (!FAST) return make_float2(atan2f(y.x, x.x), atan2f(y.y, x.y));
    return arg_fast2(y, x);
}

// Local energy Re(e^{i theta} S) of a link from (cos, sin) of its angle.  Here
// and in the heat-bath's other sums of products the fused operation is
// written out, so every place and build that forms them rounds alike.
__device__ __forceinline__ float link_energy(float c, float s, float Sr, float Si)
{
    return fmaf(c, Sr, -__fmul_rn(s, Si));
}

// Coordinates of the h-th site of parity p (lexicographic, x0 fastest).
__device__ __forceinline__ int decode_half(int h, int p, int L, uint32_t magic, int x[4])
{
    const int n = 2 * h;
    const int q = (int)__umulhi((uint32_t)n, magic);
    const int x0e = n - q * L;
    const int q2 = (int)__umulhi((uint32_t)q, magic);
    x[1] = q - q2 * L;
    const int q3 = (int)__umulhi((uint32_t)q2, magic);
    x[2] = q2 - q3 * L;
    x[3] = q3;
    const int b = (p + x[1] + x[2] + x[3]) & 1;
    x[0] = x0e + b;
    return n + b;
}

// Staple sum S = sum_j exp(i phi_j) of link theta_MU(x), x of parity p:
// forward  phi = theta_nu(x+mu) - theta_mu(x+nu) - theta_nu(x)
// backward phi = theta_nu(x-nu) - theta_nu(x-nu+mu) - theta_mu(x-nu)
// so that the link's local energy is sum_j cos(theta + phi_j) = Re(e^{i theta} S).
//
// In a heat-bath pass a producer thread proposes for two links at a time, half
// sites h and h + 1 (h even), so index arithmetic, the sampler's later calls
// and the prefix sums serve two, and the staples are summed in packed
// arithmetic.  With rows of even length (ROW) both lie in one x0 row and share
// their neighbours' rows: 14 of the 18 neighbour pairs are one 8-byte access.
// The neighbour angles are copied asynchronously (cp.async, cached in L1) to
// the thread's own column of a stage buffer while it works on the pair before,
// or, where the whole lattice is in shared memory (RES), read there.  A thread
// only reads what it copied itself, so cp.async.wait_group is the only
// synchronisation.  The copies read through L1 like plain loads: other classes
// of this lattice were written earlier in the same launch (same CTA, or
// another CTA before the acquire of the lattice's done counter).
constexpr int kStaged = 19;   // pairs in a stage column: 18 neighbours and the links themselves

__device__ __forceinline__ void cp_async16(float *dst, const float *src)   // through L2 only
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void cp_async(float *dst, const float *src)   // through L1
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(BYTES)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The two links of a thread (half sites h, h + 1 of parity p): sites and the
// half-site distances to the neighbours x +- nu.
template <bool ROW>
struct LinkPair {
    int up0[4], dn0[4], up1[4], dn1[4];   // ROW: up1, dn1 differ from up0, dn0 in [0] only
    int site0, site1;

    static __device__ __forceinline__ int around(int h, int p, int L, uint32_t magic, int up[4],
                                                 int dn[4])
    {
        int x[4];
        const int site = decode_half(h, p, L, magic, x);
        const int Lh = L >> 1, S1 = L * Lh, S = S1 * L;
        const bool odd = x[0] & 1;
        up[0] = odd ? (x[0] == L - 1 ? 1 - Lh : 1) : 0;
        dn[0] = odd ? 0 : (x[0] == 0 ? Lh - 1 : -1);
        up[1] = x[1] == L - 1 ? Lh - S1 : Lh;
        dn[1] = x[1] == 0 ? S1 - Lh : -Lh;
        up[2] = x[2] == L - 1 ? S1 - S : S1;
        dn[2] = x[2] == 0 ? S - S1 : -S1;
        up[3] = x[3] == L - 1 ? S - S * L : S;
        dn[3] = x[3] == 0 ? S * L - S : -S;
        return site;
    }

    __device__ __forceinline__ LinkPair(int h, int p, int L, uint32_t magic)
    {
        site0 = around(h, p, L, magic, up0, dn0);
        if (ROW) {
            // the second link, at x0 + 2: never at the start of the row
            const bool odd = site0 & 1;
            const int Lh = L >> 1;
            const int k = h - (int)__umulhi(2u * (uint32_t)h, magic) * Lh;   // position in the row
            site1 = site0 + 2;
#pragma unroll
            for (int nu = 1; nu < 4; ++nu) {
                up1[nu] = up0[nu];
                dn1[nu] = dn0[nu];
            }
            up1[0] = odd ? (k + 2 == Lh ? 1 - Lh : 1) : 0;
            dn1[0] = odd ? 0 : -1;
        } else {
            site1 = around(h + 1, p, L, magic, up1, dn1);
        }
    }
};

// The 18 neighbour pairs of the staples of theta_MU at half site h, h + 1 and
// the pair itself, in the order of the staple sum, each handed to
// put(k, aligned, o0, o1): pair k at offsets o0, o1 of the lattice, adjacent and
// 8-byte aligned if `aligned`.
template <int MU, bool ROW, class Put>
__device__ __forceinline__ void neighbour_pairs(const LinkPair<ROW> &n, int half, int h, int p,
                                                Put put)
{
    const int q = p ^ 1;
    int k = 0;
    auto at = [&](int nu, int par, bool x0, int d0, int d1) {
        const int o = (2 * nu + par) * half + h;
        put(k++, ROW && !x0, o + d0, o + 1 + d1);
    };
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == MU) continue;
        at(nu, q, MU == 0, n.up0[MU], n.up1[MU]);                       // theta_nu(x+mu)
        at(MU, q, nu == 0, n.up0[nu], n.up1[nu]);                       // theta_mu(x+nu)
        at(nu, p, false, 0, 0);                                         // theta_nu(x)
        at(nu, p, MU == 0 || nu == 0, n.dn0[nu] + n.up0[MU], n.dn1[nu] + n.up1[MU]);
        at(MU, q, nu == 0, n.dn0[nu], n.dn1[nu]);                       // theta_mu(x-nu)
        at(nu, q, nu == 0, n.dn0[nu], n.dn1[nu]);                       // theta_nu(x-nu)
    }
    at(MU, p, false, 0, 0);
}

// Staple sums of two links from their neighbour pairs v(0 .. 17).
template <bool FAST, class Get>
__device__ __forceinline__ void staple_sums2(Get v, float2 &Sr, float2 &Si)
{
    Sr = Si = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float2 pf = sub2(sub2(v(6 * j), v(6 * j + 1)), v(6 * j + 2));
        const float2 pb = sub2(sub2(v(6 * j + 5), v(6 * j + 3)), v(6 * j + 4));
        float2 sf, cf, sb, cb;
        sin_cos<FAST>(pf.x, &sf.x, &cf.x);
        sin_cos<FAST>(pf.y, &sf.y, &cf.y);
        sin_cos<FAST>(pb.x, &sb.x, &cb.x);
        sin_cos<FAST>(pb.y, &sb.y, &cb.y);
        Sr = add2(Sr, add2(cf, cb));
        Si = add2(Si, add2(sf, sb));
    }
}

// Threads of the sweep kernel's CTA (one CTA per SM, 80 registers a thread) and
// the lattices one CTA works on at a time, each with a team of warps.
constexpr int kThreads = 768, kWarps = kThreads / 32, kMaxTeams = 6;

// Most producer warps of a lattice's heat-bath team, which are the 64-link groups of
// a ring stage: one warp decides, and for a lone lattice, where that warp is the
// bound, it has a quarter of the SM (a scheduler) to itself.
__host__ __device__ constexpr int producers(int teams)
{
    return teams == 1 ? kWarps / 4 * 3 : kWarps / teams - 1;
}

// Dynamic shared memory: the whole lattices where they fit (RES; then the
// heat-bath rings), otherwise used by one phase of a sweep at a time: the
// heat-bath pass's stage columns (kStaged pairs per thread) and rings, or the
// slabs of the overrelaxation pass.
extern __shared__ __align__(16) float g_dyn[];

__device__ __forceinline__ float2 *stage_col()
{
    return (float2 *)g_dyn + threadIdx.x;   // pair k at [k * kThreads]
}

// Barrier 0 is __syncthreads.  In a heat-bath pass the ring stages of team k use
// the 2 D barriers from 1 + 2 D k (full, then empty; the first also ends a
// class); in the other phases team k has barriers 1 + k and 8 + k.
__device__ __forceinline__ void bar_sync(int id, int n)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// The value of lane 0, which the compiler then knows to be the same in all lanes.
__device__ __forceinline__ int uniform(int v)
{
    return __shfl_sync(kFull, v, 0);
}

// The warps of the CTA that work on one lattice in a phase: warp w of nw,
// thread tid of nt, a barrier of their own.
struct Team {
    int w, nw, tid, nt, bar;
    __device__ __forceinline__ void sync() const { bar_sync(bar, nt); }
};

// One ring stage of a heat-bath class: a chunk of `groups` 64-link groups, two
// links per producer lane.
struct Stage {
    long long *P;      // prefix sums of dE over the group, to each of its links
    long long *d;      // dE of each link
    float2 *thn;       // the proposals
    float2 *u;         // multicanonical pass: the uniforms of the accept test
    uint2 *acc;        // written by the consumer: links 0-31 / 32-63 accepted
};

// Bytes of a stage per group: a multiple of 16, so every stage's P is aligned.
constexpr int kStageGroupBytes = 64 * 24 + 16;

__device__ __forceinline__ Stage stage_at(char *base, int groups, int s)
{
    char *p = base + (size_t)s * groups * kStageGroupBytes;
    Stage g;
    g.P = (long long *)p;
    g.d = (long long *)(p + groups * 512);
    g.thn = (float2 *)(p + groups * 1024);
    g.u = (float2 *)(p + groups * 1280);
    g.acc = (uint2 *)(p + groups * 1536);
    return g;
}

// Heat-bath team: nw warps on the lattice, warp cw of them the consumer; its
// ring of D stages of nw - 1 groups at `ring` (floats) of g_dyn, and the first
// of its 2 D ring barriers.
struct HbTeam {
    int nw, cw, ring, D, full;
};

struct Smem {
    LatState st[kMaxTeams];
    unsigned long long acc_cnt[kMaxTeams];
    unsigned long long cap_cnt[kMaxTeams];
    long long red[kWarps];
    HbTeam hb[kMaxTeams];     // the teams of a heat-bath pass
    float a_f[kMaxTeams];     // slope of the team's heat-bath proposals
    int active[kMaxTeams];    // the team's lattice takes part in the sweep
    int n_app[kMaxTeams];     // approach: sweeps done
    int item_first, item_n, item_j, item_state;
};

// Producer side of one heat-bath class (MU, p): proposals and warp prefix
// sums, chunk by chunk, into the stage ring (slope a_f, Philox tag `tag`).
// When a slot comes back from the consumer (and for the last chunks at the
// end of the class) each producer writes those of its proposals that were
// accepted.  th: the lattice (RES: at offset lat_off of g_dyn instead).
//
// The team's and the lattice's constants are read from shared memory where they
// are used: kept in registers across the loop they would be spilled.
template <int MU, bool ROW, bool RES, bool MUCA, bool FAST>
__device__ __noinline__ void produce_class(Smem &sm, int slot, int pw, float *th_, int lat_off,
                                           int p, uint32_t tag)
{
    const int lane = threadIdx.x & 31, pt = pw * 32 + lane;
    const LatState &st = sm.st[slot];
    const HbTeam &hb = sm.hb[slot];
    const int CH = (hb.nw - 1) * 64;
    float *th = RES ? g_dyn + lat_off : th_;
    unsigned cnt = 0;
    auto stage = [&](int s) { return stage_at((char *)(g_dyn + hb.ring), hb.nw - 1, s); };
    // write back chunk c of a slot the consumer has released
    auto flush = [&](const Stage &stg, int c) {
        const int h = c * CH + 2 * pt, half = st.half;
        if (h < half) {   // half is even: both links or none
            float *own = th + (2 * MU + p) * half;
            const uint2 acc = stg.acc[pw];
            const unsigned took = (lane < 16 ? acc.x : acc.y) >> (2 * (lane & 15));
            const float2 t = stg.thn[pt];
            if (took & 1u) {
                own[h] = t.x;
                ++cnt;
            }
            if (took & 2u) {
                own[h + 1] = t.y;
                ++cnt;
            }
        }
    };
    auto fetch = [&](int h) {
        const LinkPair<ROW> n(h, p, st.L, st.magic);
        float2 *col = stage_col();
        neighbour_pairs<MU, ROW>(n, st.half, h, p, [&](int k, bool aligned, int o0, int o1) {
            float *dst = (float *)(col + k * kThreads);
            if (aligned) {
                cp_async<8>(dst, th + (unsigned)o0);
            } else {
                cp_async<4>(dst, th + (unsigned)o0);
                cp_async<4>(dst + 1, th + (unsigned)o1);
            }
        });
    };
    if (!RES) {
        if (2 * pt < st.half) fetch(2 * pt);
        cp_async_commit();
    }
    int ch = 0;
#pragma unroll 1
    for (; ch * CH < st.half; ++ch) {
        const int h = ch * CH + 2 * pt;
        const bool valid = h < st.half;
        float2 thn = make_float2(0.0f, 0.0f);
        long long d0 = 0, d1 = 0;
        float2 Sr, Si, t0;
        if (!RES) cp_async_wait<0>();
        if (valid) {
            if (RES) {
                const LinkPair<ROW> n(h, p, st.L, st.magic);
                float2 v[kStaged];
                neighbour_pairs<MU, ROW>(n, st.half, h, p, [&](int k, bool aligned, int o0, int o1) {
                    v[k] = aligned ? *(const float2 *)(th + o0) : make_float2(th[o0], th[o1]);
                });
                staple_sums2<FAST>([&](int k) { return v[k]; }, Sr, Si);
                t0 = v[18];
            } else {
                const float2 *col = stage_col();
                staple_sums2<FAST>([&](int k) { return col[k * kThreads]; }, Sr, Si);
                t0 = col[18 * kThreads];
            }
        }
        // the next pair's neighbours, on their way while this one is sampled
        if (!RES) {
            if (h + CH < st.half) fetch(h + CH);
            cp_async_commit();
        }
        if (valid) {
            float s0, c0, s1, c1;
            sin_cos<FAST>(t0.x, &s0, &c0);
            sin_cos<FAST>(t0.y, &s1, &c1);
            // the old local energies |S| cos(theta + alpha)
            const float e0 = link_energy(c0, s0, Sr.x, Si.x), e1 = link_energy(c1, s1, Sr.y, Si.y);
            const float S0 = sqrt_fast(fmaf(Si.x, Si.x, __fmul_rn(Sr.x, Sr.x)));
            const float S1 = sqrt_fast(fmaf(Si.y, Si.y, __fmul_rn(Sr.y, Sr.y)));
            int x[4];
            const uint32_t base = (uint32_t)MU * 2u * (uint32_t)st.half;
            const uint32_t l0 = base + (uint32_t)decode_half(h, p, st.L, st.magic, x);
            const uint32_t l1 =
                ROW ? l0 + 2u : base + (uint32_t)decode_half(h + 1, p, st.L, st.magic, x);
            float2 cX, sX;
            bool ok0, ok1;
            const float a_f = sm.a_f[slot];
            von_mises2(-a_f * S0, -a_f * S1, l0, l1, st.sweep, tag, st.key0, st.key1, cX, sX, ok0,
                       ok1);
            // theta' = X - alpha, alpha = arg S: e^{i theta'} = e^{iX} conj(S) / |S|
            thn = arg2<FAST>(make_float2(fmaf(sX.x, Sr.x, -__fmul_rn(cX.x, Si.x)),
                                         fmaf(sX.y, Sr.y, -__fmul_rn(cX.y, Si.y))),
                             make_float2(fmaf(cX.x, Sr.x, __fmul_rn(sX.x, Si.x)),
                                         fmaf(cX.y, Sr.y, __fmul_rn(sX.y, Si.y))));
            // dE of the angle actually stored, evaluated exactly like the old
            // energy (same staple sum, same sine/cosine): the approximation
            // errors of one link's successive evaluations then cancel along its
            // chain of updates and leave only random noise.  Taking
            // |S| cos X instead carried a systematic -3.5e-8 per move (the
            // rounded atan2 and (cos X, sin X) are not exactly the angle
            // X - alpha), which drifted the running energy by -4.8e-4 per
            // heat-bath pass at L = 8 and shifted the window it enforces.
            sin_cos<FAST>(thn.x, &s0, &c0);
            sin_cos<FAST>(thn.y, &s1, &c1);
            d0 = to_fx(__fsub_rn(link_energy(c0, s0, Sr.x, Si.x), e0));
            d1 = to_fx(__fsub_rn(link_energy(c1, s1, Sr.y, Si.y), e1));
            if (!(ok0 && ok1)) {
                if (!ok0) {
                    thn.x = t0.x;
                    d0 = 0;
                }
                if (!ok1) {
                    thn.y = t0.y;
                    d1 = 0;
                }
                atomicAdd(&sm.cap_cnt[slot], (unsigned long long)(!ok0 + !ok1));
            }
        }
        __syncwarp();
        long long P = d0 + d1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(kFull, P, o);
            if (lane >= o) P += y;
        }
        const int D = hb.D, s = ch & (D - 1), bar = hb.full + s, NT = hb.nw * 32;
        const Stage stg = stage(s);
        if (ch >= D) {
            bar_sync(bar + D, NT);
            flush(stg, ch - D);
        }
        stg.thn[pt] = thn;
        if (MUCA && valid) {   // the uniforms of the links' accept tests
            int x[4];
            const uint32_t base = (uint32_t)MU * 2u * (uint32_t)st.half;
            const uint32_t l0 = base + (uint32_t)decode_half(h, p, st.L, st.magic, x);
            const uint32_t l1 =
                ROW ? l0 + 2u : base + (uint32_t)decode_half(h + 1, p, st.L, st.magic, x);
            stg.u[pt] = make_float2(
                u01(philox4x32_10(l0, st.sweep, kTagMuca, 0u, st.key0, st.key1).x),
                u01(philox4x32_10(l1, st.sweep, kTagMuca, 0u, st.key0, st.key1).x));
        }
        ((longlong2 *)stg.P)[pt] = make_longlong2(P - d1, P);
        ((longlong2 *)stg.d)[pt] = make_longlong2(d0, d1);
        bar_arrive(bar, NT);
    }
    const int D = hb.D;
    for (int c = max(ch - D, 0); c < ch; ++c) {
        const int s = c & (D - 1);
        bar_sync(hb.full + D + s, hb.nw * 32);
        flush(stage(s), c);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(kFull, cnt, o);
    if (lane == 0) atomicAdd(&sm.acc_cnt[slot], (unsigned long long)cnt);
}

// Neighbour angles of link theta_MU(x) (site s, parity p) loaded straight into
// registers v[18], in the order of neighbour_pairs.
template <int MU>
__device__ __forceinline__ void staple_load(const float *th, int half, int L, const int x[4],
                                            int s, int p, float v[18])
{
    const int st[4] = {1, L, L * L, L * L * L};
    const int dmu = (x[MU] == L - 1) ? -(L - 1) * st[MU] : st[MU];
    const int spmu = s + dmu;
    const int q = p ^ 1;
    const float *thmu_q = th + (2 * MU + q) * half;
    int j = 0;
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == MU) continue;
        const int dnf = (x[nu] == L - 1) ? -(L - 1) * st[nu] : st[nu];
        const int dnb = (x[nu] == 0) ? (L - 1) * st[nu] : -st[nu];
        const int spnu = s + dnf;
        const int smnu = s + dnb;
        const int smnu_pmu = smnu + dmu;
        const float *thnu_p = th + (2 * nu + p) * half;
        const float *thnu_q = th + (2 * nu + q) * half;
        v[6 * j + 0] = thnu_q[spmu >> 1];
        v[6 * j + 1] = thmu_q[spnu >> 1];
        v[6 * j + 2] = thnu_p[s >> 1];
        v[6 * j + 3] = thnu_p[smnu_pmu >> 1];
        v[6 * j + 4] = thmu_q[smnu >> 1];
        v[6 * j + 5] = thnu_q[smnu >> 1];
        ++j;
    }
}

// Staple sum of one link from its 18 neighbour angles, formed exactly as in
// staple_sums2.
template <bool FAST>
__device__ __forceinline__ void staple_sum_regs(const float v[18], float &Sr, float &Si)
{
    Sr = 0.0f;
    Si = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float pf = v[6 * j] - v[6 * j + 1] - v[6 * j + 2];
        const float pb = v[6 * j + 5] - v[6 * j + 3] - v[6 * j + 4];
        float sf, cf, sb, cb;
        sin_cos<FAST>(pf, &sf, &cf);
        sin_cos<FAST>(pb, &sb, &cb);
        Sr += cf + cb;
        Si += sf + sb;
    }
}

// Overrelaxation and the window.  A reflection keeps the local energy
// |S| cos(theta + alpha) exactly; a move changes E only through float32
// rounding (the reflection axis alpha carries the staple sum's error, ~1e-6 /
// |S|, the stored angle its rounding), and its float32 dE estimate is as
// uncertain as that change.  So the running energy is not changed by
// overrelaxation, and a block of a group is taken iff E -- the running energy
// at the start of the group -- lies outside the window, or E + dE_block lies
// inside it (reading R19).  Every |dE| is below 2^-14 (a move whose float32
// estimate exceeds that is refused, a guard never expected to act), so while
// E is outside the window, or inside and farther than B * 2^-14 from both
// edges, every move is taken without evaluating a dE.
constexpr float kOrDeltaMax = 6.103515625e-05f;   // 2^-14
constexpr long long kOrDeltaMaxFx = 1ll << 18;
constexpr int kOrRefused = (int)0x80000000;

// theta' = -theta - 2 alpha of link theta_MU at half-site h of parity p, with
// alpha = arg S (S from the 18 neighbour angles, plain loads); optionally the
// float32 dE estimate in fixed point, evaluated like the heat-bath's: the local
// energy Re(e^{i theta} S) at the stored new angle minus at the old one, same
// staple sum, same sine/cosine (dfx = kOrRefused beyond the guard).
template <int MU, bool FAST, bool WITH_DE>
__device__ __forceinline__ float overrelax_link(const float *th, const float *own, int half, int L,
                                                uint32_t magic, int p, int h, int &dfx)
{
    float va[18];
    int x[4];
    const int site = decode_half(h, p, L, magic, x);
    staple_load<MU>(th, half, L, x, site, p, va);
    const float t0 = own[h];
    float Sr, Si;
    staple_sum_regs<FAST>(va, Sr, Si);
    const float tn = wrap_angle(-t0 - 2.0f * arg<FAST>(Si, Sr));
    if (WITH_DE) {
        float sn, cn, so, co;
        sin_cos<FAST>(tn, &sn, &cn);
        sin_cos<FAST>(t0, &so, &co);
        const float d = __fsub_rn(link_energy(cn, sn, Sr, Si), link_energy(co, so, Sr, Si));
        dfx = fabsf(d) <= kOrDeltaMax ? __float2int_rn(d * 4294967296.0f) : kOrRefused;
    }
    return tn;
}

// One overrelaxation group (the links of class (MU, p) with half-site index
// in [h0, h0 + count)) of a lattice with planes of more pairs than the team has
// threads: every thread reflects its links, neighbours by plain loads.
template <int MU, bool FAST>
__device__ __noinline__ void overrelax_class(const LatState &st, const Team &t, float *th, int p,
                                             int h0, int count)
{
    const int L = st.L, half = st.half;
    const uint32_t magic = st.magic;
    float *own = th + (2 * MU + p) * half;
    for (int local = t.tid; local < count; local += t.nt) {
        int dfx;
        own[h0 + local] =
            overrelax_link<MU, FAST, false>(th, own, half, L, magic, p, h0 + local, dfx);
    }
}

// Heat-bath window decisions of one group in link order, by the calling warp.
// Lane k holds Pk, the inclusive prefix sum of dE over the group's lanes 0..k;
// em marks the lanes that end a block (blocks of B lanes start at multiples
// of B).  A block is taken iff dist(E + dE_block) <=
// dist(E), dist the distance from the closed window (inside the window: iff
// the energy after the block is inside).  Returns the mask of taken block
// ends and advances E.
__device__ __forceinline__ unsigned window_scan_group(long long Pk, unsigned em, int B,
                                                      long long &E, long long lo, long long hi)
{
    const int lane = threadIdx.x & 31;
    unsigned rem = em, acc = 0u;
    // the sum of the block ending at this lane
    const int bstart = lane & ~(B - 1);
    const long long Pprev = __shfl_sync(kFull, Pk, bstart > 0 ? bstart - 1 : 0);
    const long long bk = Pk - (bstart > 0 ? Pprev : 0ll);
    if (em != 0u && E >= lo && E <= hi) {
        // Inside the window (the usual case, and E stays inside): a block is
        // taken iff lo - E <= Pk - R <= hi - E, R the sum of the blocks
        // refused so far.  Keep the bounds rlo = lo - E + R, rhi = hi - E + R;
        // a refusal at j adds its block sum bj.
        long long rlo = lo - E, rhi = hi - E;
        while (rem) {
            const bool mine = (rem >> lane) & 1u;
            const bool viol = mine && (Pk < rlo || Pk > rhi);
            const unsigned vm = __ballot_sync(kFull, viol);
            if (vm == 0u) {
                acc |= rem;
                break;
            }
            const int j = __ffs(vm) - 1;
            acc |= rem & ((1u << j) - 1u);
            const long long bj = __shfl_sync(kFull, bk, j);
            rlo += bj;
            rhi += bj;
            rem &= ~((2u << j) - 1u);
        }
        // E after the group = E + P_last - R = lo + P_last - rlo
        E = lo + __shfl_sync(kFull, Pk, 31 - __clz(em)) - rlo;
    } else {
        // Outside the window: every remaining block is decided as if the
        // earlier ones were taken; the first refusal (one ballot) fixes the
        // blocks before it, its dE is dropped and the rest is decided again.
        long long base = 0;
        while (rem) {
            const long long Ea = E + (Pk - base);
            const long long Eb = Ea - bk;
            const bool mine = (rem >> lane) & 1u;
            const bool ok = dist_fx(Ea, lo, hi) <= dist_fx(Eb, lo, hi);
            const unsigned vm = __ballot_sync(kFull, mine && !ok);
            if (vm == 0u) {
                const int last = 31 - __clz(rem);
                E += __shfl_sync(kFull, Pk, last) - base;
                acc |= rem;
                rem = 0u;
            } else {
                const int j = __ffs(vm) - 1;
                acc |= rem & ((1u << j) - 1u);
                const long long Pj = __shfl_sync(kFull, Pk, j);
                const long long bj = __shfl_sync(kFull, bk, j);
                E += (Pj - bj) - base;   // energy before the refused block
                base = Pj;               // skip its contribution
                rem &= ~((2u << j) - 1u);
            }
        }
    }
    return acc;
}

// One overrelaxation group whose running energy E is inside the window and
// within B * 2^-14 of an edge: every thread forms its links' moves and float32
// dE estimates;
// the blocks of B links (starting at the group's first link; a block lies in
// one warp) sum their dE with shuffles, and a block is taken iff E lies
// outside the window or E + dE_block inside it.  Decisions are independent of
// one another (E does not move), so no barrier is needed.  Returns the number
// of moves this thread took.
template <int MU, bool FAST>
__device__ __noinline__ int overrelax_class_near(const LatState &st, const Team &t, float *th,
                                                 int p, int h0, int count, int B, long long E)
{
    const int L = st.L, half = st.half;
    const uint32_t magic = st.magic;
    const long long lo = st.lo_fx, hi = st.hi_fx;
    const bool outside = E < lo || E > hi;
    float *own = th + (2 * MU + p) * half;
    int taken = 0;
    for (int c0 = 0; c0 < count; c0 += t.nt) {
        const int local = c0 + t.tid;
        const bool valid = local < count;
        int dfx = 0;
        float tn = 0.0f;
        bool ok = false;
        if (valid) {
            tn = overrelax_link<MU, FAST, true>(th, own, half, L, magic, p, h0 + local, dfx);
            ok = dfx != kOrRefused;
            if (!ok) dfx = 0;
        }
        long long d = dfx;   // the block's dE (lanes of one block are an aligned segment)
        for (int o = 1; o < B; o <<= 1) d += __shfl_xor_sync(kFull, d, o);
        const long long Eb = E + d;
        if (valid && ok && (outside || (Eb >= lo && Eb <= hi))) {
            own[h0 + local] = tn;
            ++taken;
        }
    }
    return taken;
}

// The same for 32 links with blocks of one link and the energy inside the window
// (the usual case; it stays inside).  This is the deciding warp's critical path,
// so it is short: the links run from lane 31 down (the first refusal is the
// highest bit of a ballot), lane k holds the dE d of its link and the sum P of the
// dE up to it; u is the energy before all links that P counts, less the dE refused
// among them, above the lower edge.  A link is taken iff the energy after it, u + P,
// is at most the width: one unsigned comparison.  Every undecided link is decided
// as if the ones before it were taken; the first refusal takes its dE out.  Lanes
// past the end of the class (d = 0) never refuse.  Returns the lanes refused.
__device__ __forceinline__ unsigned window_scan_inside(long long P, long long d, long long &u,
                                                       unsigned long long width)
{
    unsigned rem = kFull, refused = 0u;
    for (;;) {
        const unsigned m = __ballot_sync(kFull, (unsigned long long)(u + P) > width) & rem;
        if (m == 0u) break;
        const int j = 31 - __clz(m);
        u -= __shfl_sync(kFull, d, j);
        refused |= 1u << j;
        rem = (1u << j) - 1u;
    }
    return refused;
}

// The same wherever the energy is; `valid` marks the lanes that hold a link, and E
// is the energy before all links that P counts, less the dE refused among them.
__device__ __forceinline__ unsigned window_scan_links(long long P, long long d, unsigned valid,
                                                      long long &E, long long lo, long long hi)
{
    unsigned rem = valid, refused = 0u;
    const int lane = threadIdx.x & 31;
    const bool mine = (valid >> lane) & 1u;
    // Far outside, where even all moves towards the window together do not reach
    // it, a link is taken iff its move does not lead away.
    const long long E0 = E + __shfl_sync(kFull, P - d, 31);   // before the first link
    const bool below = E0 < lo, above = E0 > hi;
    const bool away = mine && (below ? d < 0 : d > 0);
    long long sum = mine && !away ? d : 0, drop = away ? d : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(kFull, sum, o);
        drop += __shfl_xor_sync(kFull, drop, o);
    }
    if ((below && E0 + sum < lo) || (above && E0 + sum > hi)) {
        E -= drop;
        return __ballot_sync(kFull, away);
    }
    // near an edge: as inside, with the rule in full
    for (;;) {
        const long long e = E + P;   // after the link
        const unsigned m =
            __ballot_sync(kFull, dist_fx(e, lo, hi) > dist_fx(e - d, lo, hi)) & rem;
        if (m == 0u) break;
        const int j = 31 - __clz(m);
        E -= __shfl_sync(kFull, d, j);
        refused |= 1u << j;
        rem = (1u << j) - 1u;
    }
    return refused;
}

// Consumer side: sequential Metropolis accept of the chunk's blocks in link
// order; publishes the accepted links of each group (the producers write the
// angles).  Runs in one of the team's warps.
__device__ __noinline__ void consume_class(LatState &st, const HbTeam &hb, int B)
{
    const int lane = threadIdx.x & 31, nwp = hb.nw - 1, D = hb.D, NT = hb.nw * 32;
    const int half = st.half, CH = nwp * 64, nchunk = (half + CH - 1) / CH;
    long long E = st.E_fx;
    const long long lo = st.lo_fx, hi = st.hi_fx;
    for (int ch = 0; ch < nchunk; ++ch) {
        const int s = ch & (D - 1);
        bar_sync(hb.full + s, NT);
        const Stage stg = stage_at((char *)(g_dyn + hb.ring), nwp, s);
        const int left = half - ch * CH;   // links of the class from this chunk on
        if (B == 1) {
            // 32 links at a time, the two halves of a group after another
            const int groups = min(nwp, (left + 63) >> 6);
            const long long *Pp = stg.P + 31 - lane, *dp = stg.d + 31 - lane;
            long long P0 = Pp[0], P1 = Pp[32], d0 = dp[0], d1 = dp[32], sum = stg.P[63];
            for (int g = 0; g < groups; ++g) {
                // the next group's, on their way during the scan
                const int nx = min(g + 1, groups - 1) * 64;
                const long long nP0 = Pp[nx], nP1 = Pp[nx + 32], nd0 = dp[nx], nd1 = dp[nx + 32],
                                nsum = stg.P[nx + 63];
                unsigned r0, r1;
                if (E >= lo && E <= hi) {
                    long long u = E - lo;
                    r0 = window_scan_inside(P0, d0, u, (unsigned long long)(hi - lo));
                    r1 = window_scan_inside(P1, d1, u, (unsigned long long)(hi - lo));
                    E = lo + u;
                } else {
                    const int n0 = min(32, left - g * 64), n1 = min(32, left - g * 64 - 32);
                    r0 = window_scan_links(P0, d0, kFull << (32 - n0), E, lo, hi);
                    r1 = n1 > 0 ? window_scan_links(P1, d1, kFull << (32 - n1), E, lo, hi) : 0u;
                }
                E += sum;
                if (lane == 0) stg.acc[g] = make_uint2(__brev(~r0), __brev(~r1));
                P0 = nP0, P1 = nP1, d0 = nd0, d1 = nd1, sum = nsum;
            }
        } else {
            for (int g = 0; g < nwp; ++g) {
                const int nl = min(64, left - g * 64) >> 1;   // lanes, two links each
                if (nl <= 0) break;
                // blocks of B links end at second links: blocks of B / 2 lanes
                const int Bl = B >> 1;
                const bool isend = lane < nl && ((lane & (Bl - 1)) == Bl - 1 || lane == nl - 1);
                const unsigned em = __ballot_sync(kFull, isend);
                const unsigned ends =
                    window_scan_group(stg.P[g * 64 + 2 * lane + 1], em, Bl, E, lo, hi);
                const int end = min(lane | (Bl - 1), nl - 1);   // of this lane's block
                const unsigned took = __ballot_sync(kFull, lane < nl && ((ends >> end) & 1u));
                const unsigned x = __ballot_sync(kFull, (took >> (lane >> 1)) & 1u);
                const unsigned y = __ballot_sync(kFull, (took >> (16 + (lane >> 1))) & 1u);
                if (lane == 0) stg.acc[g] = make_uint2(x, y);
            }
        }
        bar_arrive(hb.full + D + s, NT);
    }
    if (lane == 0) st.E_fx = E;
}

// ln rho~ of the multicanonical weight at the fixed-point energy E: the
// piecewise-linear function of eq. (2.10) on the table's intervals,
// continued with the first / last slope beyond them (Sec. 2.6, eq. (2.50)).
__device__ __forceinline__ double muca_lnrho(const KernelArgs &a, long long E_fx)
{
    const double E = (double)E_fx * kInvFx;
    int k = (int)floor((E - a.muca_e0) / a.muca_de);
    k = k < 0 ? 0 : (k > a.muca_n - 1 ? a.muca_n - 1 : k);
    return a.muca_lnr[k] + a.muca_a[k] * (E - (a.muca_e0 + (double)k * a.muca_de));
}

// The multicanonical accept test of one link: whether a move of dE d (fixed point)
// from the energy E is refused, i.e. not u < exp(x),
// x = a0 d - (ln rho~(E + d) - ln rho~(E)).
__device__ __forceinline__ bool muca_refuses(const KernelArgs &a, long long E, long long d, float u)
{
    const double x = a.muca_a0 * ((double)d * kInvFx) - (muca_lnrho(a, E + d) - muca_lnrho(a, E));
    return !((double)u < exp(x));
}

// The same in float32 where that is sure of the outcome: sure = false where u is
// within the error of exp(x).  E and E + d lie in interval k0 and k1 of the table
// (q0, q1 in units of its intervals); with at most one edge between them
//   x = (a0 - a[k0]) d - (a[k1] - a[k0]) (E + d - that edge).
// ln rho~ is continuous, so an energy rounded across an edge costs no more than
// the rounding of q (at most 3e-7 |q|) times de times the jump of the slope,
// which muca_jump bounds.  FP64 runs at 1/73 of the float32 rate: the exact test
// of every link made the deciding warp the pass's bound.
__device__ __forceinline__ bool muca_refuses_fast(const KernelArgs &a, long long E, long long d,
                                                  float u, bool &sure)
{
    const float inv = a.muca_inv_de;
    const float q0 = (float)(E - a.muca_e0_fx) * inv, q1 = (float)(E + d - a.muca_e0_fx) * inv;
    const int top = a.muca_n - 1;
    const int k0 = min(max((int)floorf(q0), 0), top), k1 = min(max((int)floorf(q1), 0), top);
    const double s0 = a.muca_a[k0];
    const float df = (float)d * (float)kInvFx;
    float x = (float)(a.muca_a0 - s0) * df;
    if (k1 != k0) x -= (float)(a.muca_a[k1] - s0) * ((q1 - (float)max(k0, k1)) * a.muca_de_f);
    const float err = 1e-6f * (a.muca_jump * (1.0f + fabsf(q0) + fabsf(q1)) + fabsf(x)) + 1e-7f;
    const float e = __expf(x);
    // 2 err bounds exp(err) - 1 up to 1.25 (a table that starts 1e9 below the energies,
    // where float32 places them to 32 only, has err in the thousands)
    sure = abs(k1 - k0) <= 1 && err < 1.0f &&
           fabsf(u - e) > e * (2.0f * err + 4e-6f * (1.0f + fabsf(x))) + 1e-7f;
    return !(u < e);
}

// Consumer side of a multicanonical heat-bath class (Sec. 2.6): the links
// are taken in link order by Metropolis-Hastings for the weight 1/rho~ with
// the proposal at slope a0, i.e. with probability
// min(1, exp(a0 dE - (ln rho~(E + dE) - ln rho~(E)))), E the running energy
// before the link; the uniform comes from Philox counter (link, sweep, 12, 0).
// 32 links at a time (half a 64-link group): speculatively every remaining
// link is decided as if all earlier ones were taken; the first refusal (one
// ballot) fixes the links before it, its dE is dropped and the rest is decided
// again.  Blocks of one link.
__device__ __noinline__ void consume_class_muca(LatState &st, const HbTeam &hb,
                                                const KernelArgs &args)
{
    const int lane = threadIdx.x & 31, nwp = hb.nw - 1, CH = nwp * 64, D = hb.D, NT = hb.nw * 32;
    const int half = st.half, nchunk = (half + CH - 1) / CH;
    long long E = st.E_fx;
    for (int ch = 0; ch < nchunk; ++ch) {
        const int s = ch & (D - 1);
        bar_sync(hb.full + s, NT);
        const Stage stg = stage_at((char *)(g_dyn + hb.ring), nwp, s);
        for (int g = 0; g < 2 * nwp; ++g) {
            const int nval = min(32, half - (ch * CH + g * 32));
            if (nval <= 0) break;
            const long long *Pg = stg.P + g * 32;
            // the prefix sums run over 64 links: take the first half's out of the second's
            const long long off = (g & 1) ? Pg[-1] : 0ll;
            const long long Pk = Pg[lane] - off, dk = stg.d[g * 32 + lane];
            const float u = ((const float *)stg.u)[g * 32 + lane];
            const unsigned em = kFull >> (32 - nval);
            unsigned rem = em, acc = 0u;
            long long R = 0;
            while (rem) {
                const long long Eb = E + (Pk - dk) - R;
                bool sure;
                bool refuse = muca_refuses_fast(args, Eb, dk, u, sure);
                if (!sure && ((rem >> lane) & 1u)) refuse = muca_refuses(args, Eb, dk, u);
                __syncwarp();
                const unsigned vm = __ballot_sync(kFull, refuse) & rem;
                if (vm == 0u) {
                    acc |= rem;
                    break;
                }
                const int j = __ffs(vm) - 1;
                acc |= rem & ((1u << j) - 1u);
                R += __shfl_sync(kFull, dk, j);
                rem &= ~((2u << j) - 1u);
            }
            E += __shfl_sync(kFull, Pk, nval - 1) - R;
            if (lane == 0) ((unsigned *)(stg.acc + (g >> 1)))[g & 1] = acc;
        }
        bar_arrive(hb.full + D + s, NT);
    }
    if (lane == 0) st.E_fx = E;
}

// ---------------------------------------------------------------------------
// Overrelaxation pass slab by slab, the current slab in shared memory where it fits.
//
// The pass goes slab by slab of x3, in each slab class by class, so every class
// reads the same 8 class arrays of the slab (4 L^3 angles) again: they are
// copied to shared memory once per slab (16 L^3 bytes, 128 KB at L = 20) and
// the classes read 13 to 14 of a link's 18 neighbours there; the others lie in
// the slabs before and after and are plain loads (neither slab changes during
// this one).  New angles go to shared memory and to global memory.  Slabs of
// L > 24 do not fit and are read in place, one lattice at a time (304 of L = 28: two
// sweeps 111 ms; link by link, two or three lattices at a time, 150 to 167 ms).
//
// A thread reflects two links at a time, so the index arithmetic and (with
// rows of even length, ROW) the loads serve two: links k, k + 1 of one x0 row
// (one 8-byte load each), or, where the half row L / 2 is odd, the links at x2
// and x2 + L / 2.  With ROW threads map to (x2 plane, x1, k) and step over planes,
// so only x2 changes from one unit of a thread to the next; planes of odd half
// rows fill a team's threads badly (196 of 256 at L = 14, four iterations where
// the units need three: 0.55 against 0.50 ms a pass of 456 lattices), so there a
// thread takes every nt-th unit.
// ---------------------------------------------------------------------------
constexpr int kSlabMaxL = 24;       // 16 * 24^3 bytes = 216 KB
constexpr int kResidentMaxL = 10;   // 16 * 10^4 bytes = 156 KB

struct SlabGeo {
    int L, Lh, S1, S, half, SH;   // side, half row, plane, slab, class array, half slab (floats)
    int step, nit, planes;        // planes (ROW) or units per iteration, iterations, planes in all
    uint32_t mL, mLh;             // magic divisors of the units (mLh = 0: by one)
    int x2, h;                    // the unit's plane (beyond all: idle) and link
    int d1p, d1m, rdn, rup, par;  // x1 neighbours, x0 wraps, parity of x1

    // the x1, k part of a unit's place
    __device__ __forceinline__ void place(bool row, int x1, int k)
    {
        h = x2 * S1 + x1 * Lh + k;
        d1p = x1 == L - 1 ? Lh - S1 : Lh;
        d1m = x1 == 0 ? S1 - Lh : -Lh;
        rdn = k == 0 ? Lh - 1 : -1;
        rup = row ? (k + 2 == Lh ? 2 - Lh : 2) : (k == Lh - 1 ? 1 - Lh : 1);
        par = x1 & 1;
    }
    // unit u of a slab's S / 2 (not ROW)
    __device__ __forceinline__ void unit(int u)
    {
        const int r = mLh ? (int)__umulhi((uint32_t)u, mLh) : u;
        x2 = (int)__umulhi((uint32_t)r, mL);
        place(false, r - x2 * L, u - r * Lh);
    }
};

template <bool ROW>
__device__ __forceinline__ SlabGeo slab_geo(int L, int nt, int tid)
{
    SlabGeo g;
    g.L = L;
    g.Lh = L >> 1;
    g.S1 = L * g.Lh;
    g.S = g.S1 * L;
    g.half = g.S * L;
    g.SH = g.S >> 1;
    g.planes = ROW ? L : g.Lh;
    g.mL = 0xffffffffu / (uint32_t)L + 1u;
    g.mLh = g.Lh > 1 ? 0xffffffffu / (uint32_t)g.Lh + 1u : 0u;
    if (ROW) {
        const int pr = L >> 2, pp = pr * L;   // pairs per row, per plane
        int f = nt / pp;
        f = f > L ? L : (f < 1 ? 1 : f);
        g.nit = (L + f - 1) / f;
        g.step = (L + g.nit - 1) / g.nit;     // the same number of iterations, evenly
        const int pl = tid / pp, r = tid - pl * pp, x1 = r / pr;
        g.x2 = pl;
        g.place(true, x1, 2 * (r - x1 * pr));
        if (pl >= g.step) g.x2 = 1 << 20;
    } else {
        g.step = nt;
        g.nit = (g.SH + nt - 1) / nt;
    }
    return g;
}

// x0 neighbours of a unit.  A link at x0 = 2 k + b has its neighbour x0 + 1 at
// half row position k + b and x0 - 1 at k + b - 1.  ROW: r0, r1, r2 are the
// positions -1 + b, b, 1 + b relative to the first link (wrapped), so x0 + 1 of
// the pair is (r1, r2), x0 - 1 is (r0, r1).  Otherwise r0, r1 (first link) and
// r2, r3 (second, of the other parity) are x0 + 1 and x0 - 1.
template <bool ROW>
struct X0Off {
    int r0, r1, r2, r3;
    __device__ __forceinline__ X0Off(const SlabGeo &g, int x2, int pt)
    {
        const int b = (pt + g.par + x2) & 1;
        if (ROW) {
            r0 = b ? 0 : g.rdn;
            r1 = b;
            r2 = b ? g.rup : 1;
            r3 = 0;
        } else {
            r0 = b ? g.rup : 0;
            r1 = b ? 0 : g.rdn;
            r2 = b ? 0 : g.rup;
            r3 = b ? g.rdn : 0;
        }
    }
};

// The pair of angles at offsets oA (first link) and oB (second; ROW: oA + 1),
// and of its x0 neighbours.
template <bool ROW>
__device__ __forceinline__ float2 pair_at(const float *a, int oA, int oB)
{
    if (ROW) return *(const float2 *)(a + oA);
    return make_float2(a[oA], a[oB]);
}
template <bool ROW>
__device__ __forceinline__ float2 pair_up0(const float *a, const X0Off<ROW> &x, int oA, int oB)
{
    if (ROW) return make_float2(a[oA + x.r1], a[oA + x.r2]);
    return make_float2(a[oA + x.r0], a[oB + x.r2]);
}
template <bool ROW>
__device__ __forceinline__ float2 pair_dn0(const float *a, const X0Off<ROW> &x, int oA, int oB)
{
    if (ROW) return make_float2(a[oA + x.r0], a[oA + x.r1]);
    return make_float2(a[oA + x.r1], a[oB + x.r3]);
}

// Reflect the pair of links theta_MU of parity p at plane x2, offset h of the
// slab; sl: the slab's class arrays, COPY: in shared memory (stride S), otherwise
// where they are (stride half); th: the lattice, tc / tp / tm its offsets of this
// slab, the next and the one before.
template <int MU, bool ROW, bool COPY, bool FAST>
__device__ __forceinline__ void reflect_pair(const SlabGeo &g, int x2, int h, int p, int t,
                                             float *sl, float *th, int tc, int tp, int tm)
{
    const int q = p ^ 1, SH = g.SH, half = g.half, S = COPY ? g.S : half, wr = g.S - g.S1;
    const int d1p = g.d1p, d1m = g.d1m;
    // x2 neighbours of the first link; of the second, relative to h
    const int d2p = (ROW && x2 == g.L - 1) ? -wr : g.S1, d2m = x2 == 0 ? wr : -g.S1;
    const int e2p = SH + (x2 == g.Lh - 1 ? -wr : g.S1), e2m = SH - g.S1;
    const X0Off<ROW> x(g, x2, p + t);
    auto at = [&](int nu, int par, int dA, int dB) {
        return pair_at<ROW>(sl, h + (2 * nu + par) * S + dA, h + (2 * nu + par) * S + dB);
    };
    auto up0 = [&](int nu, int par, int dA, int dB) {
        return pair_up0<ROW>(sl, x, h + (2 * nu + par) * S + dA, h + (2 * nu + par) * S + dB);
    };
    auto dn0 = [&](int nu, int par, int dA, int dB) {
        return pair_dn0<ROW>(sl, x, h + (2 * nu + par) * S + dA, h + (2 * nu + par) * S + dB);
    };
    // the same in another slab (global memory, at offset ts)
    auto gat = [&](int ts, int nu, int par, int dA, int dB) {
        return pair_at<ROW>(th, h + (2 * nu + par) * half + ts + dA,
                            h + (2 * nu + par) * half + ts + dB);
    };
    float2 g0, g1, g2, g3, g4, g5;
    if (MU < 3) {
        g0 = gat(tp, MU, q, 0, SH);      // theta_mu(x+3)
        g1 = gat(tm, MU, q, 0, SH);      // theta_mu(x-3)
        g2 = gat(tm, 3, q, 0, SH);       // theta_3(x-3)
        const int o = h + (6 + p) * half + tm;   // theta_3(x-3+mu)
        g3 = MU == 0   ? pair_up0<ROW>(th, x, o, o + SH)
             : MU == 1 ? pair_at<ROW>(th, o + d1p, o + SH + d1p)
                       : pair_at<ROW>(th, o + d2p, o + e2p);
        g4 = g5 = g3;
    } else {
        g0 = gat(tp, 0, q, 0, SH);       // theta_nu(x+3), theta_nu(x-nu+3) for nu = 0, 1, 2
        const int o = h + p * half + tp;
        g1 = pair_dn0<ROW>(th, x, o, o + SH);
        g2 = gat(tp, 1, q, 0, SH);
        g3 = gat(tp, 1, p, d1m, SH + d1m);
        g4 = gat(tp, 2, q, 0, SH);
        g5 = gat(tp, 2, p, d2m, e2m);
    }
    float2 Sr = make_float2(0.0f, 0.0f), Si = Sr;
    const float2 t0 = at(MU, p, 0, SH);
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == MU) continue;
        // a1 = theta_nu(x+mu), a2 = theta_mu(x+nu), a3 = theta_nu(x),
        // b1 = theta_nu(x-nu+mu), b2 = theta_mu(x-nu), b3 = theta_nu(x-nu)
        float2 a1, a2, a3, b1, b2, b3;
        a3 = at(nu, p, 0, SH);
        if (MU == 0) a1 = up0(nu, q, 0, SH);
        else if (MU == 1) a1 = at(nu, q, d1p, d1p + SH);
        else if (MU == 2) a1 = at(nu, q, d2p, e2p);
        else a1 = nu == 0 ? g0 : nu == 1 ? g2 : g4;
        if (nu == 0) {
            a2 = up0(MU, q, 0, SH);
            b2 = dn0(MU, q, 0, SH);
            b3 = dn0(0, q, 0, SH);
            if (MU == 1) b1 = dn0(0, p, d1p, d1p + SH);
            else if (MU == 2) b1 = dn0(0, p, d2p, e2p);
            else b1 = g1;
        } else if (nu == 1) {
            a2 = at(MU, q, d1p, d1p + SH);
            b2 = at(MU, q, d1m, d1m + SH);
            b3 = at(1, q, d1m, d1m + SH);
            if (MU == 0) b1 = up0(1, p, d1m, d1m + SH);
            else if (MU == 2) b1 = at(1, p, d2p + d1m, e2p + d1m);
            else b1 = g3;
        } else if (nu == 2) {
            a2 = at(MU, q, d2p, e2p);
            b2 = at(MU, q, d2m, e2m);
            b3 = at(2, q, d2m, e2m);
            if (MU == 0) b1 = up0(2, p, d2m, e2m);
            else if (MU == 1) b1 = at(2, p, d2m + d1p, e2m + d1p);
            else b1 = g5;
        } else {
            a2 = g0;
            b2 = g1;
            b3 = g2;
            b1 = g3;
        }
        // the staple sums of both links, formed exactly as in staple_sums2
        const float2 pf = sub2(sub2(a1, a2), a3), pb = sub2(sub2(b3, b1), b2);
        float2 sf, cf, sb, cb;
        sin_cos<FAST>(pf.x, &sf.x, &cf.x);
        sin_cos<FAST>(pf.y, &sf.y, &cf.y);
        sin_cos<FAST>(pb.x, &sb.x, &cb.x);
        sin_cos<FAST>(pb.y, &sb.y, &cb.y);
        Sr = add2(Sr, add2(cf, cb));
        Si = add2(Si, add2(sf, sb));
    }
    const float2 al = arg2<FAST>(Si, Sr);
    float2 tn;
    tn.x = wrap_angle(-t0.x - 2.0f * al.x);
    tn.y = wrap_angle(-t0.y - 2.0f * al.y);
    const int so = h + (2 * MU + p) * S, go = h + (2 * MU + p) * half + tc;
    if (ROW) {
        if (COPY) *(float2 *)(sl + so) = tn;
        *(float2 *)(th + go) = tn;
    } else {
        if (COPY) {
            sl[so] = tn.x;
            sl[so + SH] = tn.y;
        }
        th[go] = tn.x;
        th[go + SH] = tn.y;
    }
}

// The two classes of direction MU in one slab.
template <int MU, bool ROW, bool COPY, bool FAST>
__device__ __forceinline__ void reflect_dir(SlabGeo &g, const Team &tm_, int t, int mask,
                                            float *sl, float *th, int tc, int tp, int tm)
{
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        if (!((mask >> (2 * MU + p)) & 1)) continue;
        if (ROW) {
            int x2 = g.x2, h = g.h;
#pragma unroll 1
            for (int i = 0; i < g.nit; ++i) {
                if (x2 < g.planes)
                    reflect_pair<MU, ROW, COPY, FAST>(g, x2, h, p, t, sl, th, tc, tp, tm);
                x2 += g.step;
                h += g.step * g.S1;
            }
        } else {
#pragma unroll 1
            for (int u = tm_.tid; u < g.SH; u += g.step) {
                g.unit(u);
                reflect_pair<MU, ROW, COPY, FAST>(g, g.x2, g.h, p, t, sl, th, tc, tp, tm);
            }
        }
        tm_.sync();   // the next class reads the angles written here
    }
}

// The whole pass of the team's lattice: every reflection is taken (see
// overrelax_pass).  slab_off: the team's slab in g_dyn (COPY).  The team shrinks to
// the warps that hold a link; the others return.
template <bool ROW, bool COPY, bool FAST>
__device__ __noinline__ void reflect_slabs(Team team, int L_, float *th_, int slab_off, int mask)
{
    const int L = uniform(L_);
    float *th = (float *)__shfl_sync(kFull, (unsigned long long)th_, 0);
    float *sl = g_dyn + uniform(slab_off);
    SlabGeo g = slab_geo<ROW>(L, team.nt, team.tid);
    const int need = ((ROW ? g.step * (L >> 2) * L : min(g.SH, g.step)) + 31) >> 5;
    if (team.w >= need) return;
    team.nw = need < team.nw ? need : team.nw;
    team.nt = team.nw * 32;
    const int S = g.S, half = g.half;
#pragma unroll 1
    for (int t = 0; t < L; ++t) {
        const int tc = t * S, tp = (t == L - 1 ? 0 : t + 1) * S, tm = (t == 0 ? L - 1 : t - 1) * S;
        if (COPY) {
            // S = L^3 / 2 is a multiple of 4 floats for even L, as are all offsets
#pragma unroll 1
            for (int a = 0; a < 8; ++a)
                for (int i = 4 * team.tid; i < S; i += 4 * team.nt)
                    cp_async16(sl + a * S + i, th + tc + a * half + i);
            cp_async_commit();
            // the next slab on its way from HBM to L2
#pragma unroll 1
            for (int a = 0; a < 8; ++a)
                for (int i = 32 * team.tid; i < S; i += 32 * team.nt)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(th + tp + a * half + i));
            cp_async_wait<0>();
            team.sync();
        } else {
            sl = th + tc;
        }
        reflect_dir<0, ROW, COPY, FAST>(g, team, t, mask, sl, th, tc, tp, tm);
        reflect_dir<1, ROW, COPY, FAST>(g, team, t, mask, sl, th, tc, tp, tm);
        reflect_dir<2, ROW, COPY, FAST>(g, team, t, mask, sl, th, tc, tp, tm);
        reflect_dir<3, ROW, COPY, FAST>(g, team, t, mask, sl, th, tc, tp, tm);
    }
}

// ---------------------------------------------------------------------------
// Overrelaxation pass of a lattice that is in shared memory as a whole.  A
// class of a slab has at most as many links as the team has threads, so the
// pass is a chain of 8 L short steps, and the time is the step's latency: one
// link per thread, the side a compile-time constant (every class array and wrap
// an immediate of the load), the thread's place in the slab worked out once.
// ---------------------------------------------------------------------------
template <int MU, int L, bool FAST>
__device__ __forceinline__ void reflect_resident(float *l, int p, int up0, int dn0, int d1p,
                                                 int d1m, int d2p, int d2m, int d3p, int d3m)
{
    // l: the link's half site in class array 0; up / dn: half-site distances to
    // x + nu, x - nu
    constexpr int half = L * L * L * L / 2;
    const int up[4] = {up0, d1p, d2p, d3p}, dn[4] = {dn0, d1m, d2m, d3m};
    float *lp = l + p * half;               // arrays of parity p at 2 nu half
    const float *lq = l + (p ^ 1) * half;   // of the other parity
    const float t0 = lp[2 * MU * half];
    float v[18];
    int j = 0;
#pragma unroll
    for (int nu = 0; nu < 4; ++nu) {
        if (nu == MU) continue;
        v[6 * j + 0] = lq[2 * nu * half + up[MU]];
        v[6 * j + 1] = lq[2 * MU * half + up[nu]];
        v[6 * j + 2] = lp[2 * nu * half];
        v[6 * j + 3] = lp[2 * nu * half + dn[nu] + up[MU]];
        v[6 * j + 4] = lq[2 * MU * half + dn[nu]];
        v[6 * j + 5] = lq[2 * nu * half + dn[nu]];
        ++j;
    }
    float Sr, Si;
    staple_sum_regs<FAST>(v, Sr, Si);
    lp[2 * MU * half] = wrap_angle(-t0 - 2.0f * arg<FAST>(Si, Sr));
}

template <int L, bool FAST>
__device__ __noinline__ void reflect_lattice(Team team, int lat_off, int mask)
{
    constexpr int Lh = L / 2, S1 = L * Lh, S = S1 * L, nw = (S + 31) / 32;
    if (team.w >= nw) return;
    const int h = team.tid;
    const bool mine = h < S;
    const int row = h / Lh, k = h - row * Lh, x2 = row / L, x1 = row - x2 * L;
    const int d1p = x1 == L - 1 ? Lh - S1 : Lh, d1m = x1 == 0 ? S1 - Lh : -Lh;
    const int d2p = x2 == L - 1 ? S1 - S : S1, d2m = x2 == 0 ? S - S1 : -S1;
    const int dn = k == 0 ? Lh - 1 : -1, up = k == Lh - 1 ? 1 - Lh : 1;
    float *l = g_dyn + lat_off + h;
#pragma unroll 1
    for (int t = 0; t < L; ++t, l += S) {
        const int d3p = t == L - 1 ? S - S * L : S, d3m = t == 0 ? S * L - S : -S;
        const int c = (x1 + x2 + t) & 1;
#define LLR_CLASS(MU)                                                                            \
    _Pragma("unroll 1") for (int p = 0; p < 2; ++p)                                              \
    {                                                                                            \
        if (!((mask >> (2 * MU + p)) & 1)) continue;                                             \
        const bool odd = p ^ c; /* x0 = 2 k + odd */                                             \
        if (mine)                                                                                \
            reflect_resident<MU, L, FAST>(l, p, odd ? up : 0, odd ? 0 : dn, d1p, d1m, d2p, d2m,  \
                                          d3p, d3m);                                             \
        bar_sync(team.bar, nw * 32); /* the next class reads the angles written here */          \
    }
        LLR_CLASS(0)
        LLR_CLASS(1)
        LLR_CLASS(2)
        LLR_CLASS(3)
#undef LLR_CLASS
    }
}

// One overrelaxation pass of a lattice by a team, over the selected classes,
// slab by slab of the last coordinate (x3 = t, the h range [t S, (t+1) S) of
// every class array, S = L^3 / 2) and the classes within each slab, under the
// window rule of the running energy (windowed false: no window, every
// reflection is taken -- the multicanonical run).
template <bool FAST>
__device__ __noinline__ void overrelax_pass(Smem &sm, int slot, const Team &team, float *th,
                                            int slab_off, bool res, int B, int class_mask,
                                            bool windowed)
{
    const LatState &st = sm.st[slot];
    const int half = st.half, L = st.L, S = half / L;
    const long long lo = windowed ? st.lo_fx : -(1ll << 62);
    const long long hi = windowed ? st.hi_fx : (1ll << 62);
    // a block's |dE| is below B 2^-14, so no block can be refused unless E is
    // inside the window and within that of an edge
    const long long bound = (long long)B * kOrDeltaMaxFx;
    const long long E = st.E_fx;   // the running energy; overrelaxation leaves it
    const bool free_all = E < lo || E > hi || (E - bound >= lo && E + bound <= hi);
    // the L^2 / 4 pairs of a plane need a thread each
    const bool in_slabs = free_all && (res || (L & 3) != 0 || L * L <= 4 * team.nt);
    if (in_slabs && res) {
        switch (L) {
            case 2: reflect_lattice<2, FAST>(team, slab_off, class_mask); break;
            case 4: reflect_lattice<4, FAST>(team, slab_off, class_mask); break;
            case 6: reflect_lattice<6, FAST>(team, slab_off, class_mask); break;
            case 8: reflect_lattice<8, FAST>(team, slab_off, class_mask); break;
            default: reflect_lattice<10, FAST>(team, slab_off, class_mask); break;
        }
    } else if (in_slabs && L <= kSlabMaxL) {
        if ((L & 3) == 0)
            reflect_slabs<true, true, FAST>(team, L, th, slab_off, class_mask);
        else
            reflect_slabs<false, true, FAST>(team, L, th, slab_off, class_mask);
    } else if (in_slabs) {
        if ((L & 3) == 0)
            reflect_slabs<true, false, FAST>(team, L, th, slab_off, class_mask);
        else
            reflect_slabs<false, false, FAST>(team, L, th, slab_off, class_mask);
    }
    int taken = 0;              // moves taken by this thread in near-edge groups
    if (!in_slabs) {
#pragma unroll 1
        for (int t = 0; t < L; ++t) {
#pragma unroll 1
            for (int cls = 0; cls < 8; ++cls) {
                if (!((class_mask >> cls) & 1)) continue;
                const int p = cls & 1;
                if (free_all) {
                    switch (cls >> 1) {
                        case 0: overrelax_class<0, FAST>(st, team, th, p, t * S, S); break;
                        case 1: overrelax_class<1, FAST>(st, team, th, p, t * S, S); break;
                        case 2: overrelax_class<2, FAST>(st, team, th, p, t * S, S); break;
                        default: overrelax_class<3, FAST>(st, team, th, p, t * S, S); break;
                    }
                } else {
                    switch (cls >> 1) {
                        case 0: taken += overrelax_class_near<0, FAST>(st, team, th, p, t * S, S, B, E); break;
                        case 1: taken += overrelax_class_near<1, FAST>(st, team, th, p, t * S, S, B, E); break;
                        case 2: taken += overrelax_class_near<2, FAST>(st, team, th, p, t * S, S, B, E); break;
                        default: taken += overrelax_class_near<3, FAST>(st, team, th, p, t * S, S, B, E); break;
                    }
                }
                team.sync();   // the next group reads the angles written here
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) taken += __shfl_down_sync(kFull, taken, o);
        if ((threadIdx.x & 31) == 0 && taken)
            atomicAdd(&sm.acc_cnt[slot], (unsigned long long)taken);
    }
    if (team.tid == 0 && free_all)
        atomicAdd(&sm.acc_cnt[slot], (unsigned long long)__popc(class_mask & 0xFF) *
                                         (unsigned long long)half);
}

// What the phases of a sweep need of the launch.
struct Phase {
    int teams, tw;        // lattices a CTA works on, warps per lattice
    int nl;               // lattices of this item (<= teams)
    int or_teams;         // lattices in overrelaxation at a time (their slabs in shared memory)
    int slab;             // floats of shared memory per slab (res: per lattice)
    bool res;             // the item's lattices are in shared memory as a whole
    int ring;             // offset of the heat-bath rings in g_dyn (floats)
    int D;                // ring stages

    // the links of lattice `slot` of the item
    __device__ __forceinline__ float *links(const Smem &sm, const KernelArgs &args, int slot) const
    {
        return res ? g_dyn + slot * slab : args.theta + sm.st[slot].off;
    }
};

// One class of a heat-bath pass by the team's producers.
template <int MU, bool MUCA, bool FAST>
__device__ __forceinline__ void produce(Smem &sm, const Phase &ph, int slot, int pw, float *th,
                                        int p, uint32_t tag)
{
    // the accurate sine / cosine dominates without fast math: one form for any L
    const bool row = FAST && (sm.st[slot].L & 3) == 0;
    const int off = slot * ph.slab;
    if (ph.res) {
        if (row)
            produce_class<MU, FAST, true, MUCA, FAST>(sm, slot, pw, th, off, p, tag);
        else
            produce_class<MU, false, true, MUCA, FAST>(sm, slot, pw, th, off, p, tag);
    } else {
        if (row)
            produce_class<MU, FAST, false, MUCA, FAST>(sm, slot, pw, th, off, p, tag);
        else
            produce_class<MU, false, false, MUCA, FAST>(sm, slot, pw, th, off, p, tag);
    }
}

template <bool MUCA, bool FAST>
__device__ __forceinline__ void produce(Smem &sm, const Phase &ph, int slot, int pw, float *th,
                                        int mu, int p, uint32_t tag)
{
    switch (mu) {
        case 0: produce<0, MUCA, FAST>(sm, ph, slot, pw, th, p, tag); break;
        case 1: produce<1, MUCA, FAST>(sm, ph, slot, pw, th, p, tag); break;
        case 2: produce<2, MUCA, FAST>(sm, ph, slot, pw, th, p, tag); break;
        default: produce<3, MUCA, FAST>(sm, ph, slot, pw, th, p, tag); break;
    }
}

// Heat-bath pass of every active lattice of the item, each by its team, one
// class at a time over the whole lattice, so the producer/consumer pipeline
// drains once per class.  kind 0: window rule, 2: multicanonical.
template <bool FAST>
__device__ __noinline__ void heatbath_phase(Smem &sm, const Phase &ph, const KernelArgs &args,
                                            int kind, uint32_t tag, int B, int class_mask)
{
    if (threadIdx.x < ph.nl) {
        const int k = threadIdx.x;
        sm.acc_cnt[k] = 0ull;
        HbTeam &hb = sm.hb[k];
        // no more producers than groups
        const int most = producers(ph.teams);
        hb.nw = 1 + min(most, (sm.st[k].half + 63) / 64);
        // the consumers of different teams on different quarters of the SM
        hb.cw = hb.nw - 1;
        for (int c = hb.nw - 1; c >= max(0, hb.nw - 4); --c)
            if (((k * ph.tw + c) & 3) == 3 - (k & 3)) hb.cw = c;
        hb.D = ph.D;
        hb.ring = ph.ring + k * ph.D * most * (kStageGroupBytes / 4);
        hb.full = 1 + 2 * ph.D * k;
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, slot = warp / ph.tw, w = warp - slot * ph.tw;
    if (slot < ph.nl && sm.active[slot]) {
        LatState &st = sm.st[slot];
        const int nw = sm.hb[slot].nw;
        // consumer or not, and the rank among the producers (nw - 1 of them)
        bool consumer;
        int pw;
        if (ph.teams == 1) {
            consumer = w == kWarps - 1;
            pw = (w & 3) == 3 ? nw : w / 4 * 3 + (w & 3);
        } else {
            const int cw = sm.hb[slot].cw;
            consumer = w == cw;
            pw = w - (w > cw ? 1 : 0);
        }
        if (consumer || pw < nw - 1) {
            float *th = args.theta + st.off;
#pragma unroll 1
            for (int cls = 0; cls < 8; ++cls) {
                if (!((class_mask >> cls) & 1)) continue;
                const int mu = cls >> 1, p = cls & 1;
                if (consumer) {
                    if (kind == 2)
                        consume_class_muca(st, sm.hb[slot], args);
                    else
                        consume_class(st, sm.hb[slot], B);
                } else {
                    if (kind == 2)
                        produce<true, FAST>(sm, ph, slot, pw, th, mu, p, tag);
                    else
                        produce<false, FAST>(sm, ph, slot, pw, th, mu, p, tag);
                }
                // the next class reads the angles written here
                bar_sync(sm.hb[slot].full, nw * 32);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < ph.nl && sm.active[threadIdx.x]) {
        LatState &st = sm.st[threadIdx.x];
        st.hb_acc += sm.acc_cnt[threadIdx.x];
        st.hb_tot += (unsigned long long)__popc(class_mask & 0xFF) * (unsigned long long)st.half;
    }
    __syncthreads();
}

// Overrelaxation pass of every active lattice of the item, or_teams of them at a
// time, each by its share of the warps.
template <bool FAST>
__device__ __noinline__ void overrelax_phase(Smem &sm, const Phase &ph, const KernelArgs &args,
                                             int B, int class_mask, bool windowed)
{
    if (threadIdx.x < kMaxTeams) sm.acc_cnt[threadIdx.x] = 0ull;
    __syncthreads();
    const int tw = kWarps / ph.or_teams, warp = threadIdx.x >> 5, k = warp / tw;
    if (k < ph.or_teams) {
        const Team t{warp - k * tw, tw, (int)threadIdx.x - k * tw * 32, tw * 32, 1 + k};
        for (int slot = k; slot < ph.nl; slot += ph.or_teams) {
            if (!sm.active[slot]) continue;
            overrelax_pass<FAST>(sm, slot, t, ph.links(sm, args, slot),
                                 (ph.res ? slot : k) * ph.slab, ph.res, B, class_mask, windowed);
            // a pass may end with some of the team's warps only, and the next
            // lattice's slab takes this one's place
            bar_sync(8 + k, t.nt);
        }
    }
    __syncthreads();
    if (threadIdx.x < ph.nl && sm.active[threadIdx.x]) {
        LatState &st = sm.st[threadIdx.x];
        st.or_acc += sm.acc_cnt[threadIdx.x];
        st.or_tot += (unsigned long long)__popc(class_mask & 0xFF) * (unsigned long long)st.half;
    }
    __syncthreads();
}

// cos(x) for x = hi + lo (|hi| <= 4 pi, |lo| tiny), accurate to about one
// ulp and without systematic error, for the fixed-point plaquette sums: a
// per-plaquette bias of 1e-9 would add up to ~1e-3 over the 960000
// plaquettes of an L = 20 lattice (the accurate sincosf showed a mean error of
// that order there), shifting the measured <<dE>>.
//   Reduction (Cody & Waite, "Software Manual for the Elementary Functions",
//   1980): k = nearest integer to hi 2/pi and x - k pi/2 = rh + rl with pi/2
//   split into P1 + P2 + P3 (P1, P2 of 20 significant bits, so k P1 and k P2
//   are exact for |k| <= 8): rh = hi - k P1 is exact and rl = lo - k P2 - k P3
//   is tiny.  Rounding x - k P2 to one float instead would repeat the same
//   rounding error for every angle of a binade (hi - k P1 lies on the float
//   grid), a bias of ~2e-10 per plaquette.
//   Evaluation: the Taylor series of cos and sin at rh in z = rh^2, truncated
//   where the next term is below 1e-15; the coefficients 1/4!, 1/3! and 1/5!
//   are carried as float pairs (their float rounding alone would bias the
//   result by up to 5e-9); then cos(rh + rl) = cos rh - rl sin rh and
//   sin(rh + rl) = sin rh + rl cos rh (plus the rl^2 terms), and
//   cos x = cos r, -sin r, -cos r, sin r for k = 0, 1, 2, 3 (mod 4).
// Two angles at a time in packed arithmetic.
__device__ __forceinline__ float2 cos_unbiased2(float2 hi, float2 lo)
{
    const float2 k = make_float2(rintf(hi.x * 0.636619747f), rintf(hi.y * 0.636619747f));
    const float2 nk = make_float2(-k.x, -k.y);
    const float2 rh = fma2(nk, both(1.5707950592041016f), hi);
    float2 rl = fma2(nk, both(1.2675900507019833e-06f), lo);
    rl = fma2(nk, both(7.4435477313145038e-13f), rl);
    const float2 z = mul2(rh, rh);
    // cos rh = 1 - z/2 + z^2/4! - ... - z^7/14!
    float2 c = both(-1.147074536e-11f);
    c = fma2(c, z, both(2.087675588e-09f));
    c = fma2(c, z, both(-2.755731998e-07f));
    c = fma2(c, z, both(2.480158764e-05f));
    c = fma2(c, z, both(-1.388888923e-03f));
    c = fma2(c, z, both(-1.241763470e-09f));   // 1/4! = 4.166666791e-02 - 1.241763470e-09
    c = add2(c, both(4.166666791e-02f));
    c = fma2(c, z, both(-0.5f));
    c = fma2(c, z, both(1.0f));
    // sin rh = rh (1 - z/3! + z^2/5! - ... - z^7/15!)
    float2 t = both(-7.647163610e-13f);
    t = fma2(t, z, both(1.605904437e-10f));
    t = fma2(t, z, both(-2.505210794e-08f));
    t = fma2(t, z, both(2.755731884e-06f));
    t = fma2(t, z, both(-1.984127011e-04f));
    t = fma2(t, z, both(-4.346172033e-10f));   // 1/5! = 8.333333768e-03 - 4.346172033e-10
    t = add2(t, both(8.333333768e-03f));
    t = fma2(t, z, both(4.967053879e-09f));    // 1/3! = 1.666666716e-01 - 4.967053879e-09
    t = sub2(t, both(1.666666716e-01f));
    t = mul2(rh, fma2(t, z, both(1.0f)));
    // cos(rh + rl), sin(rh + rl) to second order in rl (|rl| <= 1e-5: the
    // dropped -rl^2/2 alone would bias cos by up to -5e-11); the small terms
    // are summed first, so the correction is not rounded away
    const float2 h = mul2(mul2(both(0.5f), rl), rl);
    const float2 cr = sub2(c, fma2(t, rl, mul2(c, h)));
    const float2 sr = add2(t, fma2(c, rl, mul2(make_float2(-t.x, -t.y), h)));
    auto pick = [](float kf, float cv, float sv) {
        const int q = (int)kf & 3;
        const float v = (q & 1) ? sv : cv;
        return (q == 1 || q == 2) ? -v : v;
    };
    return make_float2(pick(k.x, cr.x, sr.x), pick(k.y, cr.y, sr.y));
}

__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = add2(a, b);
    const float2 bb = sub2(s, a);
    e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// cos of the plaquette angles a + b - c - d of two plaquettes, in packed
// arithmetic: each angle is formed exactly as hi + lo and its cosine taken by
// cos_unbiased2.
__device__ __forceinline__ float2 plaquette_cos2(float2 a, float2 b, float2 c, float2 d)
{
    float2 s1, e1, s2, e2, hi, e3;
    two_sum2(a, b, s1, e1);
    two_sum2(c, d, s2, e2);
    two_sum2(s1, make_float2(-s2.x, -s2.y), hi, e3);
    return cos_unbiased2(hi, add2(sub2(e1, e2), e3));
}

// Fresh energy of the team's lattice in fixed point: sum over the 6 V
// plaquettes, exact int64 accumulation and reduction.  Two sites per thread (half
// sites h, h + 1 of a parity), their plaquettes in packed arithmetic.  Valid in
// the team's thread 0.  Angles that are no numbers leave no energy: kNoEnergy, found
// apart from the sum, in which the parts of several such plaquettes could cancel.
template <bool ROW>
__device__ __noinline__ long long fresh_energy_fx(const LatState &st_, const Team &team,
                                                  long long *red, const float *th)
{
    const int lane = team.tid & 31;
    const int L = uniform(st_.L), half = uniform(st_.half);
    const uint32_t magic = uniform(st_.magic);
    long long acc = 0;
    unsigned wild = 0;   // 2^21 or more: a plaquette was no number
#pragma unroll 1
    for (int p = 0; p < 2; ++p)
#pragma unroll 1
        for (int h = 2 * team.tid; h < half; h += 2 * team.nt) {
            const LinkPair<ROW> n(h, p, L, magic);
            const float *tp = th + p * half + h, *tq = th + (p ^ 1) * half + h;
            auto up = [&](int nu, int mu) {   // theta_nu(x + mu)
                const float *a = tq + 2 * nu * half;
                if (ROW && mu > 0) return *(const float2 *)(a + n.up0[mu]);
                return make_float2(a[n.up0[mu]], a[1 + n.up1[mu]]);
            };
            float2 t[4];
            int hi = 0, lo = 0;
            bool bad = false;
#pragma unroll
            for (int mu = 0; mu < 4; ++mu) t[mu] = *(const float2 *)(tp + 2 * mu * half);
#pragma unroll
            for (int mu = 0; mu < 4; ++mu)
#pragma unroll
                for (int nu = mu + 1; nu < 4; ++nu) {
                    const float2 v = plaquette_cos2(t[mu], up(nu, mu), up(mu, nu), t[nu]);
                    int a, b;
                    fx_parts(v.x, a, b);
                    hi += a;
                    lo += b;
                    fx_parts(v.y, a, b);
                    hi += a;
                    lo += b;
                    bad |= !(fabsf(v.x) < 512.0f) || !(fabsf(v.y) < 512.0f);
                }
            // 12 cosines: sums of parts within 32 bits, and |hi| <= 12 2^12 but for NaNs:
            // each has the part 0x7fffffff - 0x4b400000, and of 1 to 12 of these none
            // sums to below 2^26 in size modulo 2^32.  (One flag would do for both
            // lines; carried through the loop as `bad` it costs the compiler's
            // schedule: 1824 of L = 20 4.37 ms, with the test of hi alone 4.03, so 3.75.)
            wild |= (unsigned)(hi + (1 << 20));
            acc += bad ? 0ll : (long long)hi * (1 << 20) + lo;
        }
    bool none = __any_sync(kFull, wild >= (1u << 21));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
    if (lane == 0) red[team.w] = none ? kNoEnergy : acc;
    team.sync();
    if (team.w != 0) return 0;
    long long tot = lane < team.nw ? red[lane] : 0;   // 24 warps at most
    none = __any_sync(kFull, tot == kNoEnergy);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(kFull, tot, o);
    return none ? kNoEnergy : tot;
}

// Fresh energies of the active lattices of the item, each by its team, into
// the tracked energy.  resync: at the end of a composite sweep, which records
// the drift, counts the sweep and measures.
__device__ __noinline__ void energy_phase(Smem &sm, const Phase &ph, const KernelArgs &args,
                                          bool resync, bool measure)
{
    const int warp = threadIdx.x >> 5, slot = warp / ph.tw;
    if (slot < ph.nl && sm.active[slot]) {
        const Team t{warp - slot * ph.tw, ph.tw, (int)threadIdx.x - slot * ph.tw * 32, ph.tw * 32,
                     1 + slot};
        LatState &st = sm.st[slot];
        const float *th = ph.links(sm, args, slot);
        long long *red = sm.red + slot * ph.tw;
        const long long fresh = (st.L & 3) == 0 ? fresh_energy_fx<true>(st, t, red, th)
                                                : fresh_energy_fx<false>(st, t, red, th);
        if (t.tid == 0) {
            if (fresh == kNoEnergy) st.status = -5;   // LLR_ERR_NUMERIC
            if (resync) {
                const double drift = fabs((double)(st.E_fx - fresh) * kInvFx);
                if (drift > st.max_drift) st.max_drift = drift;
                st.sweep += 1u;
                st.sweeps_done += 1ull;
                if (measure) {
                    const double dEm = energy_of(fresh) - (st.E_lo + 0.5 * st.dE);
                    st.sum_dE += dEm;
                    st.sum_dE2 += dEm * dEm;
                    st.n_meas += 1;
                }
            }
            st.E_fx = fresh;
        }
    }
    __syncthreads();
}

template <bool FAST>
__device__ void composite_sweep(Smem &sm, const Phase &ph, const KernelArgs &args, uint32_t tag,
                                bool measure)
{
    heatbath_phase<FAST>(sm, ph, args, 0, tag, args.block, 0xFF);
    for (int k = 0; k < args.n_or; ++k)
        overrelax_phase<FAST>(sm, ph, args, args.block, 0xFF, true);
    energy_phase(sm, ph, args, true, measure);
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Robbins-Monro update of the CTA's lattice (thread 0).
__device__ __noinline__ void rm_update(LatState &st, const KernelArgs &args, int lat)
{
    const int step = args.step_dev ? *args.step_dev : 0;
    const double mean = st.n_meas > 0 ? st.sum_dE / st.n_meas : 0.0;
    const double a_new =
        st.a + 12.0 * mean / (st.dE * st.dE * (double)(args.rm_index + step + 1));
    if (!isfinite(a_new)) st.status = -5;   // LLR_ERR_NUMERIC
    st.a = a_new;
    if (args.a_out) args.a_out[lat] = a_new;
    if (args.mean_out) args.mean_out[lat] = mean;
    if (args.hist) args.hist[(size_t)step * (size_t)args.n_lat + (size_t)lat] = a_new;
}

// The item's lattices into shared memory (in) and back to global memory.
__device__ __noinline__ void copy_lattices(const Smem &sm, const Phase &ph, const KernelArgs &args,
                                           bool in)
{
    for (int slot = 0; slot < ph.nl; ++slot) {
        float *g = args.theta + sm.st[slot].off, *l = g_dyn + slot * ph.slab;
        const int n = 8 * sm.st[slot].half;   // a multiple of 4, lattices 128-byte aligned
        for (int i = 4 * threadIdx.x; i < n; i += 4 * kThreads) {
            if (in)
                cp_async16(l + i, g + i);
            else
                *(float4 *)(g + i) = *(const float4 *)(l + i);
        }
    }
    if (in) {
        cp_async_commit();
        cp_async_wait<0>();
    }
    __syncthreads();
}

// One CTA per SM.  Work items are (composite sweep j, group of up to `teams`
// lattices); the lattices of a group advance together, phase by phase.
template <bool FAST>
__global__ void __launch_bounds__(kThreads, 1) llr_kernel(const __grid_constant__ KernelArgs args)
{
    __shared__ Smem sm;
    const int tid = threadIdx.x;
    const bool multi =
        args.program == kProgSweeps || args.program == kProgRM || args.program == kProgMuca;
    const int per_lat = multi ? args.n_therm + args.n_meas : 1;
    Phase ph;
    ph.teams = args.teams;
    ph.tw = kWarps / args.teams;
    ph.or_teams = args.or_teams;
    ph.slab = args.slab;
    ph.res = args.resident != 0;
    ph.ring = args.ring_off;
    ph.D = args.ring;
    const unsigned n_groups = (unsigned)((args.n_lat + args.teams - 1) / args.teams);
    const unsigned n_items = n_groups * (unsigned)per_lat;
    unsigned *err = args.sync;
    unsigned *counter = args.sync + 1;
    unsigned *done = args.sync + 2;
    for (;;) {
        if (tid == 0) {
            const unsigned i = atomicAdd(counter, 1u);
            int state = 0;
            if (i < n_items) {
                const int j = (int)(i / n_groups);
                const unsigned grp = i % n_groups;
                state = 1;
                if (j > 0) {
                    // sweep j-1 of this group was dequeued earlier by a running
                    // CTA; wait for it, but never longer than wait_limit_ns.  Once
                    // any wait has run out (the error word is set; it stays set
                    // until the host reads it), an item that would wait skips at
                    // once: the sweep before it may never come.
                    const unsigned long long t0 = global_ns();
                    while (ld_acquire(done + grp) < (unsigned)j) {
                        if (ld_acquire(err) != 0u) {
                            state = 2;
                            break;
                        }
                        if (global_ns() - t0 > args.wait_limit_ns) {
                            atomicOr(err, 1u);
                            state = 2;
                            break;
                        }
                        __nanosleep(256);
                    }
                }
                sm.item_first = (int)grp * args.teams;
                sm.item_n = min(args.teams, args.n_lat - (int)grp * args.teams);
                sm.item_j = j;
            }
            sm.item_state = state;
        }
        __syncthreads();
        const int state = sm.item_state;
        if (state == 0) break;
        if (state == 2) {
            __syncthreads();
            continue;   // timed out: leave these lattices alone, the host reads the error word
        }
        const int j = sm.item_j;
        ph.nl = sm.item_n;
        // thread k < nl looks after lattice k of the item
        const bool mine = tid < ph.nl;
        int lat = 0;
        if (mine) {
            const int slot = sm.item_first + tid;
            lat = args.order ? args.order[slot] : slot;
            sm.st[tid] = args.lats[lat];
            LatState &st = sm.st[tid];
            sm.cap_cnt[tid] = 0ull;
            sm.active[tid] = 1;
            if (args.program == kProgSweeps || args.program == kProgRM ||
                args.program == kProgBegin) {
                if (j == 0) {
                    if (args.a_in) st.a = args.a_in[lat];
                    st.sum_dE = 0.0;
                    st.sum_dE2 = 0.0;
                    st.n_meas = 0;
                }
            } else if (args.program == kProgPass && args.a_in) {
                st.a = args.a_in[lat];
            }
            const bool muca = args.program == kProgMuca ||
                              (args.program == kProgPass && args.pass_kind == 2);
            sm.a_f[tid] = muca ? (float)args.muca_a0 : (float)st.a;
            sm.n_app[tid] = 0;
        }
        __syncthreads();
        if (ph.res) copy_lattices(sm, ph, args, true);

        switch (args.program) {
            case kProgSweeps:
            case kProgRM: {
                composite_sweep<FAST>(sm, ph, args, kTagSweep, args.measure && j >= args.n_therm);
                if (j == per_lat - 1 && mine) {
                    if (args.program == kProgRM)
                        rm_update(sm.st[tid], args, lat);
                    else if (args.mean_out)
                        args.mean_out[lat] = sm.st[tid].sum_dE;
                }
                break;
            }
            case kProgApproach: {
                for (;;) {
                    bool go = false;
                    if (mine) {
                        LatState &st = sm.st[tid];
                        go = dist_fx(st.E_fx, st.lo_fx, st.hi_fx) != 0;
                        if (go && sm.n_app[tid] >= args.max_approach) {
                            st.status = -3;   // LLR_ERR_WINDOW
                            go = false;
                        }
                        sm.active[tid] = go;
                        sm.a_f[tid] = (float)(st.E_fx < st.lo_fx ? -args.beta_up : -args.beta_dn);
                        sm.n_app[tid] += go;
                    }
                    if (!__syncthreads_or(go)) break;
                    composite_sweep<FAST>(sm, ph, args, kTagApproach, false);
                }
                if (mine && args.approach_sweeps) args.approach_sweeps[lat] = sm.n_app[tid];
                break;
            }
            case kProgResync:
                energy_phase(sm, ph, args, false, false);
                break;
            case kProgPass: {
                if (args.pass_kind == 2)   // multicanonical heat-bath pass at slope a0
                    heatbath_phase<FAST>(sm, ph, args, 2, kTagSweep, 1, args.class_mask);
                else if (args.pass_kind == 3)   // the end of a composite sweep
                    energy_phase(sm, ph, args, true, false);
                else if (args.pass_kind == 1)
                    overrelax_phase<FAST>(sm, ph, args, args.block, args.class_mask, true);
                else
                    heatbath_phase<FAST>(sm, ph, args, 0, kTagSweep, args.block, args.class_mask);
                break;
            }
            case kProgMuca: {
                // one multicanonical composite sweep (Sec. 2.6): heat-bath pass
                // for the weight 1/rho~, n_or overrelaxation passes (they keep
                // E, so every weight of E takes them), resync, energy history
                heatbath_phase<FAST>(sm, ph, args, 2, kTagSweep, 1, 0xFF);
                for (int k = 0; k < args.n_or; ++k)
                    overrelax_phase<FAST>(sm, ph, args, 1, 0xFF, false);
                energy_phase(sm, ph, args, true, false);
                if (mine && args.e_hist)
                    args.e_hist[(size_t)j * (size_t)args.n_lat + (size_t)lat] =
                        energy_of(sm.st[tid].E_fx);
                break;
            }
            case kProgFinish:
                energy_phase(sm, ph, args, true, args.measure != 0);
                break;
            case kProgUpdate:
                if (mine) rm_update(sm.st[tid], args, lat);
                break;
            default:
                break;
        }
        __syncthreads();
        if (ph.res) copy_lattices(sm, ph, args, false);
        if (mine) {
            sm.st[tid].caps += sm.cap_cnt[tid];
            args.lats[lat] = sm.st[tid];
            __threadfence();
        }
        __syncthreads();
        if (tid == 0) {
            __threadfence();
            st_release(done + (unsigned)(sm.item_first / args.teams), (unsigned)(j + 1));
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Hot start: theta = -pi + 2 pi u (Haar measure), u from Philox with counter
// (link, 0, init tag, 0); computed in FP64 and rounded once to float.
// ---------------------------------------------------------------------------
__global__ void hot_start_kernel(LatState *lats, float *theta)
{
    const LatState st = lats[blockIdx.y];
    const int V = 2 * st.half;
    const int n = 4 * V;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        const int mu = l / V, s = l - mu * V;
        const int L = st.L;
        const int x0 = s % L, x1 = (s / L) % L, x2 = (s / (L * L)) % L, x3 = s / (L * L * L);
        const int p = (x0 + x1 + x2 + x3) & 1;
        const U4 w = philox4x32_10((uint32_t)l, 0u, kTagInit, 0u, st.key0, st.key1);
        const double u = (double)((w.x >> 9) * 2u + 1u) * (1.0 / 16777216.0);
        const double t = __dadd_rn(-3.14159265358979323846, __dmul_rn(6.28318530717958647692, u));
        theta[st.off + (size_t)(2 * mu + p) * st.half + (s >> 1)] = (float)t;
    }
}

// FP64 fresh energy: plaquette angle and cos in double, warp-shuffle FP64
// reduction.  Bound by the FP64 cosines (about 1.6 DFMA per clock and SM), so a
// lattice is spread over gridDim.x CTAs, one part of the sum each: one lattice of
// L = 20 takes 0.10 ms a call where one CTA took 6.7 ms.
constexpr int kEnergyThreads = 256, kEnergyCtas = 4096;

__global__ void __launch_bounds__(kEnergyThreads)
    energy_part_kernel(const LatState *lats, const float *theta, double *part)
{
    __shared__ double red[kEnergyThreads / 32];
    const LatState &st = lats[blockIdx.y];
    const float *th = theta + st.off;
    const int L = st.L, half = st.half, V = 2 * half;
    const int stv[4] = {1, L, L * L, L * L * L};
    double acc = 0.0;
    for (int s = blockIdx.x * kEnergyThreads + threadIdx.x; s < V;
         s += gridDim.x * kEnergyThreads) {
        int x[4];
        x[0] = s % L;
        x[1] = (s / L) % L;
        x[2] = (s / (L * L)) % L;
        x[3] = s / (L * L * L);
        const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
        double t[4];
        int sp[4];
        for (int mu = 0; mu < 4; ++mu) {
            t[mu] = (double)th[(2 * mu + p) * half + (s >> 1)];
            sp[mu] = s + ((x[mu] == L - 1) ? -(L - 1) * stv[mu] : stv[mu]);
        }
        for (int mu = 0; mu < 4; ++mu)
            for (int nu = mu + 1; nu < 4; ++nu) {
                const double b = (double)th[(2 * nu + (p ^ 1)) * half + (sp[mu] >> 1)];
                const double c = (double)th[(2 * mu + (p ^ 1)) * half + (sp[nu] >> 1)];
                acc += cos(((t[mu] + b) - c) - t[nu]);
            }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < kEnergyThreads / 32; ++w) tot += red[w];
        part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
    }
}

// The parts of each lattice (one warp), in a fixed order.
__global__ void __launch_bounds__(32) energy_sum_kernel(const double *part, int n, double *E_out)
{
    double acc = 0.0;
    for (int k = threadIdx.x; k < n; k += 32) acc += part[(size_t)blockIdx.x * n + k];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
    if (threadIdx.x == 0) E_out[blockIdx.x] = acc;
}

__global__ void set_energy_kernel(LatState *lat, const double *E)
{
    lat->E_fx = __double2ll_rn(*E * kFx);
}

__global__ void to_canonical_kernel(const LatState *lat, const float *theta, float *out, int n)
{
    const LatState st = *lat;
    const int V = 2 * st.half, L = st.L;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        const int mu = l / V, s = l - mu * V;
        const int p = (s % L + (s / L) % L + (s / (L * L)) % L + s / (L * L * L)) & 1;
        out[l] = theta[st.off + (size_t)(2 * mu + p) * st.half + (s >> 1)];
    }
}

__global__ void from_canonical_kernel(const LatState *lat, float *theta, const float *in, int n)
{
    const LatState st = *lat;
    const int V = 2 * st.half, L = st.L;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < n; l += gridDim.x * blockDim.x) {
        const int mu = l / V, s = l - mu * V;
        const int p = (s % L + (s / L) % L + (s / (L * L)) % L + s / (L * L * L)) & 1;
        theta[st.off + (size_t)(2 * mu + p) * st.half + (s >> 1)] = in[l];
    }
}

// Shared memory an SM gives to one CTA (227 KB) less the kernel's static part.
constexpr size_t kDynMax = 227 * 1024 - ((sizeof(Smem) + 127) / 128) * 128;

constexpr size_t slab_bytes(int L) { return 16u * (size_t)L * L * L; }
constexpr size_t lattice_bytes(int L) { return slab_bytes(L) * (size_t)L; }
static_assert(slab_bytes(kSlabMaxL) <= kDynMax, "the largest slab fits");

// SMs of the current device, with the kernel's shared-memory limit and
// carve-out preference (percent of the unified L1/shared storage, or -1 for
// the driver's default) set.  Queried once per process, device and carve-out;
// the carve-out is a property of the kernel function in this process, so the
// last one configured applies to every handle that launches it.
template <bool FAST>
int prepare_kernel(int carveout)
{
    static int sms[64] = {};
    static int applied[64] = {};   // carve-out index + 1 last applied per device
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    const int ci = carveout < 0 ? 0 : carveout <= 50 ? 1 : carveout <= 75 ? 2 : 3;
    if (applied[dev] != ci + 1) {
        cudaFuncSetAttribute(llr_kernel<FAST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kDynMax);
        const int pct = ci == 0 ? (int)cudaSharedmemCarveoutDefault : ci == 1 ? 50 : ci == 2 ? 75 : 100;
        cudaFuncSetAttribute(llr_kernel<FAST>, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
        applied[dev] = ci + 1;
    }
    if (sms[dev] == 0) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms[dev] = n > 0 ? n : 1;
    }
    return sms[dev];
}

// Lattices a CTA works on at a time: those that let the launch end soonest.
//
// A CTA takes longer over G lattices than over one, but less than G times as long.
// kGroupTime has what the phases of a composite sweep take for G = 1, 2, 3, 4, 6, in
// percent of the sweep of one (measured with 152 G lattices and windows of width L^2 / 8;
// the rest: four overrelaxation passes and the energy).
//   * L <= 6 leaves most of a CTA idle, so six go in little more than the time of one.
//   * L = 8: up to three are held in shared memory.
//   * L >= 18: the slabs go one or two at a time, and a fourth lattice keeps the
//     heat-bath's schedulers fuller.
// A deciding warp takes 2.75 + 40 / width ns a link (6.0, 9.4 and 12.7 measured at widths
// 12, 6 and 4; 22 in a multicanonical pass): in narrow windows it is the heat-bath's
// bound and company costs less.  The two times are joined by the sum of their cubes.
// A launch of `groups` groups takes ceil(groups / SMs) rounds; of several sweeps, which
// run into one another, half a round more than fills the SMs, but no fewer than the sweeps.
// A larger group has to gain 2 %.
// One sweep of 200 lattices of L = 4 / 8 / 12: 0.247 / 0.613 / 1.97 ms one to a CTA,
// 0.149 / 0.383 / 1.60 ms two to a CTA; six sweeps of 200 of L = 12 7.74 and 9.33 ms; six
// of 608 of L = 16 in windows of 6 54.0 ms three to a CTA, 60.7 ms two.
struct GroupTime {
    int max_L;
    double link;        // ns a link of the sweep of one
    int hb[5], rest[5];
};
constexpr int kGroups[5] = {1, 2, 3, 4, 6};
constexpr GroupTime kGroupTime[] = {
    {4, 98.0, {54, 59, 58, 60, 70}, {46, 43, 49, 48, 67}},
    {6, 37.0, {58, 61, 66, 72, 86}, {42, 50, 52, 57, 69}},
    {8, 18.3, {63, 72, 82, 97, 0}, {37, 47, 57, 163, 0}},
    {10, 12.5, {62, 84, 109, 142, 0}, {38, 96, 122, 196, 0}},
    {12, 12.2, {52, 74, 103, 131, 0}, {48, 88, 107, 178, 0}},
    {16, 10.8, {52, 77, 110, 144, 0}, {48, 77, 109, 178, 0}},
    {18, 11.0, {54, 80, 114, 151, 0}, {46, 81, 138, 163, 0}},
    {kSlabMaxL, 9.7, {56, 82, 120, 154, 0}, {44, 89, 134, 175, 0}},
    {64, 9.7, {56, 82, 120, 0, 0}, {44, 89, 134, 0, 0}},
};

int choose_teams(const LaunchCfg &cfg, const KernelArgs &a, int per_lat, int sms)
{
    if (cfg.threads != 256) {
        // asked for, but no more than the batch has for every SM (152 lattices of
        // L = 8 asked to run six to a CTA: 1.90 ms on 26 SMs, 0.65 ms on all)
        const int most = cfg.threads >= 512 ? 1 : cfg.threads >= 160 ? 4 : 6;
        const int each = (a.n_lat + sms - 1) / sms;
        return each >= most ? most : each == 5 ? 4 : each;
    }
    const GroupTime *t = kGroupTime;
    while (a.max_L > t->max_L) ++t;
    const bool pass = a.program == kProgPass, approach = a.program == kProgApproach;
    const bool muca = a.program == kProgMuca || (pass && a.pass_kind == 2);
    const double heatbath = pass && (a.pass_kind == 1 || a.pass_kind == 3) ? 0.0 : 1.0;
    const double rest = pass ? 1.0 - heatbath : (a.n_or + 0.5) / 4.5;
    // the deciding warp's time, and that in the measured hb
    const double usual = (2.75 + 320.0 / (a.max_L * a.max_L)) / t->link * 100.0;
    const double decide =
        (muca ? 22.0 : 2.75 + (approach ? 0.0 : 40.0 * a.inv_width / a.block)) / t->link * 100.0;
    const double more = std::max(0.0, std::pow(decide, 3) - std::pow(usual, 3));
    const int work = std::min(a.n_lat, a.work);
    int best = 1;
    double least = INFINITY;
    for (int k = 0; k < 5 && t->hb[k] > 0; ++k) {
        const int groups = (work + kGroups[k] - 1) / kGroups[k];
        const double rounds = groups <= sms  ? per_lat
                              : per_lat == 1 ? (groups + sms - 1) / sms
                                             : (double)groups * per_lat / sms + 0.5;
        const double hb = k == 0 ? std::max((double)t->hb[0], decide)
                                 : std::cbrt(std::pow((double)t->hb[k], 3) + more);
        const double time = rounds * (heatbath * hb + rest * t->rest[k]);
        if (time * 1.02 < least) {
            least = time;
            best = kGroups[k];
        }
    }
    return best;
}

template <bool FAST>
cudaError_t launch_t(KernelArgs a, const LaunchCfg &cfg, cudaStream_t s, int *grid_out)
{
    const bool multi = a.program == kProgSweeps || a.program == kProgRM || a.program == kProgMuca;
    const int per_lat = multi ? (a.n_therm + a.n_meas) : 1;
    if ((long long)a.n_lat * per_lat <= 0) return cudaSuccess;
    const int sms = prepare_kernel<FAST>(cfg.carveout);
    a.teams = choose_teams(cfg, a, per_lat, sms);
    // Two stages, where there are barriers for them (15 named ones, two per ring stage
    // of each team).  Four take L1 from the other passes: ten sweeps of 128 of L = 20
    // 63.2 ms, 60.9 with two, 59.7 with one; of L = 12 9.77, 9.66 and 9.85.
    const int most = a.teams <= 3 ? 2 : 1;
    a.ring = cfg.ring < most ? cfg.ring : most;
    const int groups = producers(a.teams);
    const size_t stage1 = (size_t)a.teams * groups * kStageGroupBytes;
    const size_t lattices = (size_t)a.teams * lattice_bytes(a.max_L);
    // a lattice may be resident if a team of the overrelaxation pass has a
    // thread for each of the L^3 / 2 links of a slab's class
    const int links = a.max_L <= kResidentMaxL ? a.max_L * a.max_L * a.max_L / 2 : kThreads;
    const int or_most = links <= kWarps / a.teams * 32 ? a.teams : std::min(a.teams, 3);
    // A launch that only sums energies reads every angle a few times and writes none:
    // lattices stay where they are (2000 of L = 4 / 8: 66 / 217 us copied in, 58 / 169).
    const bool sums = a.program == kProgResync || a.program == kProgFinish ||
                      a.program == kProgBegin || a.program == kProgUpdate ||
                      (a.program == kProgPass && a.pass_kind == 3);
    a.resident = !sums && a.max_L <= kResidentMaxL && lattices + stage1 <= kDynMax &&
                 links <= kWarps / or_most * 32;
    while (a.resident && lattices + stage1 * a.ring > kDynMax) a.ring >>= 1;
    size_t rings = stage1 * a.ring;
    size_t dyn;
    if (a.resident) {
        a.or_teams = or_most;
        a.slab = (int)(lattice_bytes(a.max_L) / sizeof(float));
        a.ring_off = (int)(lattices / sizeof(float));
        dyn = lattices + rings;
    } else if (sums) {
        a.or_teams = 1;
        a.slab = a.ring_off = 0;
        dyn = 0;
    } else {
        const size_t slab = a.slab_L > 0 ? slab_bytes(a.slab_L) : 0;
        const size_t stage = (size_t)kStaged * kThreads * sizeof(float2);
        while (a.ring > 1 && stage + stage1 * a.ring > kDynMax) a.ring >>= 1;
        rings = stage1 * a.ring;
        // lattices read in place go one by one, which leaves each the L1 (a sweep
        // of 304 of L = 28: 56 ms against 82 ms two at a time)
        a.or_teams = a.max_L > kSlabMaxL ? 1 : std::min(a.teams, 3);
        while (a.or_teams > 1 && slab * a.or_teams > kDynMax) --a.or_teams;
        a.slab = (int)(slab / sizeof(float));
        a.ring_off = (int)(stage / sizeof(float));
        dyn = std::max(stage + rings, slab * a.or_teams);
    }
    const long long items = (long long)((a.n_lat + a.teams - 1) / a.teams) * per_lat;
    const int grid = (int)(items < sms ? items : sms);
    if (grid_out) *grid_out = grid;
    // the item counter and the done counters; the error word sync[0] is left
    // alone (sticky until the host reads and clears it)
    cudaError_t e = cudaMemsetAsync(a.sync + 1, 0, sizeof(unsigned) * (size_t)(1 + a.n_lat), s);
    if (e != cudaSuccess) return e;
    llr_kernel<FAST><<<grid, kThreads, dyn, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

void prime_launch(const LaunchCfg &cfg)
{
    cfg.fast_math ? prepare_kernel<true>(cfg.carveout) : prepare_kernel<false>(cfg.carveout);
}

cudaError_t launch_llr(const KernelArgs &args, const LaunchCfg &cfg, cudaStream_t s, int *grid_out)
{
    if (args.n_lat <= 0) return cudaSuccess;
    return cfg.fast_math ? launch_t<true>(args, cfg, s, grid_out)
                         : launch_t<false>(args, cfg, s, grid_out);
}

__global__ void step_increment_kernel(int *step)
{
    *step += 1;
}

cudaError_t launch_step_increment(int *step, cudaStream_t s)
{
    step_increment_kernel<<<1, 1, 0, s>>>(step);
    return cudaGetLastError();
}

cudaError_t launch_hot_start(LatState *lats, float *theta, int n_lat, int max_half,
                             cudaStream_t s)
{
    if (n_lat <= 0) return cudaSuccess;
    const int n = 8 * max_half;
    dim3 grid((unsigned)((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024), (unsigned)n_lat);
    hot_start_kernel<<<grid, 256, 0, s>>>(lats, theta);
    return cudaGetLastError();
}

size_t energy_parts(int n_lat)
{
    return (size_t)std::max(n_lat, kEnergyCtas);
}

cudaError_t launch_energy_fp64(const LatState *lats, const float *theta, int n_lat, int max_half,
                               double *part, double *E_out, cudaStream_t s)
{
    if (n_lat <= 0) return cudaSuccess;
    // two sites per thread, no more CTAs in all than fill the GPU a few times over
    const int tiles = (2 * max_half + 2 * kEnergyThreads - 1) / (2 * kEnergyThreads);
    const int ctas = std::max(1, std::min(tiles, kEnergyCtas / n_lat));
    // lattices along the grid's second dimension, 65535 at most a launch
    for (int i = 0; i < n_lat; i += 65535) {
        const int m = std::min(n_lat - i, 65535);
        energy_part_kernel<<<dim3(ctas, m), kEnergyThreads, 0, s>>>(lats + i, theta,
                                                                   part + (size_t)i * ctas);
    }
    energy_sum_kernel<<<n_lat, 32, 0, s>>>(part, ctas, E_out);
    return cudaGetLastError();
}

cudaError_t launch_set_energy(LatState *lat_dev, const double *E_dev, cudaStream_t s)
{
    set_energy_kernel<<<1, 1, 0, s>>>(lat_dev, E_dev);
    return cudaGetLastError();
}

cudaError_t launch_to_canonical(const LatState *lat_dev, const float *theta, float *out,
                                int n_links, cudaStream_t s)
{
    to_canonical_kernel<<<(n_links + 255) / 256, 256, 0, s>>>(lat_dev, theta, out, n_links);
    return cudaGetLastError();
}

cudaError_t launch_from_canonical(const LatState *lat_dev, float *theta, const float *in,
                                  int n_links, cudaStream_t s)
{
    from_canonical_kernel<<<(n_links + 255) / 256, 256, 0, s>>>(lat_dev, theta, in, n_links);
    return cudaGetLastError();
}

}  // namespace llr
