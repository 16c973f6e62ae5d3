// llr_recon.cu -- FP64 reconstruction of ln rho and of action observables
// from the Robbins-Monro slopes a_k.
//
// Paper: Langfeld, Lucini, Pellegrini, Rago (arXiv:1509.08391).
//   eqs. (2.6), (2.7)  ln rho(c_{k+1}) - ln rho(c_k) = (c_{k+1} - c_k) (a_k + a_{k+1}) / 2
//   eqs. (2.46), (2.47)    Z(beta) = sum_k w rho(c_k) e^{beta c_k},
//                    <E^m> = sum_k w c_k^m rho(c_k) e^{beta c_k} / Z
//   Sec. 3.4         C_V = <E^2> - <E>^2, beta_c at its maximum
//   Sec. 2.6, eq. (2.56)   multicanonical reweighting: a sample E_i of the run
//                    with weight 1/rho~ carries exp(beta E_i + ln rho~(E_i));
//                    tunnellings of a chain between the ends of the range
//
// Sizes are small (hundreds to thousands of intervals): one CTA scans ln rho, one
// CTA per coupling forms the log-sum-exp observables, and the C_V peak is a grid
// scan and a golden-section search on the device, many couplings at once.
#include <algorithm>
#include <climits>
#include <cmath>
#include <string>

#include "../../include/llr.h"
#include "llr_internal.h"

// Scratch of llr_observables_noalloc: ln rho at up to LLR_NOALLOC_MAX_CENTRES
// interval centres, in a fixed device array that every GPU loading this
// library holds until the process exits.  Host code must not pass the symbol
// itself to a kernel (on the host it names a host-side stand-in); it uses the
// device address that cudaGetSymbolAddress returns.
static __device__ __align__(256) double g_noalloc_lnrho[LLR_NOALLOC_MAX_CENTRES];

namespace llr {
namespace {

constexpr int kT = 256;
constexpr unsigned kFull = 0xffffffffu;

__device__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < kT / 32; ++w) t += red[w];
    return t;
}

__device__ double block_max(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(kFull, v, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = red[0];
    for (int w = 1; w < kT / 32; ++w) t = fmax(t, red[w]);
    return t;
}

// Inclusive block scan of the trapezium increments, chunk by chunk.
__device__ void lnrho_scan(int n, const double *c, const double *a, double *out)
{
    __shared__ double buf[kT];
    __shared__ double carry;
    if (threadIdx.x == 0) carry = 0.0;
    __syncthreads();
    for (int base = 0; base < n; base += kT) {
        const int k = base + threadIdx.x;
        // increment arriving at centre k (0 for k = 0)
        double inc = 0.0;
        if (k > 0 && k < n) inc = 0.5 * (c[k] - c[k - 1]) * (a[k - 1] + a[k]);
        buf[threadIdx.x] = inc;
        __syncthreads();
        for (int o = 1; o < kT; o <<= 1) {
            const double y = threadIdx.x >= o ? buf[threadIdx.x - o] : 0.0;
            __syncthreads();
            buf[threadIdx.x] += y;
            __syncthreads();
        }
        if (k < n) out[k] = carry + buf[threadIdx.x];
        __syncthreads();
        if (threadIdx.x == 0) carry += buf[kT - 1];
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kT) lnrho_kernel(int n, const double *c, const double *a,
                                                   double *out)
{
    lnrho_scan(n, c, a, out);
}

// (ln Z, <E>, <E^2>) at coupling beta; ln rho given.  Every thread returns them.
__device__ void moments_at(int n, const double *c, const double *lr, double beta, double *red,
                           double &lnZ, double &E1, double &E2)
{
    double m = -INFINITY;
    for (int k = threadIdx.x; k < n; k += kT) m = fmax(m, lr[k] + beta * c[k]);
    m = block_max(m, red);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int k = threadIdx.x; k < n; k += kT) {
        const double e = exp(lr[k] + beta * c[k] - m);
        s0 += e;
        s1 += c[k] * e;
        s2 += c[k] * c[k] * e;
    }
    s0 = block_sum(s0, red);
    s1 = block_sum(s1, red);
    s2 = block_sum(s2, red);
    const double w = n > 1 ? (c[n - 1] - c[0]) / (double)(n - 1) : 1.0;
    lnZ = m + log(w * s0);
    E1 = s1 / s0;
    E2 = s2 / s0;
}

__global__ void __launch_bounds__(kT) observables_kernel(int n, const double *c,
                                                         const double *lr, const double *beta,
                                                         double *lnZ, double *E1, double *E2)
{
    __shared__ double red[kT / 32];
    double z, e1, e2;
    moments_at(n, c, lr, beta[blockIdx.x], red, z, e1, e2);
    if (threadIdx.x == 0) {
        lnZ[blockIdx.x] = z;
        E1[blockIdx.x] = e1;
        E2[blockIdx.x] = e2;
    }
}

__device__ double cv_at(int n, const double *c, const double *lr, double beta, double *red)
{
    double z, e1, e2;
    moments_at(n, c, lr, beta, red, z, e1, e2);
    return e2 - e1 * e1;
}

// C_V at the grid point of every block.
__global__ void __launch_bounds__(kT) cv_grid_kernel(int n, const double *c, const double *lr,
                                                     double blo, double bhi, int n_grid,
                                                     double *cv)
{
    __shared__ double red[kT / 32];
    const int i = blockIdx.x;
    const double b = n_grid > 1 ? blo + (bhi - blo) * (double)i / (double)(n_grid - 1) : blo;
    const double v = cv_at(n, c, lr, b, red);
    if (threadIdx.x == 0) cv[i] = v;
}

// Golden-section search on the device.  One evaluation is a chain of exps and
// block reductions on one SM (8 us at 512 centres, mostly FP64 latency), and a
// step needs the comparison before it, so the steps are taken several at a
// time: a round evaluates the points of all outcomes of the next comparisons at
// once, one block each, and the next round replays the comparisons on the
// values found.  512 centres, 1601 grid points, tol 1e-10 (26 steps): a call takes
// 15.6 ms with one block for everything, 0.47 ms with the grid in parallel and 5
// rounds.
constexpr int kFirstDepth = 6, kDepth = 7;            // comparisons ahead per round
constexpr int kFirstNodes = 2 + 2 * ((1 << kFirstDepth) - 1);   // x1, x2, a tree per outcome
constexpr int kNodes = (1 << kDepth) - 1;             // one tree: the first outcome is known
constexpr int kMaxSteps = 200;

struct Golden {
    double lo, hi, x1, x2, f1, f2;
    int it;
    __device__ bool open(double tol) const { return it < kMaxSteps && hi - lo > tol; }
    // narrow the interval by the outcome of f1 < f2; returns the new point
    __device__ double step(bool less)
    {
        const double g = 0.6180339887498949;   // (sqrt 5 - 1) / 2
        ++it;
        if (less) {
            lo = x1;
            x1 = x2;
            f1 = f2;
            x2 = lo + g * (hi - lo);
            return x2;
        }
        hi = x2;
        x2 = x1;
        f2 = f1;
        x1 = hi - g * (hi - lo);
        return x1;
    }
};

// The search's state after `rounds` rounds, whose values are F[round][node]; the
// start from the best of the grid values cv (the first of the largest).
__device__ Golden golden_replay(const double *cv, double blo, double bhi, int n_grid, double tol,
                                const double *F, int rounds)
{
    __shared__ double bv[kT / 32];
    __shared__ int bi[kT / 32];
    double v = -INFINITY;
    int best = n_grid;
    for (int i = threadIdx.x; i < n_grid; i += kT)
        if (cv[i] > v) {
            v = cv[i];
            best = i;
        }
    for (int o = 16; o > 0; o >>= 1) {
        const double w = __shfl_xor_sync(kFull, v, o);
        const int j = __shfl_xor_sync(kFull, best, o);
        if (w > v || (w == v && j < best)) {
            v = w;
            best = j;
        }
    }
    if ((threadIdx.x & 31) == 0) {
        bv[threadIdx.x >> 5] = v;
        bi[threadIdx.x >> 5] = best;
    }
    __syncthreads();
    for (int w = 0; w < kT / 32; ++w)
        if (bv[w] > v || (bv[w] == v && bi[w] < best)) {
            v = bv[w];
            best = bi[w];
        }
    if (best == n_grid) best = 0;   // no value above -inf
    Golden s;
    const double step = n_grid > 1 ? (bhi - blo) / (double)(n_grid - 1) : 0.0;
    s.lo = blo + step * (double)(best > 0 ? best - 1 : 0);
    s.hi = blo + step * (double)(best < n_grid - 1 ? best + 1 : n_grid - 1);
    const double g = 0.6180339887498949;
    s.x1 = s.hi - g * (s.hi - s.lo);
    s.x2 = s.lo + g * (s.hi - s.lo);
    s.f1 = s.f2 = 0.0;
    s.it = 0;
    for (int r = 0; r < rounds; ++r, F += kFirstNodes) {
        if (r == 0) {
            s.f1 = F[0];
            s.f2 = F[1];
        }
        const double *tree = F + (r > 0 ? 0 : s.f1 < s.f2 ? 2 + kFirstNodes / 2 - 1 : 2);
        const int depth = r > 0 ? kDepth : kFirstDepth;
        int node = 1;
        for (int d = 0; d < depth && s.open(tol); ++d) {
            const bool less = s.f1 < s.f2;
            if (d > 0) node = 2 * node + less;
            s.step(less);
            (less ? s.f2 : s.f1) = tree[node - 1];
        }
    }
    return s;
}

// Round `round`: block k evaluates node k.  In a tree, node 1 is the point after
// the first comparison, nodes 2 m and 2 m + 1 those after node m's comparison
// came out not less / less.
__global__ void __launch_bounds__(kT) golden_round_kernel(int n, const double *c, const double *lr,
                                                          double blo, double bhi, int n_grid,
                                                          double tol, const double *cv,
                                                          double *F, int round)
{
    __shared__ double red[kT / 32];
    Golden s = golden_replay(cv, blo, bhi, n_grid, tol, F, round);
    int node = blockIdx.x + 1;
    bool less = s.f1 < s.f2;
    double x;
    if (round == 0 && blockIdx.x < 2) {
        x = blockIdx.x == 0 ? s.x1 : s.x2;
    } else {
        if (round == 0) {
            node = blockIdx.x - 2;
            less = node >= kFirstNodes / 2 - 1;
            node = node % (kFirstNodes / 2 - 1) + 1;
        }
        if (!s.open(tol)) return;
        x = s.step(less);
        for (int bit = 31 - __clz(node) - 1; bit >= 0; --bit) {
            if (!s.open(tol)) return;   // a point the search never asks for
            x = s.step((node >> bit) & 1);
        }
    }
    const double v = cv_at(n, c, lr, x, red);
    if (threadIdx.x == 0) F[(size_t)round * kFirstNodes + blockIdx.x] = v;
}

__global__ void __launch_bounds__(kT) golden_result_kernel(int n, const double *c, const double *lr,
                                                           double blo, double bhi, int n_grid,
                                                           double tol, const double *cv,
                                                           const double *F, int rounds,
                                                           double *out)
{
    __shared__ double red[kT / 32];
    const Golden s = golden_replay(cv, blo, bhi, n_grid, tol, F, rounds);
    const double b = 0.5 * (s.lo + s.hi);
    const double v = cv_at(n, c, lr, b, red);
    if (threadIdx.x == 0) {
        out[0] = b;
        out[1] = v;
    }
}

// Rounds that are sure to reach the tolerance (two steps of slack for rounding), or,
// for one below a few units in the last place of the couplings, the width at which
// the interval stops shrinking (the steps a longer search would add leave its
// middle where it is).
int golden_rounds(double blo, double bhi, int n_grid, double tol)
{
    const double len = 2.0 * (bhi - blo) / (double)(n_grid - 1);
    int steps = kMaxSteps;
    if (tol > 0.0 && std::isfinite(len / tol))
        steps = (int)std::min<double>(
            kMaxSteps, std::max(0.0, std::ceil(std::log(len / tol) / 0.48121182505960347)) + 2.0);
    return 1 + std::max(0, (steps - kFirstDepth + kDepth - 1) / kDepth);
}

// ---------------------------------------------------------------------------
// Multicanonical reweighting (Sec. 2.6, eq. (2.56)).  The moments at beta are
// log-space sums over all samples; they run over d = E - shift (shift = the
// table start, close to the samples), so that <E^2> - <E>^2 keeps its digits.

// ln rho~ of eq. (2.10) at E: lnr[k] = ln rho~(e0 + k de), slope a[k] on
// [e0 + k de, e0 + (k + 1) de), the first / last slope beyond the table.
__device__ __forceinline__ double lnrho_piecewise(const double *lnr, const double *a, int n,
                                                  double e0, double de, double E)
{
    const double q = fmin(fmax(floor((E - e0) / de), 0.0), (double)(n - 1));
    const int k = (int)q;
    return lnr[k] + a[k] * (E - (e0 + (double)k * de));
}

__global__ void __launch_bounds__(kT) muca_lnrho_kernel(long long ns, const double *E,
                                                        const double *lnr, const double *a,
                                                        int n, double e0, double de,
                                                        double *out)
{
    const long long stride = (long long)gridDim.x * kT;
    for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < ns; i += stride)
        out[i] = lnrho_piecewise(lnr, a, n, e0, de, E[i]);
}

// Exponents of any size (the table form below takes those within 2^39).
// Block (x, y): coupling beta[y] over the samples of kT-wide tiles x,
// x + gridDim.x, ...  Each thread keeps a running maximum m of the exponent
// and rescales its sums when it grows; the block then brings its threads to
// the block maximum M.  Writes (M, s0, s1, s2), s_j = sum d^j exp(x - M).
__global__ void __launch_bounds__(kT) reweight_partial_kernel(long long ns, const double *E,
                                                              const double *lr, double shift,
                                                              const double *beta, double *part)
{
    __shared__ double red[kT / 32];
    const double b = beta[blockIdx.y];
    double m = -INFINITY, s0 = 0.0, s1 = 0.0, s2 = 0.0;
    const long long stride = (long long)gridDim.x * kT;
    for (long long i = (long long)blockIdx.x * kT + threadIdx.x; i < ns; i += stride) {
        const double e_i = E[i];
        const double x = b * e_i + lr[i];
        if (x > m) {
            const double r = exp(m - x);      // 0 on a thread's first sample
            s0 *= r;
            s1 *= r;
            s2 *= r;
            m = x;
        }
        const double w = exp(x - m);
        const double d = e_i - shift;
        s0 += w;
        s1 += d * w;
        s2 += d * d * w;
    }
    const double M = block_max(m, red);
    const double r = m == -INFINITY ? 0.0 : exp(m - M);
    s0 = block_sum(s0 * r, red);
    s1 = block_sum(s1 * r, red);
    s2 = block_sum(s2 * r, red);
    if (threadIdx.x == 0) {
        double *p = part + 4 * ((size_t)blockIdx.y * gridDim.x + blockIdx.x);
        p[0] = M;
        p[1] = s0;
        p[2] = s1;
        p[3] = s2;
    }
}

// The same for NB couplings a block, with the exponentials by table (Tang, "Table-
// driven implementation of the exponential function in IEEE floating-point
// arithmetic", 1989): exp(y) = 2^(k / 2048) (1 + r + r^2 / 2 + r^3 / 6) with k the
// integer nearest 2048 y / ln 2 and |r| <= ln 2 / 4096 the rest of y (r^4 / 24 <
// 4e-17).  The kernel is bound by the FP64 pipe (1.6 operations per clock and
// SM), so everything that need not be FP64 is not: k's power of two goes into the
// exponent field, and the sums' scale is an exact power of two, found and kept as
// an integer.  12 FP64 operations per sample and coupling (87 % of the pipe's time)
// where the library's exp and the running maximum took about twice as many, and
// fewer, longer blocks: a coupling of 512000 samples among 300 50 us -> 15 us.  The exponent
// is formed over d = E - shift, whose rounding is smaller than E's.  Writes
// (N, s0, s1, s2), s_j = sum d^j exp(b d + lr) / 2^N.
constexpr int kExpBits = 11, kExpTable = 1 << kExpBits;
constexpr long long kNoTerm = -(1ll << 62);   // the scale before the first term

__global__ void __launch_bounds__(kT) exp_table_kernel(double *tab)
{
    const int j = blockIdx.x * kT + threadIdx.x;
    if (j < kExpTable) tab[j] = exp2((double)j / kExpTable);
}

// 2^-d, d >= 0, from the exponent field (0 below the normal numbers).
__device__ __forceinline__ double pow2_down(long long d)
{
    return d < 1022 ? __hiloint2double((1023 - (int)d) << 20, 0) : 0.0;
}

// Sums of n values over a warp, every value in the order of a xor butterfly; a
// step hands half of the values to each half of the lanes, so 12 values take 13
// additions and not 60 (the FP64 pipe is the kernel's bound).  Returns which value
// the lane's v[0] is the sum of (n or more: none; one lane for every value).
template <int n, int o = 16>
__device__ __forceinline__ int warp_sums(double *v, int lane)
{
    if constexpr (o == 0) {
        return 0;
    } else if constexpr (n == 1) {
        v[0] += __shfl_xor_sync(kFull, v[0], o);
        const int at = warp_sums<1, o / 2>(v, lane);
        return (lane & o) ? 1 : at;   // one lane answers
    } else {
        constexpr int h = (n + 1) / 2;
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double other = i + h < n ? v[i + h] : 0.0;
            const double give = up ? v[i] : other, keep = up ? other : v[i];
            v[i] = keep + __shfl_xor_sync(kFull, give, o);
        }
        const int at = warp_sums<h, o / 2>(v, lane);
        return at < h && at + (up ? h : 0) < n ? at + (up ? h : 0) : n;
    }
}

// Part x of the samples: tiles x, x + parts, ...  A block takes parts blockIdx.x,
// blockIdx.x + gridDim.x, ... for its couplings.  The parts are set by the number of
// samples alone and each is summed in an order of its own, so a coupling's result
// does not depend on how many are asked for with it.
template <int NB>
__global__ void __launch_bounds__(kT) reweight_table_kernel(long long ns, int parts,
                                                            const double *E, const double *lr,
                                                            double shift, int n_beta,
                                                            const double *beta,
                                                            const double *tab, double *part)
{
    __shared__ double T[kExpTable];
    static_assert(kT / 32 == 8 && (NB == 1 || NB == 4), "the first warp has a lane for each sum");
    __shared__ long long redN[2][8][NB];
    __shared__ double redS[2][8][3 * NB];
    constexpr double kMagic = 6755399441055744.0;   // 1.5 2^52: rounds to an integer in the low bits
    constexpr double kInv = 2954.639443740597;     // 2048 / ln 2
    constexpr double kHi = 3.384507717577858e-4;   // ln 2 / 2048, and what its rounding leaves
    constexpr double kLo = 1.1323470770733885e-20;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = threadIdx.x; j < kExpTable; j += kT) T[j] = tab[j];
    const int b0 = blockIdx.y * NB;
    double b[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) b[q] = beta[min(b0 + q, n_beta - 1)];
    __syncthreads();
    const long long stride = (long long)parts * kT;
    for (int x = blockIdx.x, buf = 0; x < parts; x += gridDim.x, buf ^= 1) {
        double s0[NB], s1[NB], s2[NB];
        long long N[NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            s0[q] = s1[q] = s2[q] = 0.0;
            N[q] = kNoTerm;
        }
        for (long long i = (long long)x * kT + threadIdx.x; i < ns; i += stride) {
            const double d = E[i] - shift, l = lr[i], d2 = d * d;
#pragma unroll
            for (int q = 0; q < NB; ++q) {
                const double y = fma(b[q], d, l);
                const double kd = fma(y, kInv, kMagic);
                const double kf = kd - kMagic;
                const double r = fma(kf, -kLo, fma(kf, -kHi, y));
                const long long k = __double_as_longlong(kd) - 0x4338000000000000ll;
                const long long n = k >> kExpBits;   // power of two
                if (n > N[q]) {   // a larger term than any before: rescale, rarely
                    const double f = pow2_down(n - N[q]);
                    s0[q] *= f;
                    s1[q] *= f;
                    s2[q] *= f;
                    N[q] = n;
                }
                const double t = T[(int)k & (kExpTable - 1)];
                double w = fma(t, r * fma(r, fma(r, 1.0 / 6.0, 0.5), 1.0), t);   // in [1, 2)
                const long long down = N[q] - n;
                w = down < 1000 ? __hiloint2double(__double2hiint(w) - ((int)down << 20),
                                                   __double2loint(w))
                                : 0.0;
                s0[q] += w;
                s1[q] = fma(d, w, s1[q]);
                s2[q] = fma(d2, w, s2[q]);
            }
        }
        // the block's sums: within the warps, then over them
        double v[3 * NB];
#pragma unroll
        for (int q = 0; q < NB; ++q) {
            long long M = N[q];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) M = max(M, __shfl_xor_sync(kFull, M, o));
            const double f = pow2_down(M - N[q]);
            v[3 * q] = s0[q] * f;
            v[3 * q + 1] = s1[q] * f;
            v[3 * q + 2] = s2[q] * f;
            if (lane == 0) redN[buf][warp][q] = M;
        }
        const int at = warp_sums<3 * NB>(v, lane);
        if (at < 3 * NB) redS[buf][warp][at] = v[0];
        __syncthreads();
        // lane 8 q + w of the first warp: warp w's sums of coupling q.  The other warps
        // go on to the next part, which has the other buffer.
        const int q = lane >> 3, w = lane & 7;
        if (warp == 0 && q < NB) {
            const unsigned lanes = NB == 4 ? kFull : (1u << (8 * NB)) - 1u;
            const long long n = redN[buf][w][q];
            long long M = n;
            for (int o = 4; o > 0; o >>= 1) M = max(M, __shfl_xor_sync(lanes, M, o));
            const double f = pow2_down(M - n);
            double t[3];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                t[m] = redS[buf][w][3 * q + m] * f;
                for (int o = 4; o > 0; o >>= 1) t[m] += __shfl_xor_sync(lanes, t[m], o);
            }
            if (w == 0 && b0 + q < n_beta) {
                double *p = part + 4 * ((size_t)(b0 + q) * parts + x);
                p[0] = (double)M;
                p[1] = t[0];
                p[2] = t[1];
                p[3] = t[2];
            }
        }
    }
}

// One block per coupling: combine the gx partials of reweight_partial_kernel or
// (pow2) reweight_table_kernel.  E1 = <E>, var = <E^2> - <E>^2, E2 = <E^2> (any of
// them may be null).
__global__ void __launch_bounds__(kT) reweight_combine_kernel(int gx, const double *part,
                                                              bool pow2, double shift, double *E1,
                                                              double *E2, double *var)
{
    __shared__ double red[kT / 32];
    const double *p = part + 4 * (size_t)blockIdx.x * gx;
    double m = -INFINITY;
    for (int j = threadIdx.x; j < gx; j += kT) m = fmax(m, p[4 * j]);
    m = block_max(m, red);
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int j = threadIdx.x; j < gx; j += kT) {
        const double mj = p[4 * j];
        if (mj == -INFINITY) continue;        // a block without samples
        const double r = pow2 ? exp2(mj - m) : exp(mj - m);
        s0 += r * p[4 * j + 1];
        s1 += r * p[4 * j + 2];
        s2 += r * p[4 * j + 3];
    }
    s0 = block_sum(s0, red);
    s1 = block_sum(s1, red);
    s2 = block_sum(s2, red);
    if (threadIdx.x == 0) {
        const double u = s1 / s0, v = s2 / s0 - u * u, e1 = shift + u;
        if (E1) E1[blockIdx.x] = e1;
        if (var) var[blockIdx.x] = v;
        if (E2) E2[blockIdx.x] = e1 * e1 + v;
    }
}

// Tunnellings of each chain (Sec. 2.6): E[t][c] in time order t; a passage
// from E < lo to E > hi or back counts once.  One thread per chain, the
// loads of a time step coalesced across chains.
__global__ void __launch_bounds__(kT) tunnelling_kernel(int n_steps, int n_chains,
                                                        const double *E, double lo, double hi,
                                                        int *out)
{
    const int c = blockIdx.x * kT + threadIdx.x;
    if (c >= n_chains) return;
    int count = 0, last = 0;
    for (int t = 0; t < n_steps; ++t) {
        const double e = E[(size_t)t * n_chains + c];
        if (e < lo) {
            count += last == 1;
            last = -1;
        } else if (e > hi) {
            count += last == -1;
            last = 1;
        }
    }
    out[c] = count;
}

}  // namespace

cudaError_t launch_muca_lnrho(long long ns, const double *E, const double *lnr, const double *a,
                              int n, double e0, double de, double *out, int grid,
                              cudaStream_t s)
{
    muca_lnrho_kernel<<<grid, kT, 0, s>>>(ns, E, lnr, a, n, e0, de, out);
    return cudaGetLastError();
}

size_t reweight_table_doubles()
{
    return kExpTable;
}

cudaError_t launch_reweight_table(double *tab, cudaStream_t s)
{
    exp_table_kernel<<<kExpTable / kT, kT, 0, s>>>(tab);
    return cudaGetLastError();
}

cudaError_t launch_reweight(long long ns, const double *E, const double *lr, double shift,
                            int n_beta, const double *beta, const double *tab, int gx,
                            int wave, double *part, double *E1, double *E2, double *var, cudaStream_t s)
{
    if (n_beta <= 0) return cudaSuccess;
    constexpr int NB = 4;   // couplings a block: samples and table are read once for all
    if (tab && n_beta >= NB) {
        // one wave over all couplings: a block's table costs as much as some hundred
        // samples
        const int groups = (n_beta + NB - 1) / NB;
        const int bx = std::max(1, std::min(gx, wave / groups));
        reweight_table_kernel<NB><<<dim3(bx, groups), kT, 0, s>>>(ns, gx, E, lr, shift, n_beta,
                                                                 beta, tab, part);
    }
    else if (tab)
        reweight_table_kernel<1><<<dim3(gx, n_beta), kT, 0, s>>>(ns, gx, E, lr, shift, n_beta,
                                                                 beta, tab, part);
    else
        reweight_partial_kernel<<<dim3(gx, n_beta), kT, 0, s>>>(ns, E, lr, shift, beta, part);
    reweight_combine_kernel<<<n_beta, kT, 0, s>>>(gx, part, tab != nullptr, shift, E1, E2, var);
    return cudaGetLastError();
}

cudaError_t launch_tunnellings(int n_steps, int n_chains, const double *E, double lo, double hi,
                               int *out, cudaStream_t s)
{
    tunnelling_kernel<<<(n_chains + kT - 1) / kT, kT, 0, s>>>(n_steps, n_chains, E, lo, hi, out);
    return cudaGetLastError();
}

cudaError_t launch_lnrho(int n, const double *c, const double *a, double *out, cudaStream_t s)
{
    lnrho_kernel<<<1, kT, 0, s>>>(n, c, a, out);
    return cudaGetLastError();
}

cudaError_t launch_observables(int n, const double *c, const double *lr, int n_beta,
                               const double *beta, double *lnZ, double *E1, double *E2,
                               cudaStream_t s)
{
    if (n_beta <= 0) return cudaSuccess;
    observables_kernel<<<n_beta, kT, 0, s>>>(n, c, lr, beta, lnZ, E1, E2);
    return cudaGetLastError();
}

size_t cv_peak_scratch(int n_grid, double beta_lo, double beta_hi, double tol)
{
    return (size_t)n_grid + (size_t)kFirstNodes * golden_rounds(beta_lo, beta_hi, n_grid, tol);
}

cudaError_t launch_cv_peak(int n, const double *c, const double *lr, double beta_lo,
                           double beta_hi, int n_grid, double tol, double *scratch, double *out,
                           cudaStream_t s)
{
    double *cv = scratch, *F = scratch + n_grid;
    const int rounds = golden_rounds(beta_lo, beta_hi, n_grid, tol);
    cv_grid_kernel<<<n_grid, kT, 0, s>>>(n, c, lr, beta_lo, beta_hi, n_grid, cv);
    for (int r = 0; r < rounds; ++r)
        golden_round_kernel<<<r > 0 ? kNodes : kFirstNodes, kT, 0, s>>>(
            n, c, lr, beta_lo, beta_hi, n_grid, tol, cv, F, r);
    golden_result_kernel<<<1, kT, 0, s>>>(n, c, lr, beta_lo, beta_hi, n_grid, tol, cv, F, rounds,
                                          out);
    return cudaGetLastError();
}

}  // namespace llr

namespace {

// Device address of the scratch array in the current device's context,
// looked up on every call (a cheap table lookup once the module is loaded):
// a cached address would dangle after the context is destroyed and created
// again (cudaDeviceReset, or the primary context released and retained).
int noalloc_scratch(double **out)
{
    void *p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_lnrho);
    if (e != cudaSuccess || !p)
        return llr::set_last_error(LLR_ERR_CUDA, (std::string("cudaGetSymbolAddress: ") +
                                                  cudaGetErrorString(e)).c_str());
    *out = (double *)p;
    return LLR_OK;
}

}  // namespace

extern "C" int llr_observables_noalloc(int n, const double *centres, const double *a,
                                       int n_beta, const double *beta, double *lnZ_out,
                                       double *E_out, double *E2_out, void *cuda_stream)
{
    if (n < 1 || n > LLR_NOALLOC_MAX_CENTRES)
        return llr::set_last_error(LLR_ERR_ARG, ("n must be in 1.." +
                                                 std::to_string(LLR_NOALLOC_MAX_CENTRES) +
                                                 " for llr_observables_noalloc").c_str());
    if (n_beta < 1 || !centres || !a || !beta || !lnZ_out || !E_out || !E2_out)
        return llr::set_last_error(LLR_ERR_ARG, "null device buffer or n_beta < 1");
    double *scratch = nullptr;
    if (int r = noalloc_scratch(&scratch)) return r;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // every call writes ln rho at all n centres before the observables read
    // them, so the scratch needs no clearing between calls
    cudaError_t e = llr::launch_lnrho(n, centres, a, scratch, s);
    if (e == cudaSuccess)
        e = llr::launch_observables(n, centres, scratch, n_beta, beta, lnZ_out, E_out, E2_out, s);
    if (e != cudaSuccess)
        return llr::set_last_error(LLR_ERR_CUDA, (std::string("launch: ") +
                                                  cudaGetErrorString(e)).c_str());
    return LLR_OK;
}
