// Eigensolver of the mode Grams (Alg. 1 step 3) on a thread-block cluster: pivoted Cholesky G = L L^T, then
// one-sided (Hestenes) Jacobi on the columns of L.
//
//  1. Pivoted Cholesky of G = Z Z^T is the column-pivoted QR of Z^T (L = R^T up to the row order), the
//     preconditioning step of Drmac and Veselic's one-sided Jacobi SVD, after which few sweeps are needed.  It ends
//     when what is left cannot matter for this mode's truncation (FP32: 1% of the budget, FP64: 1e-10 of it) or is
//     rounding noise of the Gram.  The trace of the remainder is energy the truncation discards, and is counted so.
//  2. Plane rotations from the right make the columns of L orthogonal, L J = U Sigma: the normalised columns are
//     eigenvectors of G and their squared norms its eigenvalues, and no rotation matrix is accumulated.
//  3. The columns lie in shared memory in 2 Ce blocks of b, two blocks per CTA of the cluster.  In a round every CTA
//     rotates all b^2 pairs of one column of each of its blocks, b disjoint pairs at a time (a warp to a pair; the
//     top block's columns stay in registers), then the blocks move by the circle method through distributed shared
//     memory.  2 Ce - 1 rounds and the pairs inside the blocks make a sweep in which every pair meets once.  The
//     cluster waits for itself once a round, not once a step.
//
// What bounds it: a chain of about rc steps a sweep (5 to 7 sweeps), each a dot product, its
// reduction, the rotation's parameters and the rotation.  In FP64 the arithmetic: an FP64 instruction of a warp takes
// its quarter of the SM 64 cycles, dependent or not, so a step costs what one quarter issues (13 + 4 M / 32
// instructions for one pair).  Hence one pair per quarter, on as many CTAs as the columns fill so; shears with three
// FMAs an element; everything that only steers the iteration in FP32; and no rotation of pairs far below the budget.
// Measured, FP64, a Gram of order 120 and full rank: 1.5 ms (16 CTAs), where the two-sided cyclic Jacobi on 8 CTAs that
// this replaces took 18 ms at order 97; order 32: 0.19 ms against 0.8 ms.  FP32, where a step is latency and instructions
// (0.3 us with 16-byte accesses and paired FMAs, 0.45 us without): order 128 and rank 45 0.14 ms, where a ring of columns in
// one CTA's registers with a barrier a step took 0.43 ms.
#include <math.h>

#include <string>
#include <type_traits>

#include <cooperative_groups.h>

#include "common.cuh"
#include "device.cuh"
#include "eig.cuh"
#include "recip.cuh"

namespace tpcg {

namespace cgx = cooperative_groups;

// A pair is orthogonal once |a_p . a_q| <= tau |a_p| |a_q|.  FP32: the dot product itself resolves about 4e-7 at 128
// rows.  FP64: at 2e-13 the truncated tensors were up to five times further from the 64-bit ones than at 1e-14, in
// the same time.
//
// A rotation of p and q by theta gives the product (p, r) the part sin(theta) (q, r), so what a sweep leaves behind is at
// most its largest cosine times its largest sine.  It is the last one when its cosines were all below `last` and its
// |u| = |tan(theta / 2)| all below `turn`: 2 turn last = 2e-14 (FP64) and 9e-6 (FP32) may stay.  The cosines alone say
// nothing where norms nearly coincide: there a cosine of 1e-10 turns by 45 degrees (with that rule the kept vectors of triples of
// singular values 1e-9 apart were orthonormal to 2e-10 in place of 1e-14, in FP32 to 4e-4; the flags cost the FP32 step 2.5%).
// FP32: wide turns do not count in a sweep whose cosines were all below `rest`, which may stay; pairs of equal norm would
// go on turning on the rounding of their products.
template <typename T>
__host__ __device__ constexpr T hj_tau() { return sizeof(T) == 8 ? T(1e-14) : T(5e-7); }
template <typename T>
__host__ __device__ constexpr T hj_last() { return sizeof(T) == 8 ? T(1e-8) : T(1.5e-3); }
template <typename T>
__host__ __device__ constexpr float hj_turn() { return sizeof(T) == 8 ? 1e-6f : 3e-3f; }
constexpr float HJ_REST = 3e-6f;

// what a sweep met: a large cosine (or, FP64, a wide turn); FP32: a wide turn, a cosine above HJ_REST; steered by FP32 and
// to be steered again
constexpr int HJ_LARGE = 1, HJ_TURN = 2, HJ_ABOVE = 4, HJ_AGAIN = 8;

// The sweep after one that met a cosine above this is steered in FP32 (46 us in place of 75 us at order 97).  Below it the
// products that FP32 leaves count: at 1e-3 most Grams took a sweep more (order 97: 550 us, 521 us at 2e-2, 554 us unsteered;
// order 32 188 us, 187 us and 213 us; three Grams of order 64 in a sum 703, 690 and 779 us).
constexpr float HJ_STEER = 2e-2f;

// Shape of a launch: C CTAs, a warp to a pair of columns, RPL rows a lane (orders up to 32 RPL), BT pairs a CTA takes at a
// time before another CTA joins.
template <typename T_, int C_, int RPL_, int BT_>
struct HjShape {
    using T = T_;
    static constexpr int C = C_, RPL = RPL_, BT = BT_;
    static constexpr int ROWS = 32 * RPL;
    static constexpr int BMAX = (ROWS / C + 1) / 2;              // columns of the largest block, pairs at once
    static constexpr int NT = BMAX * 32 > 128 ? BMAX * 32 : 128;
    // two sets of two blocks of columns; the Cholesky's own columns lie in the second set
    static constexpr size_t SMEM = (size_t)4 * BMAX * ROWS * sizeof(T);
};

__device__ __forceinline__ double hj_warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// This lane's rows of a column at a: rows lane + 32 q, the first rpl of them; in FP32 the four rows 4 lane + q in one 16-byte
// access (all of them: rows past the order are zero, and an FP32 FMA is cheaper than a test)
template <typename T, int RPL>
constexpr bool hj_vec = sizeof(T) == 4 && RPL == 4;
template <typename T, int RPL>
__device__ __forceinline__ void hj_load(T (&x)[RPL], const T* a, int lane, int rpl) {
    if constexpr (hj_vec<T, RPL>) {
        const float4 v = *reinterpret_cast<const float4*>(a + 4 * lane);
        x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
    } else {
#pragma unroll
        for (int q = 0; q < RPL; ++q)
            if (q < rpl) x[q] = a[lane + 32 * q];
    }
}
template <typename T, int RPL>
__device__ __forceinline__ void hj_save(const T (&x)[RPL], T* a, int lane, int rpl) {
    if constexpr (hj_vec<T, RPL>) {
        *reinterpret_cast<float4*>(a + 4 * lane) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
#pragma unroll
        for (int q = 0; q < RPL; ++q)
            if (q < rpl) a[lane + 32 * q] = x[q];
    }
}

// One pair, by a whole warp: x and y are this lane's rows of the two columns, ax and ay their squared norms.  A pair with
// |x . y| above tau |x| |y| is rotated: u = tan(theta / 2), s = sin(theta), applied as the shears x -= u y, y += s x,
// x -= u y (three FMAs an element).  The angle needs no more than FP32: an error of 1e-6 in it leaves 1e-6 of the product
// for the next sweep; s = 2 u / (1 + u^2) has the working precision, so that the shears make an orthogonal matrix.
//
// STEER (FP64, the first sweeps): everything but the shears and s in FP32 as well, the dot product and the norms included.
// Their error of 1e-6 |x| |y| stays for the sweeps that follow, and an FP64 step of 17 instructions at 32 rows becomes one of 8.
template <typename T, int RPL, bool STEER = false>
__device__ __forceinline__ void hj_pair(T (&x)[RPL], T (&y)[RPL], T& ax, T& ay, int rpl, T skip, T floor_g, int& big) {
    T g = T(0);
    if constexpr (hj_vec<T, RPL>) {
        const float2 g2 = __ffma2_rn(make_float2(x[2], x[3]), make_float2(y[2], y[3]),
                                     __fmul2_rn(make_float2(x[0], x[1]), make_float2(y[0], y[1])));
        g = g2.x + g2.y;
    } else if constexpr (!STEER) {
#pragma unroll
        for (int q = 0; q < RPL; ++q)
            if (q < rpl) g = fma(x[q], y[q], g);
    }
    if constexpr (!STEER) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    }
    float fa, fb, fg, fd;   // |x|^2, |y|^2, x . y, |y|^2 - |x|^2
    int off = 0;
    bool on;
    float g0 = 0.f, a0 = 0.f, b0 = 0.f;   // STEER: product and norms before the scaling
    if constexpr (STEER) {
#pragma unroll
        for (int q = 0; q < RPL; ++q)
            if (q < rpl) g0 = fmaf(bits_to_float(x[q]), bits_to_float(y[q]), g0);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g0 += __shfl_xor_sync(0xffffffffu, g0, o);
        a0 = bits_to_float(ax);
        b0 = bits_to_float(ay);
        const float sc = __int_as_float(0x7f000000 - (__float_as_int(fmaxf(a0, b0)) & 0x7f800000));   // larger norm to [1, 2)
        fa = a0 * sc;
        fb = b0 * sc;
        fg = g0 * sc;
        fd = fb - fa;
        const int hs = __double2hiint(skip);
        on = fa > 0.f && fb > 0.f && (__double2hiint(ax) > hs || __double2hiint(ay) > hs);
    } else if constexpr (sizeof(T) == 8) {   // by a power of two near the larger norm: nothing that counts leaves FP32's range
        const int hx = __double2hiint(ax), hy = __double2hiint(ay), hs = __double2hiint(skip);
        off = (max(hx, hy) >> 20) - 1023;
        fa = bits_to_float(ax, off);
        fb = bits_to_float(ay, off);
        fg = bits_to_float(g, off);
        fd = bits_to_float(ay - ax, off);
        on = hx > hs || hy > hs;      // both far below the budget: all discarded, whatever their products
    } else {
        fa = ax;
        fb = ay;
        fg = g;
        fd = ay - ax;
        on = fabsf(g) > floor_g;
    }
    // t = tan(theta) = 2 g / (d + sign(d) sqrt(d^2 + 4 g^2)); u = t / (1 + sqrt(1 + t^2)), its series in t^2 fitted on
    // [0, 1] to 2e-6.  Formed beside the test, not after it.
    const float ab = fa * fb, ag = fabsf(fg), f2g = 2.f * fg;
    const float h = fmaf(fd, fd, f2g * f2g);
    const float t = __fdividef(f2g, fd + copysignf(h * rsqrtf(h), fd));
    const float w = t * t;
    const float u = t * fmaf(w, fmaf(w, fmaf(w, fmaf(w, fmaf(w, -0.00342296f, 0.0151217f), -0.03403639f), 0.06147052f),
                             -0.12491905f), 0.49999894f);
    bool above, large;
    if constexpr (STEER) {
        const float cs = ag * rsqrtf(fa) * rsqrtf(fb);
        above = cs > 2e-6f;
        large = cs > HJ_STEER;
    } else if constexpr (sizeof(T) == 8) {
        const float rab = ab > 0.f ? ab * rsqrtf(ab) : 0.f;
        above = ag > (float)hj_tau<T>() * rab;
        large = ag > (float)hj_last<T>() * rab;
    } else {
        above = ag * ag > hj_tau<T>() * hj_tau<T>() * ab;
        large = ag * ag > hj_last<T>() * hj_last<T>() * ab;
    }
    if (on && above && (sizeof(T) == 4 || fabsf(u) > 1e-30f)) {
        if (large || (sizeof(T) == 8 && !STEER && fabsf(u) > hj_turn<T>())) big |= HJ_LARGE;
        if (sizeof(T) == 4 && fabsf(u) > hj_turn<T>()) big |= HJ_TURN;
        if (sizeof(T) == 4 && ag * ag > HJ_REST * HJ_REST * ab) big |= HJ_ABOVE;
        T ud, s;
        if constexpr (sizeof(T) == 8) {
            ud = bits_to_double(u);
            const double u2 = bits_to_double(2.f * u);
            if (fabsf(u) < 1e-4f && fabsf(u) > 1e-15f) {   // 2 u (1 - u^2) to u^4
                s = fma(-u2, bits_to_double(u * u), u2);
            } else {
                const float qf = fmaf(u, u, 1.f);
                s = u2 * recip_from(fma(ud, ud, 1.0), bits_to_double(__fdividef(1.f, qf)));
            }
        } else {
            ud = u;
            const float q = fmaf(u, u, 1.f);
            s = 2.f * u * recip_from(q, __fdividef(1.f, q));
        }
        if constexpr (hj_vec<T, RPL>) {
            const float2 mu = make_float2(-u, -u), s2 = make_float2(s, s);
#pragma unroll
            for (int q = 0; q < 4; q += 2) {
                float2 yq = make_float2(y[q], y[q + 1]);
                const float2 x1 = __ffma2_rn(mu, yq, make_float2(x[q], x[q + 1]));
                yq = __ffma2_rn(s2, x1, yq);
                const float2 xq = __ffma2_rn(mu, yq, x1);
                x[q] = xq.x; x[q + 1] = xq.y;
                y[q] = yq.x; y[q + 1] = yq.y;
            }
        } else {
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (q < rpl) {
                    const T x1 = fma(-ud, y[q], x[q]);
                    y[q] = fma(s, x1, y[q]);
                    x[q] = fma(-ud, y[q], x1);
                }
        }
        const float tg = t * fg;   // the norms are exact again at the next sweep
        if constexpr (STEER) {
            ax = bits_to_double(fmaxf(a0 - t * g0, 0.f));
            ay = bits_to_double(fmaxf(b0 + t * g0, 0.f));
        } else if constexpr (sizeof(T) == 8) {
            if (fabsf(tg) > 1e-30f) {
                const double v = bits_to_double(tg, off);
                ax -= v;
                ay += v;
            }
        } else {
            ax -= tg;
            ay += tg;
        }
    }
}

// Truncation rule on the decreasingly sorted eigenvalues lam[0..M) (as truncation_rule in eig.cu, sums by one warp).
// FP64: the smallest s whose discarded (clamped) eigenvalues, the remainder `rem` and, in strict mode, the rounding
// uncertainty `unc` of each stay within the budget.  FP32: trace minus the kept eigenvalues.  Returns s before the
// cap, and in *disc a table of the discarded energy by s (M + 1 entries of shared memory).
template <typename T>
__device__ int hj_rule(const double* lam, int M, double trace, double rem, double unc, double budget, double* disc) {
    const int lane = threadIdx.x & 31;
    const int per = (M + 31) / 32, lo = min(lane * per, M), hi = min(lo + per, M);
    double own = 0.0;
    for (int i = lo; i < hi; ++i) own += lam[i] > 0.0 ? lam[i] : 0.0;
    int cnt = 0;   // FP64: entries that can be discarded; FP32: kept counts that are not enough
    if (sizeof(T) == 8) {
        double after = own;   // sum over this lane's and the later lanes' entries
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_down_sync(0xffffffffu, after, o);
            if (lane + o < 32) after += v;
        }
        double t = __shfl_down_sync(0xffffffffu, after, 1);
        t = (lane < 31 ? t : 0.0) + rem;
        if (lane == 31) disc[M] = rem;
        for (int i = hi - 1; i >= lo; --i) {
            t += lam[i] > 0.0 ? lam[i] : 0.0;
            disc[i] = t;
            if (t + unc * (double)(M - i) <= budget) ++cnt;
        }
    } else {
        double before = own;
        for (int o = 1; o < 32; o <<= 1) {
            const double v = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += v;
        }
        double t = __shfl_up_sync(0xffffffffu, before, 1);
        t = trace - (lane > 0 ? t : 0.0);
        for (int i = lo; i < hi; ++i) {   // i kept
            disc[i] = t > 0.0 ? t : 0.0;
            if (!(t <= budget)) ++cnt;
            t -= lam[i];
        }
        if (hi == M && (lo < M || M == 0)) disc[M] = t > 0.0 ? t : 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    return sizeof(T) == 8 ? M - cnt : cnt;
}

template <typename SH>
__global__ void __launch_bounds__(SH::NT, 1)
    hj_eig_kernel(RoundPlan* plan, const typename SH::T* __restrict__ G, typename SH::T* __restrict__ S, double* evals,
                  int m, int max_sweeps, double* prof) {
    using T = typename SH::T;
    constexpr int C = SH::C, RPL = SH::RPL, ROWS = SH::ROWS, LD = ROWS, BMAX = SH::BMAX, NT = SH::NT;
    constexpr int NQ = 2 * BMAX;                    // columns of G per CTA (Cholesky)
    constexpr unsigned FULL = 0xffffffffu;
    static_assert(NQ <= 32, "one lane per column in the search for the pivot");
    cgx::cluster_group cluster = cgx::this_cluster();
    const int crank = (int)cluster.block_rank();
    RoundPlan& p = *plan;
    const int M = p.eM, n = p.n;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    extern __shared__ __align__(16) unsigned char hj_raw[];
    T* cols = reinterpret_cast<T*>(hj_raw);          // [set][block][position] columns, ld LD
    __shared__ T nrm[2][2][BMAX];                    // squared norms of the columns, moving with them
    __shared__ T lbuf[2][ROWS];
    __shared__ int s_key[2][C], s_idx[2][C];         // candidate pivots of every CTA, by parity of the step
    __shared__ float s_left[2][C];                   // and what is left of the trace on it
    __shared__ double s_piv[2][C], dg[NQ];           // their values; remaining diagonal of this CTA's columns
    __shared__ int dg0[NQ];                          // leading bits of what counts as noise there
    __shared__ float dgf[sizeof(T) == 4 ? ROWS : 1];
    __shared__ double dga[sizeof(T) == 8 && RPL == 1 ? ROWS : 1];   // the whole remaining diagonal
    __shared__ short piv_of[ROWS];
    __shared__ int s_flags[2][C];
    __shared__ double s_red[32], s_rem, lam[ROWS], lsort[ROWS], disc[ROWS + 1];
    __shared__ double s_tr, s_budget, s_bus;
    __shared__ T s_trs;
    __shared__ int s_exp;
    __shared__ short ord[ROWS];
    __shared__ unsigned char pivoted[ROWS];
    __shared__ int s_keep, s_nz;
    if (M <= 0) {
        if (crank == 0 && tid == 0) {
            p.s[m] = 0;
            if (m == 0) { p.norm2 = 0; p.budget = 0; }
        }
        return;
    }
    // ---- trace, budget, and the power of two that brings the trace near 1 (FP32 products of squared norms would
    // leave the exponent's range for small tensors)
    if (warp == 0) {
        double t = 0.0;
        for (int i = lane; i < M; i += 32) t += (double)G[i + (long long)i * M];
        t = hj_warp_sum(t);
        if (lane == 0) {
            s_tr = t;
            // m > 0: the budget of the first mode's kernel; m = 0: every CTA computes it, CTA 0 stores it below
            const double n2 = p.rr ? p.gtrace : t;
            const double bu = m == 0 ? fmax(p.eps * p.eps * n2, p.abs2) * (1.0 / 3.0) : p.budget;
            const int lim = sizeof(T) == 4 ? 120 : 1000;
            const int k = t > 0.0 ? max(-lim, min(lim, 1023 - ((__double2hiint(t) >> 20) & 0x7ff))) : 0;
            s_budget = bu;
            s_exp = k;
            s_trs = (T)(t * __hiloint2double((1023 + k) << 20, 0));
            s_bus = bu * __hiloint2double((1023 + k) << 20, 0);
        }
    }
    __syncthreads();
    const double trace = p.rr ? p.gtrace : s_tr;     // what the rule works with
    const double budget = s_budget;
    const double unc = sizeof(T) == 8 && p.strict ? 4.0 * 2.220446049250313e-16 * trace : 0.0;
    const bool finite = isfinite(s_tr) && isfinite(trace);
    const int cap = p.cap;
    // Nothing can be discarded (a strict rule whose budget is below the uncertainty of one eigenvalue) and nothing is
    // clipped, or there is nothing to decompose (NaN, Inf: kept as it is, so that the scalars built on it show it):
    // any orthonormal basis serves, and the identity leaves the tensor unchanged.
    if (!finite || (sizeof(T) == 8 && unc > budget && (cap <= 0 || M <= cap))) {
        const int s = cap > 0 && M > cap ? cap : M;
        for (long long e = (long long)crank * NT + tid; e < (long long)M * s; e += (long long)C * NT) {
            const int i = (int)(e % M), c = (int)(e / M);
            S[i + (long long)c * n] = (i == c) ? T(1) : T(0);
        }
        cluster.sync();   // every CTA has read the plan
        if (crank == 0 && tid == 0) {
            if (m == 0) { p.norm2 = trace; p.budget = budget; }
            p.s[m] = s;
        }
        return;
    }
    const T sc = sizeof(T) == 8 ? (T)__hiloint2double((1023 + s_exp) << 20, 0) : (T)__int_as_float((127 + s_exp) << 23);
    const double unscale = __hiloint2double((1023 - s_exp) << 20, 0);
    const double bus = s_bus;   // the budget on that scale
    const T tr = s_trs;
    const int rpl = (M + 31) / 32;
    // ---- 1. pivoted Cholesky.  How the columns of L are spread over the cluster depends on their number: they wait in
    // shared memory (FP64) or in S (FP32)
    int rc = 0;
    if constexpr (sizeof(T) == 8 && RPL == 1) {
        // Up to 32 rows every CTA factorises the whole Gram in its registers, row `lane` and columns warp + NW q (the columns
        // spread over the cluster cost a barrier of the cluster a step, more than their FMAs)
        constexpr int NW = NT / 32, NA = ROWS / NW;
        double Ar[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) {
            const int j = warp + NW * q;
            Ar[q] = lane < M && j < M ? G[lane + (long long)j * M] * sc : 0.0;
        }
        const double d0 = lane < M ? G[lane + (long long)lane * M] * sc : -1.0;
        // an entry below 8 u of what the Gram had there is rounding noise and no candidate
        const int noise = __double2hiint(fmax(8 * 1.1102230246251565e-16 * d0, 1e-30));
        if (warp == 0) dga[lane] = d0;
        __syncthreads();
        const float stop_rem = (float)(1e-10 * bus);
        unsigned gone = 0;   // pivoted rows and columns
        for (int k = 0; k < M; ++k) {
            const double d = dga[lane];   // remaining diagonal, -1 once pivoted
            const int hi = __double2hiint(d);
            const int key = hi > noise ? hi : -1;
            const int best = __reduce_max_sync(FULL, key);
            const int piv = __ffs(__ballot_sync(FULL, key == best)) - 1;
            float left = hi > 0 ? bits_to_float(d) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) left += __shfl_xor_sync(FULL, left, o);
            if (best < 0 || !(left > stop_rem)) break;   // the same in every thread of the cluster
            double* lk = lbuf[k & 1];
            if (warp == piv % NW) {
                double a = 0.0;
#pragma unroll
                for (int q = 0; q < NA; ++q) a = q == piv / NW ? Ar[q] : a;
                a = gone >> lane & 1 ? 0.0 : a;
                lk[lane] = a;
                if (k % C == crank) cols[(k / C) * LD + lane] = a;
            }
            // A -= a a^T / d of the column a as it is; the scaling of L's column waits until it is read back
            const double dp = __shfl_sync(FULL, d, piv);
            const double invd = recip_mid(dp);
            gone |= 1u << piv;
            if (tid == 0) {
                piv_of[k] = (short)piv;
                lam[k] = dp;
            }
            __syncthreads();
            const double li = -lk[lane] * invd;
#pragma unroll
            for (int q = 0; q < NA; ++q) {
                const int j = warp + NW * q;
                if (j >= M || (gone >> j & 1)) continue;
                Ar[q] = fma(li, lk[j], Ar[q]);
                if (lane == j) dga[j] = Ar[q];
            }
            if (tid == 0) dga[piv] = -1.0;
            __syncthreads();
            rc = k + 1;
        }
        if (warp == 0) {   // energy outside the columns of L
            const double d = dga[lane];
            const double t = hj_warp_sum(d > 0.0 ? d : 0.0);
            if (lane == 0) s_rem = t * unscale;
        }
        cluster.sync();   // columns complete
    } else if constexpr (sizeof(T) == 8) {
        // The columns of G are spread over the cluster, column j in CTA j mod C, and every step waits for the cluster
        // once.
        T* A = cols + 2 * BMAX * LD;                     // what other CTAs read; the own columns are in registers as well
        constexpr int RT = (ROWS + NT - 1) / NT, CT = RT == 1 && NT > ROWS ? NT / ROWS : 1, QT = (NQ + CT - 1) / CT;
        const int row = CT > 1 ? tid % ROWS : tid, cg = CT > 1 ? tid / ROWS : 0;   // rows row + NT a, columns cg + CT q
        double Ar[RT][QT];
#pragma unroll
        for (int q = 0; q < QT; ++q) {
            const int cq = cg + CT * q, j = crank + C * cq;
#pragma unroll
            for (int a = 0; a < RT; ++a) {
                const int i = row + NT * a;
                Ar[a][q] = i < M && j < M ? G[i + (long long)j * M] * sc : T(0);
                if (cq < NQ && i < ROWS) A[cq * LD + i] = Ar[a][q];
            }
        }
        for (int q = tid; q < NQ; q += NT) {
            const int j = crank + C * q;
            const T d = j < M ? G[j + (long long)j * M] * sc : T(-1);
            dg[q] = d;
            // an entry below 8 u of what the Gram had there is rounding noise and no candidate
            dg0[q] = __double2hiint(fmax(8 * 1.1102230246251565e-16 * d, 1e-30));
        }
        bool alive[RT];
#pragma unroll
        for (int a = 0; a < RT; ++a) alive[a] = row + NT * a < M;
        cluster.sync();   // everybody is in place: remote writes may begin
        const float stop_rem = (float)(1e-10 * bus);
        for (int k = 0; k < M; ++k) {
            const int par = k & 1;
            if (warp == 0) {
                // this CTA's candidate: the largest remaining diagonal entry by its leading bits (ties: the first)
                const double d = lane < NQ ? dg[lane] : -1.0;
                const int hi = __double2hiint(d);
                const int key = lane < NQ && hi > dg0[lane] ? hi : -1;
                const int best = __reduce_max_sync(FULL, key);
                const int who = __ffs(__ballot_sync(FULL, key == best)) - 1;
                const double dm = __shfl_sync(FULL, d, who);
                if (lane < C) {
                    cluster.map_shared_rank(&s_key[par][0], lane)[crank] = best;
                    cluster.map_shared_rank(&s_idx[par][0], lane)[crank] = who;
                    cluster.map_shared_rank(&s_piv[par][0], lane)[crank] = dm;
                }
            } else if (warp == 1) {   // what is left of the trace
                const double d = lane < NQ ? dg[lane] : -1.0;
                float left = __double2hiint(d) > 0 ? bits_to_float(d) : 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) left += __shfl_xor_sync(FULL, left, o);
                if (lane < C) cluster.map_shared_rank(&s_left[par][0], lane)[crank] = left;
            }
            cluster.sync();
            const int ky = lane < C ? s_key[par][lane] : -1;
            float left = lane < C ? s_left[par][lane] : 0.f;
            const int best = __reduce_max_sync(FULL, ky);
            const int own = __ffs(__ballot_sync(FULL, ky == best)) - 1;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) left += __shfl_xor_sync(FULL, left, o);
            left = __shfl_sync(FULL, left, 0);
            if (best < 0 || !(left > stop_rem)) break;   // the same in every thread of the cluster
            const int q0 = s_idx[par][own], piv = own + C * q0;
            // Column a = A[:, piv] as it is, and 1 / d: A -= a a^T / d.  The scaling of L's column waits until it is read
            // back.  The owner leaves the column alone from here on, so it is read where it lies.
            const T* src = cluster.map_shared_rank(A, own) + q0 * LD;
            T col[RT];
#pragma unroll
            for (int a = 0; a < RT; ++a) col[a] = alive[a] ? src[row + a * NT] : T(0);
            const double d = s_piv[par][own];
            const double invd = recip_mid(d);
            T* lk = lbuf[par];
            T* out = k % C == crank ? cols + (k / C) * LD : nullptr;   // (a store to global memory here makes the barrier wait)
#pragma unroll
            for (int a = 0; a < RT; ++a) {
                const int i = row + a * NT;
                if (cg == 0 && i < ROWS) {
                    lk[i] = col[a];
                    if (out) out[i] = col[a];
                }
                if (i == piv) alive[a] = false;
                col[a] *= -invd;
            }
            if (tid == 0) {
                piv_of[k] = (short)piv;
                lam[k] = d;
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < QT; ++q) {
                const int cq = cg + CT * q, j = crank + C * cq;
                if (cq >= NQ || j >= M) break;
                const T lj = lk[j];   // zero for the columns of earlier pivots
                if (__double2hiint(lj) == 0 || j == piv) continue;
#pragma unroll
                for (int a = 0; a < RT; ++a) {
                    const int i = row + a * NT;
                    Ar[a][q] = fma(col[a], lj, Ar[a][q]);
                    if (i < ROWS) A[cq * LD + i] = Ar[a][q];
                    if (i == j) dg[cq] = Ar[a][q];
                }
            }
            if (own == crank && tid == 0) dg[q0] = T(-1);
            __syncthreads();
            rc = k + 1;
        }
        // energy outside the columns of L
        if (warp == 0) {
            const double d = lane < NQ && dg[lane] > T(0) ? (double)dg[lane] : 0.0;
            const double t = hj_warp_sum(d);
            if (lane < C) cluster.map_shared_rank(&s_red[0], lane)[crank] = t;
        }
        cluster.sync();   // columns complete, remote reads done
        if (tid == 0) {
            double t = 0.0;
            for (int r = 0; r < C; ++r) t += s_red[r];
            s_rem = t * unscale;
        }
    } else {
        // FP32 arithmetic is cheaper than the cluster's barrier: every CTA factorises the whole Gram, held in registers
        // (entry (i, j) with j = warp + NW a, i = lane + 32 b), and keeps its own columns
        constexpr int NW = NT / 32, NA = ROWS / NW, NB = ROWS / 32;
        static_assert(NW == 16, "two columns of a warp to a row block");
        float Ar[NA][NB];
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const int i = lane + 32 * b, j = warp + NW * a;
                Ar[a][b] = (i < M && j < M) ? G[i + (long long)j * M] * sc : 0.f;
            }
        for (int i = tid; i < ROWS; i += NT) dgf[i] = i < M ? G[i + (long long)i * M] * sc : 0.f;
        __syncthreads();
        const float thr = 1e-9f * tr;
        const float stop_rem = fmaxf(thr, 0.01f * (float)bus);
        unsigned dead_row = 0, dead_col = 0;   // pivoted ones among this lane's rows (bit b) and this warp's columns (bit a)
        for (int k = 0; k < M; ++k) {
            // the largest remaining diagonal entry (ties: the lowest index) and the remaining trace, in every warp
            float v = -2.f, sm = 0.f;
            int bi = 0;
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const float d = dgf[lane + 32 * b];
                if (d > v) { v = d; bi = lane + 32 * b; }
                sm += fmaxf(d, 0.f);
            }
            const int key = v > thr ? __float_as_int(v) : -1;
            const int best = __reduce_max_sync(FULL, key);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sm += __shfl_xor_sync(FULL, sm, o);
            const int piv = __reduce_min_sync(FULL, key == best ? bi : ROWS);
            if (best < 0 || !(sm > stop_rem)) break;   // the same decision in every thread and CTA
            float* lk = lbuf[k & 1];
            if (warp == piv % NW) {
                // l = A[:, piv] / sqrt(d), zero on the rows of earlier pivots.  (An IEEE square root and divisions here kept
                // the other warps waiting for 1000 of 2500 cycles a step.)
                const float d = __int_as_float(best), inv = rsqrt_from(d, rsqrtf(d));
                const int ap = piv / NW;
                float* out = k % C == crank ? S + (long long)k * n : nullptr;
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    float a = 0.f;
#pragma unroll
                    for (int q = 0; q < NA; ++q) a = (q == ap) ? Ar[q][b] : a;
                    const int i = lane + 32 * b;
                    a = dead_row >> b & 1 ? 0.f : a * inv;
                    lk[i] = a;
                    if (out && i < M) out[i] = a;
                }
                dead_col |= 1u << ap;
            }
            if (lane == (piv & 31)) dead_row |= 1u << (piv >> 5);
            __syncthreads();
            float li[NB];
#pragma unroll
            for (int b = 0; b < NB; ++b) li[b] = lk[lane + 32 * b];
#pragma unroll
            for (int a = 0; a < NA; ++a) {
                const int j = warp + NW * a;
                const float lj = lk[j];
#pragma unroll
                for (int b = 0; b < NB; ++b) Ar[a][b] = fmaf(-li[b], lj, Ar[a][b]);
                // column j's diagonal is in register b = a / 2 of one lane (0 once pivoted)
                if (lane == warp + NW * (a & 1)) dgf[j] = dead_col >> a & 1 ? 0.f : Ar[a][a >> 1];
            }
            __syncthreads();
            rc = k + 1;
        }
        cluster.sync();   // columns complete; everybody is in place: remote writes may begin
    }
    // ---- 2. one-sided Jacobi
    // Ce CTAs of the cluster take part, as few as give every CTA BT pairs at a time: column k is in CTA k mod Ce, block
    // (k / Ce) & 1, position k / (2 Ce).  The others only wait with the cluster.
    const int Ce = max(1, min(C, (rc + 2 * SH::BT - 1) / (2 * SH::BT)));
    const int b = crank < Ce ? max(1, ((rc + Ce - 1) / Ce + 1) / 2) : 0;
    int set = sizeof(T) == 8 ? 1 : 0, nsweeps = 0;
    for (int e = tid; e < 2 * b * ROWS; e += NT) {
        const int i = e % ROWS, slot = e / ROWS, k = slot * Ce + crank;
        T v = T(0);
        if constexpr (sizeof(T) == 8) {   // from where the Cholesky left it, scaled by the pivot (kept by every CTA)
            if (k < rc) v = cluster.map_shared_rank(cols, k % C)[(k / C) * LD + i] * rsqrt(lam[k]);
        } else {
            if (k < rc && i < M) v = S[i + (long long)k * n];
        }
        cols[((2 * set + (slot & 1)) * BMAX + (slot >> 1)) * LD + i] = v;
    }
    if constexpr (sizeof(T) == 8) cluster.sync();   // read by everybody before the blocks move
    else __syncthreads();
    // FP64, plain rule: pairs whose squared norms are both below 1e-3 budget / M are left as they are, since all such columns
    // together are discarded, in any basis of them.  Not so where the energy outside the columns takes the budget by itself
    // (a budget below the Gram's rounding, a poor Ritz basis): then nothing is discarded, and what is kept is made orthogonal.
    T skip = T(0);
    if constexpr (sizeof(T) == 8) {
        const double outside = s_rem + (p.rr ? fmax(trace - s_tr, 0.0) + 4e-16 * (double)M * trace : 0.0);
        if (!p.strict && outside < 0.5 * budget) skip = 1e-3 * bus * (double)__fdividef(1.f, (float)M);
    }
    const T floor_g = sizeof(T) == 8 ? T(0) : T(1e-12f) * tr;   // FP32 products below this are noise of the factor
    auto column = [&](int set, int blk, int pos) -> T* { return cols + ((set * 2 + blk) * BMAX + pos) * LD; };
    T x[RPL], y[RPL];
    bool steer = sizeof(T) == 8;
    for (int sweep = 0; sweep < max_sweeps && rc > 1; ++sweep) {
        ++nsweeps;
        int big = 0;   // HJ_* of this thread's rotations
        for (int blk = 0; blk < 2; ++blk) {   // exact squared norms
            T s = T(0);
            if (warp < b) {
                hj_load<T, RPL>(x, column(set, blk, warp), lane, rpl);
#pragma unroll
                for (int q = 0; q < RPL; ++q)
                    if (q < rpl || hj_vec<T, RPL>) s = fma(x[q], x[q], s);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
            if (warp < b && lane == 0) nrm[set][blk][warp] = s;
        }
        __syncthreads();
        // pairs inside the two blocks (round robin on b rounded up to even players)
        const int be = (b + 1) & ~1;
        for (int step = 0; step < be - 1; ++step) {
            const int half = be / 2;
            const int blk = warp / half, k = warp - blk * half;
            int i = -1, j = -1;
            if (blk < 2) {
                const int P = be - 1;
                if (k == 0) { i = P; j = step; }
                else {
                    i = step + k; if (i >= P) i -= P;
                    j = step - k; if (j < 0) j += P;
                }
                if (i > j) { const int t = i; i = j; j = t; }
                if (j >= b) i = -1;
            }
            if (i >= 0) {
                T* xp = column(set, blk, i);
                T* yp = column(set, blk, j);
                T ax = nrm[set][blk][i], ay = nrm[set][blk][j];
                hj_load<T, RPL>(x, xp, lane, rpl);
                hj_load<T, RPL>(y, yp, lane, rpl);
                if (sizeof(T) == 8 && steer) hj_pair<T, RPL, sizeof(T) == 8>(x, y, ax, ay, rpl, skip, floor_g, big);
                else hj_pair<T, RPL>(x, y, ax, ay, rpl, skip, floor_g, big);
                hj_save<T, RPL>(x, xp, lane, rpl);
                hj_save<T, RPL>(y, yp, lane, rpl);
                if (lane == 0) { nrm[set][blk][i] = ax; nrm[set][blk][j] = ay; }
            }
            __syncthreads();
        }
        for (int round = 0; round < 2 * Ce - 1; ++round) {
            const bool act = warp < b;   // (b is 0 where the CTA has no columns)
            T ax = T(0);
            if (act) {
                hj_load<T, RPL>(x, column(set, 0, warp), lane, rpl);
                ax = nrm[set][0][warp];
            }
            int j = warp;
            T* yp = column(set, 1, act ? warp : 0);
            for (int k = 0; k < b; ++k) {
                if (act) {
                    T ay = nrm[set][1][j];
                    hj_load<T, RPL>(y, yp, lane, rpl);
                    if (sizeof(T) == 8 && steer) hj_pair<T, RPL, sizeof(T) == 8>(x, y, ax, ay, rpl, skip, floor_g, big);
                    else hj_pair<T, RPL>(x, y, ax, ay, rpl, skip, floor_g, big);
                    hj_save<T, RPL>(y, yp, lane, rpl);
                    if (lane == 0) nrm[set][1][j] = ay;
                    ++j;
                    yp += LD;
                    if (j == b) { j = 0; yp -= b * LD; }
                }
                __syncthreads();
            }
            if (round == 2 * Ce - 2) {   // what this sweep met, told to every CTA
                int tell = __syncthreads_or(big & HJ_LARGE) ? HJ_LARGE : 0;
                if constexpr (sizeof(T) == 4) {
                    if (__syncthreads_or(big & HJ_TURN)) tell |= HJ_TURN;
                    if (__syncthreads_or(big & HJ_ABOVE)) tell |= HJ_ABOVE;
                } else if (steer) {
                    tell = tell ? HJ_LARGE | HJ_AGAIN : HJ_LARGE;   // a steered sweep is never the last one
                }
                if (tid < C && crank < Ce) cluster.map_shared_rank(&s_flags[sweep & 1][0], tid)[crank] = tell;
            }
            if (Ce == 1) {
                if (act) {
                    hj_save<T, RPL>(x, column(set, 0, warp), lane, rpl);
                    if (lane == 0) nrm[set][0][warp] = ax;
                }
                cluster.sync();
                continue;
            }
            // circle method on the 2 Ce blocks: the top blocks move right (the first stays), the bottom blocks left
            const int ns = set ^ 1;
            const int tc = crank == 0 ? 0 : (crank == Ce - 1 ? Ce - 1 : crank + 1);
            const int tb = crank == 0 ? 0 : (crank == Ce - 1 ? 1 : 0);
            const int bc = crank == 0 ? 1 : crank - 1, bb = crank == 0 ? 0 : 1;
            if (act) {
                hj_save<T, RPL>(x, cluster.map_shared_rank(cols, tc) + ((ns * 2 + tb) * BMAX + warp) * LD, lane, rpl);
                if (lane == 0) {
                    cluster.map_shared_rank(&nrm[0][0][0], tc)[(ns * 2 + tb) * BMAX + warp] = ax;
                    cluster.map_shared_rank(&nrm[0][0][0], bc)[(ns * 2 + bb) * BMAX + warp] = nrm[set][1][warp];
                }
                hj_load<T, RPL>(y, column(set, 1, warp), lane, rpl);
                hj_save<T, RPL>(y, cluster.map_shared_rank(cols, bc) + ((ns * 2 + bb) * BMAX + warp) * LD, lane, rpl);
            }
            cluster.sync();
            set = ns;
        }
        int fl = 0;
        for (int r = 0; r < Ce; ++r) fl |= s_flags[sweep & 1][r];
        if (!(fl & HJ_LARGE) && (fl & (HJ_TURN | HJ_ABOVE)) != (HJ_TURN | HJ_ABOVE)) break;
        steer = steer && (fl & HJ_AGAIN);
    }
    // ---- 3. eigenvalues (exact squared norms) to CTA 0, decreasing order, truncation rule, normalised kept columns.
    // 2 Ce - 1 moves bring every block home, so player k is where the Cholesky put it.
    for (int blk = 0; blk < 2; ++blk) {
        T s = T(0);
        if (warp < b) {
            hj_load<T, RPL>(x, column(set, blk, warp), lane, rpl);
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (q < rpl || hj_vec<T, RPL>) s = fma(x[q], x[q], s);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
        const int k = (2 * warp + blk) * Ce + crank;
        if (warp < b && lane == 0 && k < rc)
            for (int r = 0; r < C; ++r) cluster.map_shared_rank(lam, r)[k] = (double)s;
    }
    cluster.sync();
    // ranks by counting: squared norms are not negative, so their bits order as integers (32 of them in FP32)
    using K = typename std::conditional<sizeof(T) == 8, long long, int>::type;
    K* keys = reinterpret_cast<K*>(lbuf);
    for (int i = tid; i < ROWS; i += NT) {
        K key = -1;
        if (i < rc) {
            const double v = lam[i];
            if constexpr (sizeof(T) == 8) key = v == v ? __double_as_longlong(v) : -1;
            else key = v == v ? __float_as_int((float)v) : -1;
        }
        keys[i] = key;
        if (i >= rc && i < M) lsort[i] = 0.0;
    }
    __syncthreads();
    // (four lanes per player)
    for (int e = tid; e < 4 * ROWS; e += NT) {
        const int i = e >> 2;
        int rk = 0;
        const K own = keys[i];
        for (int j = e & 3; j < rc; j += 4) rk += (keys[j] > own || (keys[j] == own && j < i)) ? 1 : 0;
        rk += __shfl_xor_sync(FULL, rk, 1);
        rk += __shfl_xor_sync(FULL, rk, 2);
        if (i < rc && (e & 3) == 0) {
            ord[i] = (short)rk;
            lsort[rk] = lam[i] * unscale;
        }
    }
    __syncthreads();
    if (crank == 0) {
        if (warp == 0) {
            double rem = s_rem;
            int nz = 0;
            if (sizeof(T) == 8 && p.rr) {   // energy outside the Rayleigh-Ritz subspace
                double all = 0.0;
                for (int i = lane; i < M; i += 32) all += lsort[i];
                all = hj_warp_sum(all);
                rem = fmax(trace - all, 0.0);
            }
            for (int i = lane; i < M; i += 32) nz += lsort[i] > 0.0 ? 1 : 0;
            for (int o = 16; o > 0; o >>= 1) nz += __shfl_xor_sync(FULL, nz, o);
            int s = hj_rule<T>(lsort, M, trace, rem, unc, budget, disc);
            __syncwarp();
            if (lane == 0) {
                if (s == 0 && trace > 0.0 && (m == 0 ? trace : p.norm2) > 0.0) s = 1;
                if (cap > 0 && s > cap) s = cap;
                // a zero column is no direction of the tensor; only the strict rule keeps such (completed below)
                if (!(sizeof(T) == 8 && p.strict) && s > nz) s = nz;
                if (m == 0) { p.norm2 = trace; p.budget = budget; }
                p.s[m] = s;
                p.discarded += disc[s];
                s_keep = s;
                s_nz = nz;
                if (prof) {   // algorithmic work: the dense symmetric eigen-decomposition count 9 M^3; Gram in, S out
                    prof[2 * PK_EIG] += 9.0 * (double)M * M * M;
                    prof[2 * PK_EIG + 1] += (double)sizeof(T) * ((double)M * M + (double)M * s);
                    prof[2 * PK_SWEEPS] += nsweeps;
                    prof[2 * PK_SWEEPS + 1] += 1.0;
                }
            }
            __syncwarp();
            if (lane < C && lane > 0) cluster.map_shared_rank(&s_keep, lane)[0] = s_keep;
        }
        for (int i = tid; i < M; i += NT) evals[i] = lsort[i];
    }
    cluster.sync();
    const int s = s_keep;
    for (int blk = 0; blk < 2; ++blk) {
        const int k = (2 * warp + blk) * Ce + crank;
        if (warp < b && k < rc && ord[k] < s && lam[k] > 0.0) {
            const T inv = (T)rsqrt(lam[k]);
            const T* a = column(set, blk, warp);
            for (int i = lane; i < M; i += 32) S[i + (long long)ord[k] * n] = a[i] * inv;
        }
    }
    if constexpr (sizeof(T) == 8) {
        // The strict rule keeps directions the Gram cannot tell from zero: the basis is completed by unit vectors of
        // rows the Cholesky did not pivot on, orthogonalised twice against what is there (one CTA; rare).
        __syncthreads();
        cluster.sync();
        if (crank == 0 && s > s_nz) {
            double* v = reinterpret_cast<double*>(cols);
            double* w = v + ROWS;
            int c = s_nz;
            for (int i = tid; i < M; i += NT) pivoted[i] = 0;
            __syncthreads();
            for (int k = tid; k < rc; k += NT) pivoted[piv_of[k]] = 1;
            __syncthreads();
            for (int j = 0; j < M && c < s; ++j) {
                if (pivoted[j] && s_nz == rc) continue;   // the same in every thread
                for (int i = tid; i < M; i += NT) v[i] = i == j ? 1.0 : 0.0;
                __syncthreads();
                for (int pass = 0; pass < 2; ++pass) {
                    for (int q = warp; q < c; q += NT / 32) {
                        double d = 0.0;
                        for (int i = lane; i < M; i += 32) d = fma(S[i + (long long)q * n], v[i], d);
                        d = hj_warp_sum(d);
                        if (lane == 0) w[q] = d;
                    }
                    __syncthreads();
                    for (int i = tid; i < M; i += NT) {
                        double a = v[i];
                        for (int q = 0; q < c; ++q) a = fma(-w[q], S[i + (long long)q * n], a);
                        v[i] = a;
                    }
                    __syncthreads();
                }
                double nn = 0.0;
                for (int i = lane; i < M; i += 32) nn = fma(v[i], v[i], nn);
                nn = hj_warp_sum(nn);   // every warp: the same sum
                if (nn > 1e-12) {
                    const double inv = 1.0 / sqrt(nn);
                    for (int i = tid; i < M; i += NT) S[i + (long long)c * n] = v[i] * inv;
                    ++c;
                }
                __syncthreads();
            }
            if (c < s && tid == 0) p.s[m] = c;
        }
    }
}

namespace {
template <typename SH>
int hj_prepare_one(bool* wide) {
    TPCG_CUDA(cudaFuncSetAttribute(hj_eig_kernel<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::SMEM));
    return allow_cluster(hj_eig_kernel<SH>, SH::C, SH::NT, SH::SMEM, wide);
}

template <typename SH>
int hj_launch_one(RoundPlan* plan, const typename SH::T* G, typename SH::T* S, double* evals, int m, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SH::C);
    cfg.blockDim = dim3(SH::NT);
    cfg.dynamicSmemBytes = SH::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = SH::C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    TPCG_CUDA(cudaLaunchKernelEx(&cfg, hj_eig_kernel<SH>, plan, G, S, evals, m, 30, prof_dev()));
    TPCG_CHECK_LAUNCH();
    return TPCG_OK;
}

// FP32: four CTAs of 16 warps; eight CTAs for the same columns were 14% slower at order 120 and full rank, 8 or 16
// instead of 12 pairs before another CTA joins within 5%.  FP64: one pair of columns for each quarter of an SM, by the
// largest order.  More CTAs for the same columns lose to the cluster's barriers (order 32 of 128 possible: 222 us on four,
// 323 us on sixteen), fewer to the FP64 pipes (order 120: 1.5 ms on sixteen, 2.0 ms on eight).
using Hj32 = HjShape<float, 4, 4, 12>;
using Hj64a = HjShape<double, 4, 1, 4>;
using Hj64b = HjShape<double, 8, 2, 4>;
using Hj64c = HjShape<double, 16, 4, 4>;
using Hj64d = HjShape<double, 16, 8, 8>;
// where the device has no clusters of 16
using Hj64c8 = HjShape<double, 8, 4, 4>;
using Hj64d8 = HjShape<double, 8, 8, 8>;
PerDevice hj_device;
}  // namespace

int hj_prepare() {
    return hj_device.prepare([](bool* wide) {
        TPCG_TRY(hj_prepare_one<Hj32>(wide));
        TPCG_TRY(hj_prepare_one<Hj64a>(wide));
        TPCG_TRY(hj_prepare_one<Hj64b>(wide));
        TPCG_TRY(hj_prepare_one<Hj64c>(wide));
        TPCG_TRY(hj_prepare_one<Hj64d>(wide));
        TPCG_TRY(hj_prepare_one<Hj64c8>(wide));
        return hj_prepare_one<Hj64d8>(wide);
    });
}

template <typename T>
int launch_hj(RoundPlan* plan, const T* G, T* S, double* evals, int m, int n, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        return hj_launch_one<Hj32>(plan, G, S, evals, m, st);
    } else {
        if (n <= Hj64a::ROWS) return hj_launch_one<Hj64a>(plan, G, S, evals, m, st);
        if (n <= Hj64b::ROWS) return hj_launch_one<Hj64b>(plan, G, S, evals, m, st);
        if (!hj_device.wide()) {
            if (n <= Hj64c8::ROWS) return hj_launch_one<Hj64c8>(plan, G, S, evals, m, st);
            return hj_launch_one<Hj64d8>(plan, G, S, evals, m, st);
        }
        if (n <= Hj64c::ROWS) return hj_launch_one<Hj64c>(plan, G, S, evals, m, st);
        return hj_launch_one<Hj64d>(plan, G, S, evals, m, st);
    }
}
template int launch_hj<float>(RoundPlan*, const float*, float*, double*, int, int, cudaStream_t);
template int launch_hj<double>(RoundPlan*, const double*, double*, double*, int, int, cudaStream_t);

}  // namespace tpcg
