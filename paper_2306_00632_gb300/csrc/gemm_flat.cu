// The contractions' grouped GEMM on a flat list of output tiles (GemmArgs as in gemm.cuh).
//
// The sizes lie on the device, so a launch is sized for the worst case: most groups of an argument list are empty, or
// far smaller than their bound.  Every CTA therefore counts the tiles of all groups itself (one thread a group, a scan)
// and takes tiles blockIdx.x, blockIdx.x + gridDim.x, ... of that list: no CTA walks over empty groups, and the tiles
// of many small products spread over the chip like those of one large one.  Sums run in the order of k as in the kernels
// this replaces, so results keep their bits.  Measured, whole truncations: operator product n = 128 (19 blocks of rank 36,
// FP32) 1.48 -> 1.23 ms, its 19 products with a long side 175 us -> 32 us; n = 512, FP32, 19.9 -> 10.7 ms; n = 97, FP64,
// 5.3 -> 3.8 ms; a scalar product of rank 6 at n = 32 130 -> 66 us.
#include <math.h>

#include "common.cuh"
#include "device.cuh"
#include "gemm.cuh"

namespace tpcg {

constexpr int GF_MAXG = TPCG_MAX_BLOCKS;   // groups of a launch: one thread each
constexpr int GF_BK = 16;

// pre[g]: tiles of the groups before g (pre[GF_MAXG]: all).  With sym set a group has the tiles of the lower triangle.
template <int TM, int TN>
__device__ __forceinline__ int gf_tiles(const GemmArgs& a) {
    const int tm = (a.M + TM - 1) / TM, tn = (a.N + TN - 1) / TN;
    const int one = TM == TN && a.sym ? tm * (tm + 1) / 2 : tm * tn;
    return a.M > 0 && a.N > 0 ? one * (a.acc ? min(a.nbatch, 1) : a.nbatch) : 0;
}

template <int TM, int TN>
__device__ int gf_list(const GemmArgs* __restrict__ args, int ng, int* pre, int* wsum) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int c = 0;
    if (tid < GF_MAXG) {
        if (tid < ng) c = gf_tiles<TM, TN>(args[tid]);
        int v = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[warp] = v;
        c = v - c;
    }
    __syncthreads();
    if (tid < GF_MAXG) {
        for (int w = 0; w < warp; ++w) c += wsum[w];
        pre[tid] = c;
    }
    __syncthreads();
    return wsum[0] + wsum[1] + wsum[2] + wsum[3];
}

struct GfTile {
    int g, ib, m0, n0;
};

template <int TM, int TN>
__device__ __forceinline__ GfTile gf_find(const GemmArgs* __restrict__ args, const int* pre, int ng, int t) {
    int lo = 0, hi = ng;   // the last group that begins at or before t
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] <= t) lo = mid; else hi = mid;
    }
    const GemmArgs& a = args[lo];
    const int tm = (a.M + TM - 1) / TM, tn = (a.N + TN - 1) / TN;
    int r = t - pre[lo];
    GfTile o;
    o.g = lo;
    if (TM == TN && a.sym) {   // r = i (i + 1) / 2 + j of tile row i and column j <= i
        const int per = tm * (tm + 1) / 2;
        o.ib = r / per;
        r -= o.ib * per;
        int i = (int)((sqrtf(8.0f * (float)r + 1.0f) - 1.0f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= r) ++i;
        while (i * (i + 1) / 2 > r) --i;
        o.m0 = i * TM;
        o.n0 = (r - i * (i + 1) / 2) * TN;
    } else {
        const int per = tm * tn;
        o.ib = r / per;
        r -= o.ib * per;
        o.m0 = (r % tm) * TM;
        o.n0 = (r / tm) * TN;
    }
    return o;
}

// ------------------------------------------------------------------------------------------------------------
// FP64.  An SM has two FP64 FMAs a cycle, a warp's instruction takes its quarter of the SM for 64 cycles: memory, shared
// memory and issue are far from it, so the only thing that counts is that no FMA is done for padding and that every
// quarter has work.  32 x 32 tiles, 128 threads: the lanes run along one side of the tile, the four warps share the other
// side's rows in nearly equal parts (1 to 8 accumulators a thread, as many as there are rows); which side the lanes
// take is the cheaper one of the two for the tile at hand.  With 64 x 64 tiles of 256 threads and 4 x 4 outputs each, a
// product of 18 columns took 20 us, its padded tile's 65536 FMAs a K-step.  The number of rows is a template parameter of
// the K-step: with a test per FMA the switched-off ones took their cycles all the same (a Z formation of 97 columns 738 us,
// now 617 us, 0.59 TFMA/s).  Where the tiles are fewer than the SMs, up to G64_PART CTAs share the rows of a tile (the 32 tiles
// of a Z formation at n = 32 and 190 columns 54 -> 22 us; 8 CTAs a tile are no faster).
// ------------------------------------------------------------------------------------------------------------
constexpr int G64_PART = 4;   // CTAs that share the rows of a tile where the tiles are fewer than the SMs
constexpr int G64_T = 32, G64_NT = 128, G64_LD = G64_T + 1, G64_Q = G64_T * GF_BK / G64_NT;

// elements (i, k) of an operand: base[i si + k sk]; the threads run along whichever index is contiguous
__device__ __forceinline__ void g64_fetch(double (&r)[G64_Q], const double* __restrict__ p, long long si, long long sk, int ni,
                                          int nk, int tid) {
#pragma unroll
    for (int q = 0; q < G64_Q; ++q) {
        const int e = tid + q * G64_NT;
        const int i = si == 1 ? e % G64_T : e / GF_BK, k = si == 1 ? e / G64_T : e % GF_BK;
        r[q] = i < ni && k < nk ? p[i * si + k * sk] : 0.0;
    }
}
__device__ __forceinline__ void g64_store(double* s, const double (&r)[G64_Q], long long si, int tid) {
#pragma unroll
    for (int q = 0; q < G64_Q; ++q) {
        const int e = tid + q * G64_NT;
        const int i = si == 1 ? e % G64_T : e / GF_BK, k = si == 1 ? e / G64_T : e % GF_BK;
        s[k * G64_LD + i] = r[q];
    }
}

// a K-step of a warp with J rows.  J is known to the compiler: FMAs that a test at run time switches off take their cycles all
// the same.
template <int J>
__device__ __forceinline__ void g64_step(double (&acc)[8], const double* X, const double* Y, int kn) {
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
        const double x = X[kk * G64_LD];
#pragma unroll
        for (int j = 0; j < J; ++j) acc[j] = fma(x, Y[kk * G64_LD + j], acc[j]);
    }
}

__global__ void __launch_bounds__(G64_NT, 4) gemm64_kernel(const GemmArgs* __restrict__ args, const int* __restrict__ count_dev,
                                                        int ngroups, int ta, int tb, int sms) {
    __shared__ double As[GF_BK * G64_LD], Bs[GF_BK * G64_LD];
    __shared__ int pre[GF_MAXG], wsum[4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ng = count_dev ? min(*count_dev, ngroups) : ngroups;
    const int total = gf_list<G64_T, G64_T>(args, ng, pre, wsum);
    int part = 1;   // CTAs a tile
    while (part < G64_PART && total * part <= sms) part *= 2;
    for (int t = blockIdx.x; t < total * part; t += gridDim.x) {
        const GfTile tl = gf_find<G64_T, G64_T>(args, pre, ng, t / part);
        const GemmArgs a = args[tl.g];
        const int mr = min(G64_T, a.M - tl.m0), nc = min(G64_T, a.N - tl.n0);
        const bool swap = mr < nc ? (mr + 3) / 4 < (nc + 3) / 4 : false;   // lanes along N, warps along M
        const int cnt = swap ? mr : nc, per = (cnt + 4 * part - 1) / (4 * part);
        const int c0 = (t % part * 4 + warp) * per, mine = max(0, min(per, cnt - c0));
        double acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = 0.0;
        const long long am = ta ? a.lda : 1, ak = ta ? 1 : a.lda, bn = tb ? 1 : a.ldb, bk = tb ? a.ldb : 1;
        const double* X = (swap ? Bs : As) + lane;
        const double* Y = (swap ? As : Bs) + c0;
        const int nb = a.acc ? a.nbatch : 1;
        for (int b = 0; b < nb; ++b) {
            const long long bi = a.acc ? b : tl.ib;
            const double* A = static_cast<const double*>(a.A) + bi * a.sA + tl.m0 * am;
            const double* B = static_cast<const double*>(a.B) + bi * a.sB + tl.n0 * bn;
            double ra[G64_Q], rb[G64_Q];
            g64_fetch(ra, A, am, ak, mr, a.K, tid);
            g64_fetch(rb, B, bn, bk, nc, a.K, tid);
            for (int k0 = 0; k0 < a.K; k0 += GF_BK) {
                __syncthreads();   // the previous K-step is consumed
                g64_store(As, ra, am, tid);
                g64_store(Bs, rb, bn, tid);
                __syncthreads();
                if (k0 + GF_BK < a.K) {
                    g64_fetch(ra, A + (k0 + GF_BK) * ak, am, ak, mr, a.K - k0 - GF_BK, tid);
                    g64_fetch(rb, B + (k0 + GF_BK) * bk, bn, bk, nc, a.K - k0 - GF_BK, tid);
                }
                const int kn = min(GF_BK, a.K - k0);
                switch (mine) {
                    case 1: g64_step<1>(acc, X, Y, kn); break;
                    case 2: g64_step<2>(acc, X, Y, kn); break;
                    case 3: g64_step<3>(acc, X, Y, kn); break;
                    case 4: g64_step<4>(acc, X, Y, kn); break;
                    case 5: g64_step<5>(acc, X, Y, kn); break;
                    case 6: g64_step<6>(acc, X, Y, kn); break;
                    case 7: g64_step<7>(acc, X, Y, kn); break;
                    case 8: g64_step<8>(acc, X, Y, kn); break;
                    default: break;
                }
            }
        }
        double* C = static_cast<double*>(a.C) + (a.acc ? 0LL : (long long)tl.ib * a.sC);
        const bool in = lane < (swap ? nc : mr);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j < mine && in) {
                const int m = tl.m0 + (swap ? c0 + j : lane), nI = tl.n0 + (swap ? lane : c0 + j);
                double* c = C + m + (long long)nI * a.ldc;
                double v = a.alpha * acc[j];
                if (a.beta != 0.0) v += a.beta * (*c);
                *c = v;
            }
    }
}

int launch_gemm64(const GemmArgs* args, const int* count_dev, int ngroups, int bmax, int Mmax, int Nmax, bool ta, bool tb,
                  cudaStream_t st) {
    const long long tiles = (long long)((Mmax + G64_T - 1) / G64_T) * ((Nmax + G64_T - 1) / G64_T) * ngroups * bmax;
    // four CTAs an SM by default: one is enough for the FP64 units, the others hide the loads of a K-step
    const int per_sm = 2 * gemm_ctas_per_sm();   // (the budget counts CTAs of 256 threads)
    const int grid = (int)std::min<long long>(tiles * G64_PART, per_sm > 0 ? (long long)per_sm * sm_count() : 65535LL);
    gemm64_kernel<<<grid, G64_NT, 0, st>>>(args, count_dev, ngroups, ta, tb, sm_count());
    TPCG_CHECK_LAUNCH();
    return TPCG_OK;
}

// ------------------------------------------------------------------------------------------------------------
// FP32.  TM x TN tiles, 8 x CPT outputs a thread as two groups of four rows (and of four columns): 16-byte shared loads
// without bank conflicts.  8 x 8 outputs are what the shared memory can feed (four 16-byte loads for 64 FMAs; 8 x 4 needs
// three for 32); 8 x 4 where a product has no more than a few 64 x 64 tiles.  Operands are copied by cp.async through
// GCP_STAGES stages, 16 bytes at a time where the layout and the alignment allow, and the last K-step stops at K.
// FMAs are paired (two rows an instruction, same rounding): the FP32 units take them at the same rate, but half the issue
// slots are left for the loads.  Truncated product n = 512 10.7 -> 10.2 ms (its largest contraction, 204 GFLOP, 3.9 ms: 52
// TFLOP/s), n = 128 983 -> 950 us, mixed solve n = 128 186 -> 180 ms.
// ------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// K-step k0 of an operand of W rows (first row i0 of ni): s[kk * (W + 4) + i]; KC: contiguous along k, else along i
template <int W, int NT, bool KC>
__device__ __forceinline__ void g32_issue(float* s, const float* p, long long ld, int i0, int ni, int k0, int K, bool vec,
                                          int tid) {
    constexpr int LD = W + 4;
    if (!KC && vec) {
#pragma unroll
        for (int q = 0; q < W * GF_BK / 4 / NT; ++q) {
            const int e = tid + q * NT;
            const int i = (e % (W / 4)) * 4, kk = e / (W / 4);
            const int left = ni - i0 - i;
            const int bytes = k0 + kk < K && left > 0 ? 4 * min(left, 4) : 0;
            cp_async16(s + kk * LD + i, bytes ? p + i0 + i + (long long)(k0 + kk) * ld : p, bytes);
        }
    } else {
#pragma unroll 2
        for (int q = 0; q < W * GF_BK / NT; ++q) {
            const int e = tid + q * NT;
            const int i = KC ? e / GF_BK : e % W, kk = KC ? e % GF_BK : e / W;
            const bool ok = i0 + i < ni && k0 + kk < K;
            const float* src = KC ? p + (k0 + kk) + (long long)(i0 + i) * ld : p + (i0 + i) + (long long)(k0 + kk) * ld;
            cp_async4(s + kk * LD + i, ok ? src : p, ok);
        }
    }
}

template <int TM, int TN, int CPT>
struct G32 {
    static constexpr int NT = (TM / 8) * (TN / CPT);
    static constexpr int MINB = NT == 256 ? 2 : (CPT == 8 ? 4 : 5);   // CTAs an SM: 128 (96) registers a thread
    static constexpr int AS = GF_BK * (TM + 4), BS = GF_BK * (TN + 4);
    static constexpr size_t SMEM = (size_t)GCP_STAGES * (AS + BS) * sizeof(float);
};

template <int TM, int TN, int CPT, bool TA, bool TB>
__global__ void __launch_bounds__(G32<TM, TN, CPT>::NT, G32<TM, TN, CPT>::MINB)
    gemm32_kernel(const GemmArgs* __restrict__ args, const int* __restrict__ count_dev, int ngroups) {
    using C32 = G32<TM, TN, CPT>;
    constexpr int NT = C32::NT, TX = TM / 8, LDA = TM + 4, LDB = TN + 4;
    static_assert(NT >= GF_MAXG, "one thread per group");
    extern __shared__ __align__(16) float g32_smem[];
    float* As = g32_smem;
    float* Bs = g32_smem + GCP_STAGES * C32::AS;
    __shared__ int pre[GF_MAXG], wsum[4];
    const int tid = threadIdx.x;
    const int tx = tid % TX, ty = tid / TX;
    const int ng = count_dev ? min(*count_dev, ngroups) : ngroups;
    const int total = gf_list<TM, TN>(args, ng, pre, wsum);
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        const GfTile tl = gf_find<TM, TN>(args, pre, ng, t);
        const GemmArgs a = args[tl.g];
        const int M = a.M, N = a.N, K = a.K, m0 = tl.m0, n0 = tl.n0;
        float2 acc[4][CPT];   // rows 2 i and 2 i + 1 of the eight
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < CPT; ++j) acc[i][j] = make_float2(0.f, 0.f);
        const int nb = a.acc ? a.nbatch : 1;
        const int nk = (K + GF_BK - 1) / GF_BK;
        for (int b = 0; b < nb; ++b) {
            const long long bi = a.acc ? b : tl.ib;
            const float* A = static_cast<const float*>(a.A) + bi * a.sA;
            const float* B = static_cast<const float*>(a.B) + bi * a.sB;
            const bool va = !TA && (a.lda & 3) == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;
            const bool vb = TB && (a.ldb & 3) == 0 && (reinterpret_cast<uintptr_t>(B) & 15) == 0;
#pragma unroll
            for (int st = 0; st < GCP_STAGES - 1; ++st) {   // the first stages (empty groups past K)
                if (st < nk) {
                    g32_issue<TM, NT, TA>(As + st * C32::AS, A, a.lda, m0, M, st * GF_BK, K, va, tid);
                    g32_issue<TN, NT, !TB>(Bs + st * C32::BS, B, a.ldb, n0, N, st * GF_BK, K, vb, tid);
                }
                cp_async_commit();
            }
            int cur = 0;
            for (int kt = 0; kt < nk; ++kt) {
                cp_async_wait<GCP_STAGES - 2>();   // this thread's copies of K-step kt have landed
                __syncthreads();                   // everyone's have, and everyone is done with K-step kt - 1
                const int nx = kt + GCP_STAGES - 1;
                if (nx < nk) {
                    const int sn = cur == 0 ? GCP_STAGES - 1 : cur - 1;
                    g32_issue<TM, NT, TA>(As + sn * C32::AS, A, a.lda, m0, M, nx * GF_BK, K, va, tid);
                    g32_issue<TN, NT, !TB>(Bs + sn * C32::BS, B, a.ldb, n0, N, nx * GF_BK, K, vb, tid);
                }
                cp_async_commit();
                const float* Ac = As + cur * C32::AS + 4 * tx;
                const float* Bc = Bs + cur * C32::BS + 4 * ty;
                const int kn = K - kt * GF_BK;
#pragma unroll 1   // (unrolled further, the loads ahead do not fit in the registers)
                for (int k4 = 0; k4 < GF_BK; k4 += 4) {
                    if (k4 >= kn) break;   // (rows past K are zero)
#pragma unroll
                    for (int k1 = 0; k1 < 4; ++k1) {
                        const int kk = k4 + k1;
                        const float4 a0 = *reinterpret_cast<const float4*>(Ac + kk * LDA);
                        const float4 a1 = *reinterpret_cast<const float4*>(Ac + kk * LDA + TM / 2);
                        const float2 av[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w), make_float2(a1.x, a1.y),
                                              make_float2(a1.z, a1.w)};
                        float bv[CPT];
                        *reinterpret_cast<float4*>(bv) = *reinterpret_cast<const float4*>(Bc + kk * LDB);
                        if constexpr (CPT == 8)
                            *reinterpret_cast<float4*>(bv + 4) = *reinterpret_cast<const float4*>(Bc + kk * LDB + TN / 2);
#pragma unroll
                        for (int j = 0; j < CPT; ++j)
#pragma unroll
                            for (int i = 0; i < 4; ++i) acc[i][j] = __ffma2_rn(av[i], make_float2(bv[j], bv[j]), acc[i][j]);
                    }
                }
                cur = cur == GCP_STAGES - 1 ? 0 : cur + 1;
            }
            cp_async_wait<0>();
            __syncthreads();   // the stages are refilled by the next batch or tile
        }
        float* C = static_cast<float*>(a.C) + (a.acc ? 0LL : (long long)tl.ib * a.sC);
        const float alpha = (float)a.alpha, beta = (float)a.beta;
        const bool vc = (a.ldc & 3) == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0 && beta == 0.f;
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            const int nI = n0 + 4 * ty + (j < 4 ? j : TN / 2 + j - 4);
            if (nI >= N) continue;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = m0 + 4 * tx + h * (TM / 2);
                float* c = C + m + (long long)nI * a.ldc;
                float v[4];
#pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    v[i] = alpha * acc[2 * h + i / 2][j].x;
                    v[i + 1] = alpha * acc[2 * h + i / 2][j].y;
                }
                if (vc && m + 3 < M) {
                    *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (m + i < M) c[i] = beta != 0.f ? v[i] + beta * c[i] : v[i];
                }
            }
        }
    }
}

namespace {
template <int TM, int TN, int CPT, bool TA, bool TB>
int g32_launch(const GemmArgs* args, const int* count_dev, int ngroups, int bmax, int Mmax, int Nmax, int per_sm,
               cudaStream_t st) {
    using C32 = G32<TM, TN, CPT>;
    const long long tiles = (long long)((Mmax + TM - 1) / TM) * ((Nmax + TN - 1) / TN) * ngroups * bmax;
    const long long cap = per_sm > 0 ? (long long)per_sm * sm_count() : 65535LL;
    gemm32_kernel<TM, TN, CPT, TA, TB>
        <<<(int)std::min(tiles, cap), C32::NT, C32::SMEM, st>>>(args, count_dev, ngroups);
    TPCG_CHECK_LAUNCH();
    return TPCG_OK;
}
}  // namespace

// The tile by the bounds of a product's sides: 128 rows or columns along a side that can be long (1024 and more: the
// products over a whole face of the tensor), 128 x 128 for the Grams above order 128, 64 x 64 else.
template <bool TA, bool TB>
int launch_gemm32(const GemmArgs* args, const int* count_dev, int ngroups, int bmax, int Mmax, int Nmax, bool sym,
                  cudaStream_t st) {
    const int per_sm = 2 * gemm_ctas_per_sm();   // (the budget counts CTAs of 256 threads)
    if (sym && Mmax > 128)
        return g32_launch<128, 128, 8, TA, TB>(args, count_dev, ngroups, bmax, Mmax, Nmax, per_sm / 2, st);
    if (!sym && Mmax >= 1024) return g32_launch<128, 64, 8, TA, TB>(args, count_dev, ngroups, bmax, Mmax, Nmax, per_sm, st);
    if (!sym && Nmax >= 1024) return g32_launch<64, 128, 8, TA, TB>(args, count_dev, ngroups, bmax, Mmax, Nmax, per_sm, st);
    return g32_launch<64, 64, 4, TA, TB>(args, count_dev, ngroups, bmax, Mmax, Nmax, per_sm, st);
}
template int launch_gemm32<false, false>(const GemmArgs*, const int*, int, int, int, int, bool, cudaStream_t);
template int launch_gemm32<false, true>(const GemmArgs*, const int*, int, int, int, int, bool, cudaStream_t);
template int launch_gemm32<true, false>(const GemmArgs*, const int*, int, int, int, int, bool, cudaStream_t);

// dynamic shared memory above 48 KB
int gemm32_prepare() {
    static PerDevice device;
    return device.prepare([](bool*) {
        const int b = (int)G32<128, 128, 8>::SMEM;
        TPCG_CUDA(cudaFuncSetAttribute(gemm32_kernel<128, 128, 8, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
        TPCG_CUDA(cudaFuncSetAttribute(gemm32_kernel<128, 128, 8, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
        TPCG_CUDA(cudaFuncSetAttribute(gemm32_kernel<128, 128, 8, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, b));
        return TPCG_OK;
    });
}

}  // namespace tpcg
