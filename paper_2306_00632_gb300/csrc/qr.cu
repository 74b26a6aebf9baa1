// Householder QR of the factors (Alg. 1 step 1): Y_t = Q_t R_t for the modes with k_t < n, one cluster of CTAs per mode.
//
// The columns are dealt to the warps of the cluster and stay in registers (rows across the lanes).  In step j every warp
// applies reflector j to its columns; the warp that holds column j + 1 does that one first, makes reflector j + 1 of it and
// writes it into every CTA's shared memory, so that one barrier a step is enough.  The columns of Q = H_0 ... H_{k-1} [I; 0]
// do not depend on each other: column c takes H_c, ..., H_0, without any barrier.
//
// What bounds it: k steps of one warp's chain (update of column j + 1, its norm, the reflector, the barrier), about 0.6 us in
// FP32 and, at 64 cycles an FP64 instruction, 2 us in FP64.  Measured at n = 128 and 106 / 60 / 30 columns, three modes: FP32
// 111 / 60 / 33 us on four CTAs of 16 warps (one CTA of 32 warps 158 / 81 / 36, eight of 16 98 / 57 / 32); FP64 445 / 222 /
// 111 us on eight CTAs of 8 warps (eight of 4 532 / 259 / 111, sixteen of 4 435 / 223 / 113; square root and division are
// CUDA's: an FP32 estimate and a correction in their place took 447 us).  The kernel this replaces, one CTA with its working
// copy in global memory, took 400 us in FP32 at 106 columns and 190 us in FP64 for 17 columns at n = 32 (now 41).
// Reflectors are kept unscaled, H = I - f v v^T with v = a -+ |a| e_1 and f = 1 / (|a| (|a| + |a_1|)).
#include <math.h>

#include <cooperative_groups.h>

#include "common.cuh"
#include "device.cuh"
#include "kernels.cuh"

namespace tpcg {

namespace cgx = cooperative_groups;

template <typename T>
__device__ __forceinline__ T qr_warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// the sums over the lanes of N values, all of them in every lane; two and four values share their additions
template <typename T, int N>
__device__ __forceinline__ void qr_warp_sums(T (&d)[N], int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    if constexpr (N == 4 || N == 2) {
        T u;
        const bool b4 = lane & 16, b3 = lane & 8;
        if constexpr (N == 4) {
            const T x0 = __shfl_xor_sync(FULL, b4 ? d[0] : d[2], 16), x1 = __shfl_xor_sync(FULL, b4 ? d[1] : d[3], 16);
            const T u0 = (b4 ? d[2] : d[0]) + x0, u1 = (b4 ? d[3] : d[1]) + x1;
            u = (b3 ? u1 : u0) + __shfl_xor_sync(FULL, b3 ? u0 : u1, 8);
        } else {
            u = (b4 ? d[1] : d[0]) + __shfl_xor_sync(FULL, b4 ? d[0] : d[1], 16);
            u += __shfl_xor_sync(FULL, u, 8);
        }
        u += __shfl_xor_sync(FULL, u, 4);
        u += __shfl_xor_sync(FULL, u, 2);
        u += __shfl_xor_sync(FULL, u, 1);
#pragma unroll
        for (int s = 0; s < N; ++s) d[s] = __shfl_sync(FULL, u, N == 4 ? 8 * s : 16 * s);
    } else {
#pragma unroll
        for (int s = 0; s < N; ++s) d[s] = qr_warp_sum(d[s]);
    }
}

// Shape of a launch: C CTAs of NW warps per mode, RPL rows a lane (n up to 32 RPL), CPW columns a warp (k up to
// C NW CPW).  VS: all reflectors stay in shared memory; else the current two, and all of them in global memory.
template <typename T_, int C_, int NW_, int RPL_, int CPW_, bool VS_>
struct QrShape {
    using T = T_;
    static constexpr int C = C_, NW = NW_, RPL = RPL_, CPW = CPW_, ROWS = 32 * RPL_;
    static constexpr bool VS = VS_;
    static constexpr size_t SMEM = ((size_t)(VS ? ROWS : 2) * ROWS + ROWS) * sizeof(T);   // reflectors, their factors f
    static_assert(C * NW * CPW >= ROWS, "a warp for every column");
};

template <typename SH>
__global__ void __launch_bounds__(32 * SH::NW, 1)
    qr_hh_kernel(const RoundPlan* __restrict__ plan, const typename SH::T* Y0, const typename SH::T* Y1, const typename SH::T* Y2,
                 typename SH::T* W0, typename SH::T* W1, typename SH::T* W2, typename SH::T* R0, typename SH::T* R1,
                 typename SH::T* R2, typename SH::T* Q0, typename SH::T* Q1, typename SH::T* Q2) {
    using T = typename SH::T;
    constexpr int C = SH::C, NW = SH::NW, RPL = SH::RPL, CPW = SH::CPW, ROWS = SH::ROWS, GW = C * NW;
    constexpr bool VS = SH::VS;
    const int t = blockIdx.x / C;
    const RoundPlan& p = *plan;
    if (!p.useQ[t]) return;   // the whole cluster
    cgx::cluster_group cluster = cgx::this_cluster();
    const int crank = C > 1 ? (int)cluster.block_rank() : 0;
    const T* Y = t == 0 ? Y0 : (t == 1 ? Y1 : Y2);
    T* W = t == 0 ? W0 : (t == 1 ? W1 : W2);
    T* R = t == 0 ? R0 : (t == 1 ? R1 : R2);
    T* Q = t == 0 ? Q0 : (t == 1 ? Q1 : Q2);
    const int n = p.n, k = p.k[t];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, gw = crank * NW + warp;
    extern __shared__ __align__(16) unsigned char qr_smem[];
    T* vs = reinterpret_cast<T*>(qr_smem);                     // reflector j at vs + (j or j & 1) ROWS
    T* fs = vs + (VS ? ROWS : 2) * ROWS;
    auto vslot = [&](int j) { return (VS ? j : (j & 1)) * ROWS; };
    auto wait = [&]() {
        if constexpr (C > 1) cluster.sync();
        else __syncthreads();
    };
    T a[CPW][RPL];
#pragma unroll
    for (int s = 0; s < CPW; ++s)
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q, c = gw + GW * s;
            a[s][q] = (i < n && c < k) ? Y[i + (long long)c * n] : T(0);
        }
    // reflector j of column x (rows >= j), to every CTA; the column keeps R's entries
    auto reflect = [&](T (&x)[RPL], int j) {
        T sig = T(0), al = T(0);
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            if (32 * q + 31 > j && i > j) sig = fma(x[q], x[q], sig);
            if (i == j) al = x[q];
        }
        sig = qr_warp_sum(sig);
        al = __shfl_sync(0xffffffffu, al, j & 31);
        T s2 = fma(al, al, sig), sc = T(1), unsc = T(1);
        if (s2 < (sizeof(T) == 8 ? T(1e-280) : T(1e-30f))) {   // squares near or below the end of the range: scaled column
            sc = sizeof(T) == 8 ? T(0x1p500) : T(0x1p60f);
            unsc = sizeof(T) == 8 ? T(0x1p-500) : T(0x1p-60f);
            sig = T(0);
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (lane + 32 * q > j) sig = fma(x[q] * sc, x[q] * sc, sig);
            sig = qr_warp_sum(sig);
            al *= sc;
            s2 = fma(al, al, sig);
        }
        const bool any = !(sig == T(0));   // (a NaN goes on through the column)
        T nrm = T(0), f = T(0), vj = T(0), beta = al * unsc;
        if (any) {
            nrm = sqrt(s2);
            f = T(1) / (nrm * (nrm + fabs(al)));
            vj = al >= T(0) ? al + nrm : al - nrm;
            beta = (al >= T(0) ? -nrm : nrm) * unsc;
        }
        T v[RPL];
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            v[q] = i > j && any ? x[q] * sc : (i == j ? vj : T(0));
            if (i == j) x[q] = beta;
        }
#pragma unroll
        for (int r = 0; r < C; ++r) {
            T* dv = vs;
            T* df = fs;
            if constexpr (C > 1) {
                dv = cluster.map_shared_rank(vs, r);
                df = cluster.map_shared_rank(fs, r);
            }
#pragma unroll
            for (int q = 0; q < RPL; ++q) dv[vslot(j) + lane + 32 * q] = v[q];
            if (lane == 0) df[j] = f;
        }
        if constexpr (!VS) {
#pragma unroll
            for (int q = 0; q < RPL; ++q)
                if (lane + 32 * q < n) W[lane + 32 * q + (long long)j * n] = v[q];
        }
    };
    wait();   // every CTA of the cluster runs: remote writes may begin
    if (gw == 0) reflect(a[0], 0);
    wait();
    for (int j = 0; j + 1 < k; ++j) {
        T v[RPL];
        const T f = fs[j];
        const int q0 = j >> 5;   // rows below 32 q0 are zero in the reflector
#pragma unroll
        for (int q = 0; q < RPL; ++q) v[q] = q >= q0 ? vs[vslot(j) + lane + 32 * q] : T(0);
        T d[CPW];
        const int own = (j + 1) % GW == gw ? (j + 1) / GW : -1;   // this warp holds column j + 1
        if (own >= 0) {
#pragma unroll
            for (int s = 0; s < CPW; ++s)
                if (s == own) {
                    T w = T(0);
#pragma unroll
                    for (int q = 0; q < RPL; ++q)
                        if (q >= q0) w = fma(v[q], a[s][q], w);
                    w = qr_warp_sum(w) * f;
#pragma unroll
                    for (int q = 0; q < RPL; ++q)
                        if (q >= q0) a[s][q] = fma(-w, v[q], a[s][q]);
                    reflect(a[s], j + 1);
                }
        }
        const int last = (k - 1 - gw) / GW;   // slots above hold no column (negative: none)
        if (gw < k && gw + GW * last > j + 1) {
#pragma unroll
            for (int s = 0; s < CPW; ++s) {
                d[s] = T(0);
                if (gw + GW * s > j + 1 && s <= last) {
#pragma unroll
                    for (int q = 0; q < RPL; ++q)
                        if (q >= q0) d[s] = fma(v[q], a[s][q], d[s]);
                }
            }
            qr_warp_sums<T, CPW>(d, lane);
#pragma unroll
            for (int s = 0; s < CPW; ++s)
                if (gw + GW * s > j + 1 && s <= last) {
                    const T w = d[s] * f;
#pragma unroll
                    for (int q = 0; q < RPL; ++q)
                        if (q >= q0) a[s][q] = fma(-w, v[q], a[s][q]);
                }
        }
        wait();
    }
    // R, and the columns of Q
#pragma unroll
    for (int s = 0; s < CPW; ++s) {
        const int c = gw + GW * s;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            if (c < k && i < k) R[i + (long long)c * n] = i <= c ? a[s][q] : T(0);
            a[s][q] = i == c ? T(1) : T(0);
        }
    }
    const int cmax = gw < k ? gw + GW * ((k - 1 - gw) / GW) : -1;   // this warp's last column
    for (int j = cmax; j >= 0; --j) {
        const T f = fs[j];
        const int q0 = j >> 5;
        T v[RPL], d[CPW];
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            if constexpr (VS) v[q] = q >= q0 ? vs[vslot(j) + i] : T(0);
            else v[q] = q >= q0 && i < n ? W[i + (long long)j * n] : T(0);
        }
#pragma unroll
        for (int s = 0; s < CPW; ++s) {
            d[s] = T(0);
            if (gw + GW * s >= j && gw + GW * s <= cmax) {
#pragma unroll
                for (int q = 0; q < RPL; ++q)
                    if (q >= q0) d[s] = fma(v[q], a[s][q], d[s]);
            }
        }
        qr_warp_sums<T, CPW>(d, lane);
#pragma unroll
        for (int s = 0; s < CPW; ++s)
            if (gw + GW * s >= j && gw + GW * s <= cmax) {
                const T w = d[s] * f;
#pragma unroll
                for (int q = 0; q < RPL; ++q)
                    if (q >= q0) a[s][q] = fma(-w, v[q], a[s][q]);
            }
    }
#pragma unroll
    for (int s = 0; s < CPW; ++s) {
        const int c = gw + GW * s;
#pragma unroll
        for (int q = 0; q < RPL; ++q) {
            const int i = lane + 32 * q;
            if (c < k && i < n) Q[i + (long long)c * n] = a[s][q];
        }
    }
}

namespace {
template <typename SH>
int qr_prepare_one(bool* wide) {
    TPCG_CUDA(cudaFuncSetAttribute(qr_hh_kernel<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::SMEM));
    return allow_cluster(qr_hh_kernel<SH>, SH::C, 32 * SH::NW, SH::SMEM, wide);
}

template <typename SH>
int qr_launch_one(const RoundPlan* plan, const typename SH::T* const* Y, typename SH::T* const* W, typename SH::T* const* R,
                  typename SH::T* const* Q, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(3 * SH::C);
    cfg.blockDim = dim3(32 * SH::NW);
    cfg.dynamicSmemBytes = SH::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = SH::C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    TPCG_CUDA(cudaLaunchKernelEx(&cfg, qr_hh_kernel<SH>, plan, Y[0], Y[1], Y[2], W[0], W[1], W[2], R[0], R[1], R[2], Q[0], Q[1],
                                 Q[2]));
    TPCG_CHECK_LAUNCH();
    return TPCG_OK;
}

using Qr32a = QrShape<float, 4, 16, 4, 2, true>;
using Qr32b = QrShape<float, 8, 16, 8, 2, false>;
using Qr32c = QrShape<float, 16, 16, 16, 2, false>;
using Qr64a = QrShape<double, 8, 4, 1, 1, true>;
using Qr64b = QrShape<double, 8, 4, 2, 2, true>;
using Qr64c = QrShape<double, 8, 8, 4, 2, true>;
using Qr64d = QrShape<double, 16, 8, 8, 2, false>;
using Qr64e = QrShape<double, 16, 16, 16, 2, false>;
PerDevice qr_device;
}  // namespace

int qr_prepare() {
    return qr_device.prepare([](bool* wide) {
        TPCG_TRY(qr_prepare_one<Qr32a>(wide));
        TPCG_TRY(qr_prepare_one<Qr32b>(wide));
        TPCG_TRY(qr_prepare_one<Qr32c>(wide));
        TPCG_TRY(qr_prepare_one<Qr64a>(wide));
        TPCG_TRY(qr_prepare_one<Qr64b>(wide));
        TPCG_TRY(qr_prepare_one<Qr64c>(wide));
        TPCG_TRY(qr_prepare_one<Qr64d>(wide));
        return qr_prepare_one<Qr64e>(wide);
    });
}

bool qr_fits(int n, int elt) {
    const int narrow = elt == 4 ? Qr32b::ROWS : Qr64c::ROWS;   // the largest on clusters of 8
    return n <= narrow || (n <= QR_MAXN && qr_device.wide());
}

template <typename T>
int launch_qr(const RoundPlan* plan, int n, const T* const* Y, T* const* W, T* const* R, T* const* Q, cudaStream_t st) {
    if constexpr (sizeof(T) == 4) {
        if (n <= Qr32a::ROWS) return qr_launch_one<Qr32a>(plan, Y, W, R, Q, st);
        if (n <= Qr32b::ROWS) return qr_launch_one<Qr32b>(plan, Y, W, R, Q, st);
        return qr_launch_one<Qr32c>(plan, Y, W, R, Q, st);
    } else {
        if (n <= Qr64a::ROWS) return qr_launch_one<Qr64a>(plan, Y, W, R, Q, st);
        if (n <= Qr64b::ROWS) return qr_launch_one<Qr64b>(plan, Y, W, R, Q, st);
        if (n <= Qr64c::ROWS) return qr_launch_one<Qr64c>(plan, Y, W, R, Q, st);
        if (n <= Qr64d::ROWS) return qr_launch_one<Qr64d>(plan, Y, W, R, Q, st);
        return qr_launch_one<Qr64e>(plan, Y, W, R, Q, st);
    }
}
template int launch_qr<float>(const RoundPlan*, int, const float* const*, float* const*, float* const*, float* const*,
                              cudaStream_t);
template int launch_qr<double>(const RoundPlan*, int, const double* const*, double* const*, double* const*, double* const*,
                               cudaStream_t);

}  // namespace tpcg
