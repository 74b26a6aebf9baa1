// FD preconditioner (Alg. 4 with App. B's eigenvectors) with the sine block as two dense half matrices, three launches.
//
// Both ends alike, the grid points lie symmetrically: U_dft[L-1-l, j] = +-U_dft[l, j], + for the even columns j.  So
// U_dft^T x needs, for even j, only x_l + x_{L-1-l} and, for odd j, only x_l - x_{L-1-l}, and U_dft e = (a + b) on the first
// half of the points and (a - b) on the other with a and b the sums over the even and the odd j: n1^2 / 2 multiply-adds a
// column.  In FP64 that is what counts (two FMAs a cycle and SM): at n1 = 126 8,000 a column, where Bluestein's two FFTs of
// length 256 take 18,000 instructions besides their trips through shared memory.
//
//   fd_fold_fwd   u = U_dft^T (W^T S), z2 = V2U2^T S (columns along the lanes, row-major), and the factors
//                 F[j][q] = exp(-alpha_j c_t lambda_q / lambda_min) (/ mu_q^2), once per term and row instead of per column
//   fd_fold_inv   A = U_dft (F_j u): 32 columns a CTA, rows over its warps; the scaled columns are made in shared memory
//   fd_fold_out   V = W A + V2U2 (F_j z2), and the descriptor
//
// Four chains of additions an output: shorter chains round less (relative error in FP32 at n1 = 126 / 254: 1.1e-7 / 1.5e-7,
// the FFTs 1.6e-7 / 1.7e-7; one chain 1.9e-7 / 2.8e-7).
//
// Measured, 12 terms on rank 44, against nine launches with FFTs: n = 128 FP64 242 -> 76 us, FP32 81 -> 25 us; rank 6,
// n = 32 FP64 80 -> 22 us; n = 256 FP64 328 -> 173 us, FP32 96 -> 36 us.  Loads one row after the other (a trip to memory for
// the row's pointer, its column and the value) cost another 26 us in FP32.
#include <math.h>

#include <algorithm>

#include "common.cuh"
#include "device.cuh"
#include "gemm.cuh"
#include "kernels.cuh"

namespace tpcg {

constexpr int FF_TC = 32;      // columns of a tile: one a lane
constexpr int FF_RW = 4;       // rows a warp of fd_fold_inv takes at most
constexpr int FF_REST = 4;     // CTAs a column tile for the factors and z2
constexpr int FF_FWD_T = 256, FF_INV_T = 128, FF_OUT_T = 256;

template <typename T>
struct FdFold {
    const TuckerDesc* sd;
    const T* S[3];
    T* F[3];          // RP x n factors
    T* u[3];          // (n1 + n2) x r, row-major: u, then z2
    T* A[3];          // n1 x RP r, row-major
    T* V[3];
    const int *wtrow, *wtcol, *wrow, *wcol;
    const T *wtval, *wval, *v2u2, *dst, *lam, *mu;
    const double *alpha, *omega;
    double lmin, cw[3];
    int n, n1, n2, RP, vcap, chunks, sms;
};

template <typename T>
constexpr size_t ff_fwd_smem(int n1) { return (size_t)n1 * (FF_TC + 1 + FF_FWD_T / 32) * sizeof(T); }
template <typename T>
constexpr size_t ff_inv_smem(int n1) { return (size_t)((n1 + 7) & ~7) * (FF_TC + 4 * FF_RW) * sizeof(T); }

// columns of mode t's output; 0 where there are none or where they exceed the output's capacity
template <typename T>
__device__ __forceinline__ int ff_cols(const FdFold<T>& a, int t) {
    const long long c = (long long)a.RP * a.sd->rank[t];
    return c > a.vcap ? 0 : (int)c;
}

// grid: (tiles of input columns, chunks of outputs and one for the rest, modes)
template <typename T>
__global__ void __launch_bounds__(FF_FWD_T) fd_fold_fwd_kernel(const FdFold<T> a) {
    const int t = blockIdx.z, r = a.sd->rank[t], n = a.n, n1 = a.n1;
    if (ff_cols(a, t) == 0) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const T* __restrict__ S = a.S[t];
    T* __restrict__ u = a.u[t];
    if ((int)blockIdx.y >= a.chunks) {   // the factors and z2
        const int nb = gridDim.x * FF_REST, b = blockIdx.x * FF_REST + blockIdx.y - a.chunks;
        for (int e = b * FF_FWD_T + tid; e < a.RP * n; e += nb * FF_FWD_T) {
            const int j = e / n, q = e % n;
            const T aj = (T)(a.alpha[j] * a.cw[t] / a.lmin);
            const T dl = exp(-aj * a.lam[q]);
            a.F[t][e] = q < n1 ? dl / (a.mu[q] * a.mu[q]) : dl;
        }
        for (int w = b * (FF_FWD_T / 32) + warp; w < a.n2 * r; w += nb * (FF_FWD_T / 32)) {
            const int q = w / r, c = w % r;
            T acc = T(0);
            for (int i = lane; i < n; i += 32) acc = fma(a.v2u2[i + (long long)q * n], S[i + (long long)c * n], acc);
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) u[(long long)(n1 + q) * r + c] = acc;
        }
        return;
    }
    const int c0 = blockIdx.x * FF_TC;
    if (c0 >= r) return;
    const int nc = min(FF_TC, r - c0);
    extern __shared__ __align__(16) unsigned char ff_smem[];
    constexpr int LD = FF_TC + 1, NW = FF_FWD_T / 32, CPW = FF_TC / NW;
    T* x = reinterpret_cast<T*>(ff_smem);   // [point][column]
    T* mrow = x + (size_t)n1 * LD + warp * n1;   // this warp's column of the sine block
    const int j = blockIdx.y * NW + warp;
    if (j < n1)
        for (int l = lane; l < n1; l += 32) mrow[l] = a.dst[(long long)j * n1 + l];
    // W^T S, points along the lanes and CPW columns a warp; a row of W^T has one entry but near the ends, and the first
    // entries of four rows are fetched together (one after the other they cost three trips to memory a row)
    for (int lb = lane; lb < n1; lb += 128) {
        int k0[4], k1[4];
        T acc[4][CPW];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int l = lb + 32 * i;
            k0[i] = l < n1 ? a.wtrow[l] : 0;
            k1[i] = l < n1 ? a.wtrow[l + 1] : 0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const bool has = k0[i] < k1[i];
            const T v = has ? a.wtval[k0[i]] : T(0);
            const T* src = S + (has ? a.wtcol[k0[i]] : 0);
#pragma unroll
            for (int q = 0; q < CPW; ++q) {
                const int c = warp + NW * q;
                acc[i][q] = has && c < nc ? v * src[(long long)(c0 + c) * n] : T(0);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            for (int k = k0[i] + 1; k < k1[i]; ++k) {
                const T v = a.wtval[k];
                const T* src = S + a.wtcol[k];
#pragma unroll
                for (int q = 0; q < CPW; ++q) {
                    const int c = warp + NW * q;
                    if (c < nc) acc[i][q] = fma(v, src[(long long)(c0 + c) * n], acc[i][q]);
                }
            }
            if (lb + 32 * i < n1)
#pragma unroll
                for (int q = 0; q < CPW; ++q) x[(lb + 32 * i) * LD + warp + NW * q] = acc[i][q];
        }
    }
    __syncthreads();
    for (int e = tid; e < (n1 / 2) * FF_TC; e += FF_FWD_T) {   // sums in the first half, differences in the second
        T* p = x + (e / FF_TC) * LD + e % FF_TC;
        T* q = x + (n1 - 1 - e / FF_TC) * LD + e % FF_TC;
        const T v = *p, w = *q;
        *p = v + w;
        *q = v - w;
    }
    __syncthreads();
    if (j < n1) {
        const bool even = (j & 1) == 0;
        const int H = even ? (n1 + 1) / 2 : n1 / 2, step = even ? LD : -LD;
        const T* xp = x + (even ? 0 : (n1 - 1) * LD) + lane;
        const T* m = mrow;
        T s[4] = {T(0), T(0), T(0), T(0)};
        int l = 0;
#pragma unroll 2
        for (; l + 4 <= H; l += 4)
#pragma unroll
            for (int k = 0; k < 4; ++k) s[k] = fma(m[l + k], xp[(l + k) * step], s[k]);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (l + k < H) s[k] = fma(m[l + k], xp[(l + k) * step], s[k]);
        if (lane < nc) u[(long long)j * r + c0 + lane] = (s[0] + s[1]) + (s[2] + s[3]);
    }
}

// Rows of one warp (the first PW of its FF_RW places in m): sums over the even and the odd sinusoids, stored to both halves
template <typename T, int PW>
__device__ __forceinline__ void ff_rows(const T* x, const T* m, int n1, int n1p, int l0, int H, bool in, T* __restrict__ A,
                                        int cols, int col) {
    T s[PW][2][4];
#pragma unroll
    for (int i = 0; i < PW; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) s[i][k & 1][k >> 1] = T(0);
    for (int q = 0; q < n1p; q += 8) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const T xv = x[(q + k) * FF_TC];
            const T* mq = m + (q + k) * 4 * FF_RW;
#pragma unroll
            for (int i = 0; i < PW; ++i) s[i][k & 1][k >> 1] = fma(mq[i], xv, s[i][k & 1][k >> 1]);
        }
    }
#pragma unroll
    for (int i = 0; i < PW; ++i) {
        const int l = l0 + i;
        if (!in || l >= H) continue;
        const T e = (s[i][0][0] + s[i][0][1]) + (s[i][0][2] + s[i][0][3]);
        const T o = (s[i][1][0] + s[i][1][1]) + (s[i][1][2] + s[i][1][3]);
        A[(long long)l * cols + col] = e + o;
        if (l != n1 - 1 - l) A[(long long)(n1 - 1 - l) * cols + col] = e - o;
    }
}

// A work item: FF_TC columns of one mode and 4 `pw` rows of the half (pw a warp).  pw is the one for which the SMs' largest
// share of items costs least: small tensors get one row a warp and all SMs, large ones four, which halves the share of the
// work that makes the scaled columns (a quarter of a row each).
template <typename T>
__global__ void __launch_bounds__(FF_INV_T) fd_fold_inv_kernel(const FdFold<T> a) {
    const int n1 = a.n1, H = (n1 + 1) / 2, n1p = (n1 + 7) & ~7;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int tiles[3], tot = 0;
    for (int t = 0; t < 3; ++t) {
        tiles[t] = (ff_cols(a, t) + FF_TC - 1) / FF_TC;
        tot += tiles[t];
    }
    int pw = 1, best = 0x7fffffff;
    for (int q = FF_RW; q >= 1; --q) {
        const int items = tot * ((H + 4 * q - 1) / (4 * q)), cost = (items + a.sms - 1) / a.sms * (4 * q + 1);
        if (cost < best) { best = cost; pw = q; }
    }
    const int per = (H + 4 * pw - 1) / (4 * pw);
    extern __shared__ __align__(16) unsigned char ff_smem[];
    T* x = reinterpret_cast<T*>(ff_smem);   // [sinusoid][column], rows past n1 zero
    T* m = x + n1p * FF_TC;                 // [sinusoid][row of the item]
    for (int w = blockIdx.x; w < tot * per; w += gridDim.x) {
        int tile = w / per, t = 0;
        const int l0 = (w % per) * 4 * pw + warp * pw;
        while (tile >= tiles[t]) tile -= tiles[t++];
        const int r = a.sd->rank[t], cols = a.RP * r;
        const int col = tile * FF_TC + lane, j = col < cols ? col / r : 0, c = col < cols ? col - j * r : 0;
        const T* __restrict__ u = a.u[t] + c;
        const T* __restrict__ f = a.F[t] + (long long)j * a.n;
        __syncthreads();   // the previous item is done with x
#pragma unroll 8
        for (int e = tid; e < n1p * 4 * FF_RW; e += FF_INV_T) {   // FF_RW places a warp, pw of them used
            const int i = e % FF_RW, q = e / (4 * FF_RW), l = (w % per) * 4 * pw + e / FF_RW % 4 * pw + i;
            m[e] = q < n1 && i < pw && l < H ? a.dst[l + (long long)q * n1] : T(0);
        }
#pragma unroll 8
        for (int q = warp; q < n1p; q += FF_INV_T / 32) x[q * FF_TC + lane] = q < n1 ? f[q] * u[(long long)q * r] : T(0);
        __syncthreads();
        const T *xl = x + lane, *mw = m + warp * FF_RW;
        const bool in = col < cols;
        switch (pw) {   // (a count known to the compiler: a test per multiply-add made five instructions of one)
            case 1: ff_rows<T, 1>(xl, mw, n1, n1p, l0, H, in, a.A[t], cols, col); break;
            case 2: ff_rows<T, 2>(xl, mw, n1, n1p, l0, H, in, a.A[t], cols, col); break;
            case 3: ff_rows<T, 3>(xl, mw, n1, n1p, l0, H, in, a.A[t], cols, col); break;
            default: ff_rows<T, FF_RW>(xl, mw, n1, n1p, l0, H, in, a.A[t], cols, col); break;
        }
    }
}

// 32 x 32 tiles of V: rows of A along the lanes, written through shared memory along V's columns
template <typename T>
__global__ void __launch_bounds__(FF_OUT_T) fd_fold_out_kernel(const FdFold<T> a, TuckerDesc* vd, int* err, double* prof, int p) {
    if (blockIdx.x == 0)
        fd_desc(a.sd, a.omega, a.lmin, a.RP, vd, a.vcap, err, prof, a.n, a.n1, a.n2, p, (int)sizeof(T));
    __shared__ T tile[FF_TC][FF_TC + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = a.n;
    const int rt = (n + FF_TC - 1) / FF_TC;
    int tiles[3], tot = 0;
    for (int t = 0; t < 3; ++t) {
        tiles[t] = (ff_cols(a, t) + FF_TC - 1) / FF_TC;
        tot += tiles[t];
    }
    for (int w = blockIdx.x; w < tot * rt; w += gridDim.x) {
        int ct = w / rt, t = 0;
        const int i0 = (w % rt) * FF_TC;
        while (ct >= tiles[t]) ct -= tiles[t++];
        const int r = a.sd->rank[t], cols = a.RP * r, c0 = ct * FF_TC;
        const int col = c0 + lane, j = col < cols ? col / r : 0, c = col < cols ? col - j * r : 0;
        const T* __restrict__ A = a.A[t];
        __syncthreads();
        constexpr int NW = FF_OUT_T / 32, RPW = FF_TC / NW;
        int k0[RPW], k1[RPW];
        T acc[RPW];
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
            const int i = i0 + warp + NW * q;
            const bool in = i < n && col < cols;
            k0[q] = in ? a.wrow[i] : 0;
            k1[q] = in ? a.wrow[i + 1] : 0;
        }
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
            const bool has = k0[q] < k1[q];
            acc[q] = has ? a.wval[k0[q]] * A[(long long)a.wcol[k0[q]] * cols + col] : T(0);
        }
        T b[RPW];
#pragma unroll
        for (int q = 0; q < RPW; ++q) b[q] = T(0);
        if (col < cols)
            for (int e = 0; e < a.n2; ++e) {
                const T z = a.F[t][(long long)j * n + a.n1 + e] * a.u[t][(long long)(a.n1 + e) * r + c];
#pragma unroll
                for (int q = 0; q < RPW; ++q) {
                    const int i = i0 + warp + NW * q;
                    if (i < n) b[q] = fma(a.v2u2[i + (long long)e * n], z, b[q]);
                }
            }
#pragma unroll
        for (int q = 0; q < RPW; ++q) {
            for (int k = k0[q] + 1; k < k1[q]; ++k) acc[q] = fma(a.wval[k], A[(long long)a.wcol[k] * cols + col], acc[q]);
            tile[warp + NW * q][lane] = acc[q] + b[q];
        }
        __syncthreads();
        T* __restrict__ V = a.V[t];
        for (int k = warp; k < FF_TC; k += FF_OUT_T / 32)
            if (i0 + lane < n && c0 + k < cols) V[i0 + lane + (long long)(c0 + k) * n] = tile[lane][k];
    }
}

// The halves while they beat the FFTs: n = 256 above; n = 384 and rank 64 FP64 650 us against 528 with the FFTs, FP32 73 against
// 137 us; n = 512 FP64 1900 against 533, FP32 213 against 141 us.  (In FP32 their rounding passes the FFTs' between.)
bool fd_fold_fits(tpcg_problem pb) { return pb->dst_sym && pb->n1 <= FD_FOLD_MAX; }

template <typename T>
int fd_fold(tpcg_problem pb, tpcg_ctx c, const tucker_t* s, tucker_t* v, const double* cw, double lmin, int* err,
            cudaStream_t st) {
    FdFold<T> a;
    a.sd = static_cast<const TuckerDesc*>(s->desc);
    for (int t = 0; t < 3; ++t) {
        a.S[t] = static_cast<const T*>(s->U[t]);
        a.F[t] = static_cast<T*>(c->fd[t][0]);
        a.u[t] = static_cast<T*>(c->fd[t][1]);
        a.A[t] = static_cast<T*>(c->fd[t][3]);
        a.V[t] = static_cast<T*>(v->U[t]);
        a.cw[t] = cw[t];
    }
    a.wtrow = pb->d_wtrow; a.wtcol = pb->d_wtcol; a.wrow = pb->d_wrow; a.wcol = pb->d_wcol;
    a.wtval = static_cast<const T*>(pb->d_wtval);
    a.wval = static_cast<const T*>(pb->d_wval);
    a.v2u2 = static_cast<const T*>(pb->d_v2u2);
    a.dst = static_cast<const T*>(pb->d_dst);
    a.lam = static_cast<const T*>(pb->d_lam);
    a.mu = static_cast<const T*>(pb->d_mu);
    a.alpha = pb->d_alpha;
    a.omega = pb->d_omega;
    a.lmin = lmin;
    a.n = pb->n; a.n1 = pb->n1; a.n2 = pb->n2; a.RP = pb->RP; a.vcap = v->cap;
    a.sms = sm_count();
    const int n1 = a.n1, kmax = std::max(1, v->cap / a.RP);   // the largest input rank with an output that fits
    const int tiles = (kmax + FF_TC - 1) / FF_TC;
    a.chunks = (n1 + FF_FWD_T / 32 - 1) / (FF_FWD_T / 32);
    fd_fold_fwd_kernel<T><<<dim3(tiles, a.chunks + FF_REST, 3), FF_FWD_T, ff_fwd_smem<T>(n1), st>>>(a);
    TPCG_CHECK_LAUNCH();
    const int H = (n1 + 1) / 2;
    const long long ct = 3LL * ((v->cap + FF_TC - 1) / FF_TC);
    fd_fold_inv_kernel<T><<<(int)std::min<long long>(4 * a.sms, ct * ((H + 3) / 4)), FF_INV_T,
                            ff_inv_smem<T>(n1), st>>>(a);
    TPCG_CHECK_LAUNCH();
    fd_fold_out_kernel<T><<<(int)std::min<long long>(4 * a.sms, ct * ((a.n + FF_TC - 1) / FF_TC)), FF_OUT_T, 0, st>>>(
        a, static_cast<TuckerDesc*>(v->desc), err, prof_dev(), pb->p);
    TPCG_CHECK_LAUNCH();
    return TPCG_OK;
}
template int fd_fold<double>(tpcg_problem, tpcg_ctx, const tucker_t*, tucker_t*, const double*, double, int*, cudaStream_t);
template int fd_fold<float>(tpcg_problem, tpcg_ctx, const tucker_t*, tucker_t*, const double*, double, int*, cudaStream_t);

template <typename T>
static int fd_fold_prepare_one() {
    const int fwd = (int)ff_fwd_smem<T>(FD_FOLD_MAX), inv = (int)ff_inv_smem<T>(FD_FOLD_MAX);
    TPCG_CUDA(cudaFuncSetAttribute(fd_fold_fwd_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, fwd));
    TPCG_CUDA(cudaFuncSetAttribute(fd_fold_inv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, inv));
    return TPCG_OK;
}

int fd_fold_prepare() {
    static PerDevice device;
    return device.prepare([](bool*) {
        TPCG_TRY(fd_fold_prepare_one<double>());
        return fd_fold_prepare_one<float>();
    });
}

}  // namespace tpcg
