// Complex GEMM on the CUDA cores: C = beta C + alpha A B for column-major views.
//
// FP64 (Z64, interleaved double2): the products of the FP64 path that are too small for digits (resid_tc.cu
// gemm_z64_dg), or have no room for them: Schur complement, LU updates; with few columns (right-hand sides)
// skinny_z64_kernel.  GB300 executes FP64 on the CUDA cores only, so this kernel is bound by the FP64
// pipe; it keeps a 64 x BN tile per CTA (BN = 16, 32 or 64, whichever pads the column count
// least) with 4 x BN/16 complex accumulators per thread staged through shared memory.
// FP32 (C32, planar): updates inside the LU panels of the pivot search.
// Mixed (A hi parts of split planes, C FP64, B FP32, FP32 arithmetic): the ordinary system's refinement
// residual update r -= A d for a small correction d.
#include "common.cuh"
#include "kernels.cuh"

#include <algorithm>
#include <type_traits>

namespace {

constexpr int BK = 16;

template <class R> BM_HD cplx_t<R> conv(double2 v);
template <class R> BM_HD cplx_t<R> conv(float2 v);
template <> BM_HD double2 conv<double>(double2 v) { return v; }
template <> BM_HD float2 conv<float>(float2 v) { return v; }

template <class VC> BM_HD typename VC::cv from_acc(double2 v) {
    typename VC::cv r;
    r.x = (typename VC::real)v.x;
    r.y = (typename VC::real)v.y;
    return r;
}
template <class VC> BM_HD typename VC::cv from_acc(float2 v) {
    typename VC::cv r;
    r.x = (typename VC::real)v.x;
    r.y = (typename VC::real)v.y;
    return r;
}

// VA, VB, VC: storage views of A, B, C; R: arithmetic precision
template <class VA, class VB, class VC, class R, int BM, int BN>
__global__ void __launch_bounds__(256) cgemm_simt_kernel(int m, int n, int k, VA A, VB B, VC C, R alpha, R beta,
                                                         const int* stop) {
    using CV = cplx_t<R>;
    constexpr int TM = BM / 16, TN = BN / 16;
    pdl_wait();
    pdl_trigger();
    if (stop != nullptr && *stop != 0) return;  // a factorisation that stopped (lu_fast_z.cu)
    __shared__ CV As[BK][BM + 1];
    __shared__ CV Bs[BK][BN + 1];
    const int t = threadIdx.x;
    const int tx = t % 16, ty = t / 16;
    const long i0 = (long)blockIdx.x * BM, j0 = (long)blockIdx.y * BN;
    CV acc[TM][TN];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int b = 0; b < TN; ++b) acc[a][b] = czero<R>();

    for (int k0 = 0; k0 < k; k0 += BK) {
#pragma unroll
        for (int e = t; e < BM * BK; e += 256) {
            const int ii = e % BM, kk = e / BM;
            long gi = i0 + ii;
            int gk = k0 + kk;
            CV v = czero<R>();
            if (gi < m && gk < k) v = conv<R>(A.get(gi, gk));
            As[kk][ii] = v;
        }
#pragma unroll
        for (int e = t; e < BN * BK; e += 256) {
            int kk = e % BK, jj = e / BK;
            long gj = j0 + jj;
            int gk = k0 + kk;
            CV v = czero<R>();
            if (gj < n && gk < k) v = conv<R>(B.get(gk, gj));
            Bs[kk][jj] = v;
        }
        __syncthreads();
#pragma unroll 4
        for (int kk = 0; kk < BK; ++kk) {
            CV av[TM], bv[TN];
#pragma unroll
            for (int a = 0; a < TM; ++a) av[a] = As[kk][tx + 16 * a];
#pragma unroll
            for (int b = 0; b < TN; ++b) bv[b] = Bs[kk][ty + 16 * b];
#pragma unroll
            for (int a = 0; a < TM; ++a)
#pragma unroll
                for (int b = 0; b < TN; ++b) cfma(acc[a][b], av[a], bv[b]);
        }
        __syncthreads();
    }
    // all of this thread's C reads are issued before its first write (the compiler cannot move a
    // read of C past a write to C, so interleaving them would cost one memory latency each)
    using OCV = typename VC::cv;
    OCV cin[TM][TN];
    if (beta != (R)0) {
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int b = 0; b < TN; ++b) {
                const long gi = i0 + tx + 16 * a, gj = j0 + ty + 16 * b;
                if (gi < m && gj < n) cin[a][b] = C.get(gi, gj);
            }
    }
#pragma unroll
    for (int a = 0; a < TM; ++a) {
        long gi = i0 + tx + 16 * a;
        if (gi >= m) continue;
#pragma unroll
        for (int b = 0; b < TN; ++b) {
            long gj = j0 + ty + 16 * b;
            if (gj >= n) continue;
            CV r;
            r.x = alpha * acc[a][b].x;
            r.y = alpha * acc[a][b].y;
            OCV out = from_acc<VC>(r);
            if (beta != (R)0) {
                out.x += (typename VC::real)beta * cin[a][b].x;
                out.y += (typename VC::real)beta * cin[a][b].y;
            }
            C.set(gi, gj, out);
        }
    }
}

template <class VA, class VB, class VC, class R>
cudaError_t launch_impl(cudaStream_t s, int m, int n, int k, VA A, VB B, VC C, R alpha, R beta,
                        const int* stop = nullptr) {
    if (m <= 0 || n <= 0) return cudaSuccess;
    // every launch may overlap the previous kernel's tail: the kernel waits (pdl_wait) before it
    // reads anything
    auto go = [&](auto kern, dim3 grid) { return launch_pdl(kern, grid, dim3(256), 0, s, m, n, k, A, B, C, alpha, beta, stop); };
    // Few right-hand sides (n <= 80, e.g. 65): one column tile covers them all, so A is streamed
    // once; 32-row tiles when 64-row ones would leave SMs idle.
    if (n > 32 && n <= 80) {
        if ((long)ceil_div(m, 64) >= 2 * 152)
            return go(cgemm_simt_kernel<VA, VB, VC, R, 64, 80>, dim3(ceil_div(m, 64), 1));
        return go(cgemm_simt_kernel<VA, VB, VC, R, 32, 80>, dim3(ceil_div(m, 32), 1));
    }
    // FP64 products too small to fill the GPU with 64-row tiles (the FP64 pipe gives each SM only
    // ~8 GFLOP/s, so idle SMs cost directly): 32 x 16 tiles
    if constexpr (std::is_same<R, double>::value) {
        static int sms = 0;
        if (sms == 0) {
            int dev = 0, v = 0;
            if (cudaGetDevice(&dev) == cudaSuccess &&
                cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
                sms = v;
            else
                sms = 1;
        }
        if ((long)ceil_div(m, 64) * ceil_div(n, 64) < sms)
            return go(cgemm_simt_kernel<VA, VB, VC, R, 32, 16>, dim3(ceil_div(m, 32), ceil_div(n, 16)));
    }
    // otherwise the column tile with the least padding (ties go to the wider tile)
    int bn = 64;
    long best = (long)ceil_div(n, 64) * 64 - n;
    for (int cand : {32, 16}) {
        long waste = (long)ceil_div(n, cand) * cand - n;
        if (waste < best) {
            best = waste;
            bn = cand;
        }
    }
    if (bn == 16) return go(cgemm_simt_kernel<VA, VB, VC, R, 64, 16>, dim3(ceil_div(m, 64), ceil_div(n, 16)));
    if (bn == 32) return go(cgemm_simt_kernel<VA, VB, VC, R, 64, 32>, dim3(ceil_div(m, 64), ceil_div(n, 32)));
    return go(cgemm_simt_kernel<VA, VB, VC, R, 64, 64>, dim3(ceil_div(m, 64), ceil_div(n, 64)));
}

// FP64 products with few columns (right-hand sides): C = beta C + alpha A B.  The tiles of the kernel above
// would leave most SMs idle (1000 rows: 32 CTAs) and pad the columns to 16, on a pipe of two multiply-adds
// a cycle per SM.  Here a CTA takes 32 rows x NC columns x one of S slices of K (a cluster of S CTAs); a
// warp takes every eighth k of the slice for all NC columns, lane = row, A straight from memory
// (coalesced), B's chunk broadcast from shared memory.  The warps' sums, then the slices', are added in
// order (through shared memory and the cluster's), so the result does not depend on scheduling.
// FP64-bound: N = 1000, four right-hand sides, both products of a solve 1.74 -> 0.2 ms.
constexpr int SK_W = 8, SK_K = 64;
template <int NC>
__global__ void __launch_bounds__(SK_W * 32) skinny_z64_kernel(int m, int n, int k, double alpha, Z64 A, Z64 B,
                                                               double beta, Z64 C) {
    __shared__ double2 Bs[SK_K][NC];
    __shared__ double2 Ps[SK_W][NC][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int S = (int)gridDim.x, z = (int)blockIdx.x;
    const long i = (long)blockIdx.y * 32 + lane;
    const int j0 = (int)blockIdx.z * NC, nc = min(NC, n - j0);
    const int kb = (int)((long)z * k / S), ke = (int)((long)(z + 1) * k / S);
    pdl_wait();
    pdl_trigger();
    double2 acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = make_double2(0.0, 0.0);
    for (int k0 = kb; k0 < ke; k0 += SK_K) {
        const int kn = min(SK_K, ke - k0);
        double2 a[SK_K / SK_W];
#pragma unroll
        for (int u = 0; u < SK_K / SK_W; ++u) {
            const int kk = warp + SK_W * u;
            a[u] = (kk < kn && i < m) ? A.get(i, k0 + kk) : make_double2(0.0, 0.0);
        }
        __syncthreads();  // the previous chunk has been read
        for (int e = threadIdx.x; e < SK_K * NC; e += SK_W * 32) {
            const int kk = e % SK_K, c = e / SK_K;
            Bs[kk][c] = (kk < kn && c < nc) ? B.get(k0 + kk, (long)j0 + c) : make_double2(0.0, 0.0);
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < SK_K / SK_W; ++u) {
            const int kk = warp + SK_W * u;
            if (kk < kn) {  // warp-uniform
#pragma unroll
                for (int c = 0; c < NC; ++c) cfma(acc[c], a[u], Bs[kk][c]);
            }
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) Ps[warp][c][lane] = acc[c];
    __syncthreads();
    for (int e = threadIdx.x; e < NC * 32; e += SK_W * 32) {
        double2 s = Ps[0][e / 32][e % 32];
#pragma unroll
        for (int w = 1; w < SK_W; ++w) s = cadd(s, Ps[w][e / 32][e % 32]);
        Ps[0][e / 32][e % 32] = s;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    // rank z adds the slices of its share of the outputs
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(&Ps[0][0][0]);
    for (int e = z * SK_W * 32 + (int)threadIdx.x; e < NC * 32; e += S * SK_W * 32) {
        double2 s = make_double2(0.0, 0.0);
        for (int r = 0; r < S; ++r) {
            uint32_t ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(base + (uint32_t)e * 16u), "r"(r));
            double2 v;
            asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(ra) : "memory");
            s = cadd(s, v);
        }
        const long row = (long)blockIdx.y * 32 + e % 32;
        const int c = e / 32;
        if (row < m && c < nc) {
            double2 o = cscale(s, alpha);
            if (beta != 0.0) {
                const double2 c0 = C.get(row, (long)j0 + c);
                o.x = fma(beta, c0.x, o.x);
                o.y = fma(beta, c0.y, o.y);
            }
            C.set(row, (long)j0 + c, o);
        }
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <int NC>
cudaError_t launch_skinny_z64(cudaStream_t s, dim3 grid, int m, int n, int k, double alpha, Z64 A, Z64 B, double beta,
                              Z64 C) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(SK_W * 32);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid.x;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, skinny_z64_kernel<NC>, m, n, k, alpha, A, B, beta, C);
}

}  // namespace

// The products of the FP64 solves and residuals.  Column tiles of at most 9 (shared memory), evenly wide; K slices until
// about two CTAs per SM are busy.
cudaError_t gemm_z64_skinny(cudaStream_t s, int num_sms, int m, int n, int k, double alpha, Z64 A, Z64 B, double beta,
                            Z64 C) {
    if (m <= 0 || n <= 0) return cudaSuccess;
    if (k <= 0) return gemm_z64(s, m, n, k, alpha, A, B, beta, C);
    const int t = ceil_div(n, 9), nc = ceil_div(n, t), rt = ceil_div(m, 32);
    const int S = (int)std::max(1L, std::min(std::min(8L, (long)ceil_div(k, SK_K)), (long)ceil_div(2L * num_sms, (long)rt * t)));
    auto go = [&](auto w) {
        constexpr int NC = decltype(w)::value;
        return launch_skinny_z64<NC>(s, dim3(S, rt, ceil_div(n, NC)), m, n, k, alpha, A, B, beta, C);
    };
    switch (nc) {
        case 1: return go(std::integral_constant<int, 1>{});
        case 2: return go(std::integral_constant<int, 2>{});
        case 3: return go(std::integral_constant<int, 3>{});
        case 4: return go(std::integral_constant<int, 4>{});
        case 5: return go(std::integral_constant<int, 5>{});
        case 6: return go(std::integral_constant<int, 6>{});
        case 7: return go(std::integral_constant<int, 7>{});
        case 8: return go(std::integral_constant<int, 8>{});
        default: return go(std::integral_constant<int, 9>{});
    }
}

cudaError_t gemm_z64(cudaStream_t s, int m, int n, int k, double alpha, Z64 A, Z64 B, double beta, Z64 C,
                     const int* stop) {
    if (k <= 0 && beta == 1.0) return cudaSuccess;
    return launch_impl<Z64, Z64, Z64, double>(s, m, n, k, A, B, C, alpha, beta, stop);
}

cudaError_t gemm_c32(cudaStream_t s, int m, int n, int k, float alpha, C32 A, C32 B, float beta, C32 C) {
    if (k <= 0 && beta == 1.0f) return cudaSuccess;
    return launch_impl<C32, C32, C32, float>(s, m, n, k, A, B, C, alpha, beta);
}

// C (FP64) += alpha A_hi (FP32 hi parts of split planes) B (FP32 planar), FP32 arithmetic
cudaError_t gemm_update_f4hi_c32(cudaStream_t s, int m, int n, int k, float alpha, F4Hi A, C32 B, Z64 C) {
    if (k <= 0) return cudaSuccess;
    return launch_impl<F4Hi, C32, Z64, float>(s, m, n, k, A, B, C, alpha, 1.0f);
}
