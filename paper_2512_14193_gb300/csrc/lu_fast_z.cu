// FP64 LU with the pivots kept on the diagonal while partial pivoting would keep them there (the FP64
// counterpart of lu_fast.cu): blocks of 32 columns without a pivot search, every candidate compared with
// its pivot.  When one is larger (or a pivot is zero or a NaN) *fail names the block, the remaining kernels of the
// sequence return, and the host restores the block and goes on from it with the search (lu_resume_enqueue).
//
// An SM does two FP64 multiply-adds a cycle, so a warp instruction costs 16 cycles of its pipe whatever the
// number of active lanes: the diagonal block stays small (32 columns, 67 us on one SM, of which its FP64
// instructions take a third: the elimination's chain is the rest), the solves and the
// rest of the trailing matrix are spread over all SMs, and outer blocks of 128 columns are applied by the
// tensor cores (gemm_z64_dg).
#include "lu_internal.cuh"

namespace lu_detail {
namespace {

constexpr int B = FZ_BLOCK, W = 8, P = B + 1;  // block, sub-step, row pitch in shared memory

__device__ __forceinline__ double2 shfl2(double2 v, int l) {
    return make_double2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
// a - b c
__device__ __forceinline__ double2 csubmul(double2 a, double2 b, double2 c) {
    return make_double2(fma(-b.x, c.x, fma(b.y, c.y, a.x)), fma(-b.x, c.y, fma(-b.y, c.x, a.y)));
}
// 1 / a for a != 0 with nine FP64 instructions (a division takes about thirty): a is scaled by a power of
// two to |a|_inf in [1, 2), 1 / |a|^2 starts from the FP32 reciprocal and takes two Newton steps (2^-23 ->
// 2^-46 -> rounding), a few ulps in all.
__device__ __forceinline__ double2 cinv_newton(double2 a) {
    const long long bx = __double_as_longlong(a.x) & 0x7FFFFFFFFFFFFFFFll, by = __double_as_longlong(a.y) & 0x7FFFFFFFFFFFFFFFll;
    const int e = (int)(max(bx, by) >> 52);
    if (e == 0 || e >= 2045) return cinv(a);  // subnormal, huge or not finite
    const double sc = __longlong_as_double((long long)(2046 - e) << 52);  // 2^(1023 - e)
    const double x = a.x * sc, y = a.y * sc;
    const double d = fma(x, x, y * y);  // in [1, 8)
    float rf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"((float)d));
    double r = (double)rf;
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    r *= sc;
    return make_double2(x * r, -y * r);
}
// |Re| + |Im|
__device__ __forceinline__ double n1(double2 a) { return fabs(a.x) + fabs(a.y); }

// Eliminates the 8 x 8 block at (c0, c0): one warp, lane = row + 8 (pair of columns).
__device__ __forceinline__ bool diag8(double2* S, int c0, double2* inv_s, double2* piv_s) {
    const int lane = threadIdx.x & 31, r = lane & 7, g = lane >> 3;
    double2* row = S + (c0 + r) * P + c0;
    double2 x[2] = {row[2 * g], row[2 * g + 1]};
    bool ok = true;
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const double2 p = shfl2(x[c & 1], c + 8 * (c / 2));
        const double2 arc = shfl2(x[c & 1], r + 8 * (c / 2));  // this row's entry of column c
        const double2 u0 = shfl2(x[0], c + 8 * g), u1 = shfl2(x[1], c + 8 * g);
        const double2 iv = cinv_newton(p);
        const double pn = n1(p);
        ok = ok && pn > 0.0 && (r <= c || n1(arc) <= pn);
        if (lane == 0) {
            inv_s[c0 + c] = iv;
            piv_s[c0 + c] = p;
        }
        const double2 l = cmul(arc, iv);
        if (r > c) {
            if (2 * g > c) x[0] = csubmul(x[0], l, u0);
            else if (2 * g == c) x[0] = l;
            if (2 * g + 1 > c) x[1] = csubmul(x[1], l, u1);
            else if (2 * g + 1 == c) x[1] = l;
        }
    }
    row[2 * g] = x[0];
    row[2 * g + 1] = x[1];
    __syncwarp();
    return ok;
}

__global__ void __launch_bounds__(256, 1) lu_diag_z_kernel(Z64 F, int J, int db, double2* __restrict__ T, int* fail) {
    __shared__ double2 S[B * P];
    __shared__ double2 inv_s[B], piv_s[B];
    __shared__ int bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (*reinterpret_cast<volatile int*>(fail) != 0) return;
    if (tid == 0) bad = 0;
    const int be = (db + W - 1) & ~(W - 1);  // past it the block is the identity's, which needs no elimination
    if (tid >= be && tid < B) inv_s[tid] = piv_s[tid] = make_double2(1.0, 0.0);
#pragma unroll
    for (int q = 0; q < B / 8; ++q) {
        const int c = warp + 8 * q;
        const bool in = lane < db && c < db;
        S[lane * P + c] = in ? F.get(J + lane, J + c) : make_double2(lane == c ? 1.0 : 0.0, 0.0);
    }
    __syncthreads();
    bool ok = true;
#pragma unroll 1
    for (int c0 = 0; c0 < be; c0 += W) {
        if (warp == 0) ok = diag8(S, c0, inv_s, piv_s) && ok;
        __syncthreads();
        const int t0 = c0 + W, rest = be - t0;
        if (warp == 0 && lane < rest) {  // a row below
            double2* row = S + (t0 + lane) * P + c0;
            double2 a[W];
#pragma unroll
            for (int k = 0; k < W; ++k) a[k] = row[k];
#pragma unroll
            for (int c = 0; c < W; ++c) {
                ok = ok && n1(a[c]) <= n1(piv_s[c0 + c]);
                a[c] = cmul(a[c], inv_s[c0 + c]);
#pragma unroll
                for (int k = c + 1; k < W; ++k) a[k] = csubmul(a[k], a[c], S[(c0 + c) * P + c0 + k]);
            }
#pragma unroll
            for (int k = 0; k < W; ++k) row[k] = a[k];
        } else if (warp == 1 && lane < rest) {  // a column on the right
            double2* col = S + c0 * P + t0 + lane;
            double2 x[W];
#pragma unroll
            for (int k = 0; k < W; ++k) x[k] = col[k * P];
#pragma unroll
            for (int k = 1; k < W; ++k)
#pragma unroll
                for (int c = 0; c < k; ++c) x[k] = csubmul(x[k], S[(c0 + k) * P + c0 + c], x[c]);
#pragma unroll
            for (int k = 1; k < W; ++k) col[k * P] = x[k];
        }
        __syncthreads();
        for (int e = tid; e < rest * rest; e += 256) {
            const int i = t0 + e / rest, j = t0 + e % rest;
            double2 v = S[i * P + j];
#pragma unroll
            for (int k = 0; k < W; ++k) v = csubmul(v, S[i * P + c0 + k], S[(c0 + k) * P + j]);
            S[i * P + j] = v;
        }
        __syncthreads();
    }
    if (!ok) bad = 1;
    __syncthreads();
    if (bad) {
        if (tid == 0) *reinterpret_cast<volatile int*>(fail) = 2 * (J + 1);
        return;
    }
    const FzT t(T);
    // U and L^T as rows [p][k], their 8 x 8 diagonal blocks inverted: warps 0 and 1 (a column per lane)
    if (warp < 2) {
        const bool up = warp == 0;
        const int d0 = lane & ~(W - 1), j = lane & (W - 1);
        double2 x[W];
#pragma unroll
        for (int i = W - 1; i >= 0; --i) {
            double2 s = make_double2(i == j ? 1.0 : 0.0, 0.0);
#pragma unroll
            for (int k = i + 1; k < W; ++k)
                s = csubmul(s, up ? S[(d0 + i) * P + d0 + k] : S[(d0 + k) * P + d0 + i], x[k]);
            x[i] = up ? cmul(s, inv_s[d0 + i]) : s;
        }
        double2* g = up ? t.U : t.L;
#pragma unroll
        for (int i = 0; i < W; ++i) g[(d0 + i) * B + d0 + j] = x[i];
    }
#pragma unroll
    for (int q = 0; q < B / 8; ++q) {
        const int p = warp + 8 * q;
        t.F[p * B + lane] = S[p * P + lane];
        if (lane / W > p / W) {
            t.U[p * B + lane] = S[p * P + lane];
            t.L[p * B + lane] = S[lane * P + p];
        }
    }
    if (tid < B) t.piv[tid] = piv_s[tid];
}

// L21 = A21 U11^{-1} by rows and U12 = L11^{-1} A12 by columns, x T = a in chunks of 8 entries as in
// lu_trsm_kernel: a CTA takes 16 rows or columns, eight threads each (one entry of a chunk per thread).
// FP64-bound: 320 warp instructions per four rows.  The last CTA writes the diagonal block's factors.  Every
// CTA saves what it overwrites.
constexpr int R = 16;
__global__ void __launch_bounds__(128) lu_trsm_z_kernel(Z64 F, int J, int db, int mm, const double2* __restrict__ T,
                                                        double2* __restrict__ bk, long n, int* fail) {
    __shared__ double2 Ts[B * B];
    __shared__ double2 Xs[R][P];
    __shared__ double2 piv_s[B];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const int f = *reinterpret_cast<volatile int*>(fail);
        if (f != 0 && f != 2 * (J + 1) + 1) return;
    }
    const FzT t(const_cast<double2*>(T));
    const FzBackup b(bk, n);
    const int nr = (mm + R - 1) / R;
    if ((int)blockIdx.x == 2 * nr) {
#pragma unroll
        for (int q = 0; q < B / 4; ++q) {
            const int j = warp + 4 * q;
            if (lane < db && j < db) {
                b.D[lane + j * B] = F.get(J + lane, J + j);
                F.set(J + lane, J + j, t.F[lane * B + j]);
            }
        }
        return;
    }
    const bool rows = (int)blockIdx.x < nr;
    const int x0 = ((int)blockIdx.x - (rows ? 0 : nr)) * R;
    const double2* src = rows ? t.U : t.L;
#pragma unroll
    for (int q = 0; q < B * B / 128; ++q) Ts[tid + 128 * q] = src[tid + 128 * q];
    if (tid < B) piv_s[tid] = t.piv[tid];
    if (rows) {
        const int r = tid & 15, k0 = tid >> 4;
#pragma unroll
        for (int q = 0; q < B / 8; ++q) {
            const int k = k0 + 8 * q;
            double2 v = make_double2(0.0, 0.0);
            if (x0 + r < mm) {
                v = F.get(J + B + x0 + r, J + k);
                b.L[x0 + r + k * n] = v;
            }
            Xs[r][k] = v;
        }
    } else {
#pragma unroll
        for (int q = 0; q < R / 4; ++q) {
            const int c = warp + 4 * q;
            double2 v = make_double2(0.0, 0.0);
            if (x0 + c < mm) {
                v = F.get(J + lane, J + B + x0 + c);
                b.U[lane + (long)(x0 + c) * B] = v;
            }
            Xs[c][lane] = v;
        }
    }
    __syncthreads();
    const int row = warp * 4 + (lane >> 3), q = lane & 7;
    bool ok = true;
#pragma unroll 1
    for (int j0 = 0; j0 < B; j0 += W) {
        double2 a = Xs[row][j0 + q];
        for (int p0 = 0; p0 < j0; p0 += W)
#pragma unroll
            for (int p = 0; p < W; ++p) a = csubmul(a, Xs[row][p0 + p], Ts[(p0 + p) * B + j0 + q]);
        __syncwarp();
        Xs[row][j0 + q] = a;
        __syncwarp();
        double2 y = make_double2(0.0, 0.0);
#pragma unroll
        for (int p = 0; p < W; ++p)  // (T^{-1} is zero below its diagonal)
            if (p <= q) cfma(y, Xs[row][j0 + p], Ts[(j0 + p) * B + j0 + q]);
        if (rows) {
            const double2 u = piv_s[j0 + q];
            ok = ok && n1(cmul(y, u)) <= n1(u);
        }
        __syncwarp();
        Xs[row][j0 + q] = y;
        __syncwarp();
    }
    if (!ok) atomicCAS(fail, 0, 2 * (J + 1) + 1);
    __syncthreads();
    if (rows) {
        const int r = tid & 15, k0 = tid >> 4;
        if (x0 + r < mm)
#pragma unroll
            for (int qq = 0; qq < B / 8; ++qq) F.set(J + B + x0 + r, J + k0 + 8 * qq, Xs[r][k0 + 8 * qq]);
    } else {
#pragma unroll
        for (int qq = 0; qq < R / 4; ++qq) {
            const int c = warp + 4 * qq;
            if (x0 + c < mm) F.set(J + lane, J + B + x0 + c, Xs[c][lane]);
        }
    }
}

// the entries lu_trsm_z_kernel overwrote, back into the matrix
__global__ void lu_restore_z_kernel(Z64 F, int J, int db, int mm, double2* __restrict__ bk, long n) {
    const FzBackup b(bk, n);
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long nl = (long)mm * B;
    if (e < nl) {
        const long r = e % mm, k = e / mm;
        F.set(J + B + r, J + k, b.L[r + k * n]);
    } else if (e < 2 * nl) {
        const long k = (e - nl) % B, c = (e - nl) / B;
        F.set(J + k, J + B + c, b.U[k + c * B]);
    } else if (e - 2 * nl < B * B) {
        const int i = (int)((e - 2 * nl) % B), j = (int)((e - 2 * nl) / B);
        if (i < db && j < db) F.set(J + i, J + j, b.D[i + j * B]);
    }
}

}  // namespace

cudaError_t launch_lu_diag_z(cudaStream_t s, Z64 F, int J, int db, double2* work, int* fail) {
    lu_diag_z_kernel<<<1, 256, 0, s>>>(F, J, db, work, fail);
    return cudaGetLastError();
}

cudaError_t launch_lu_trsm_z(cudaStream_t s, Z64 F, int J, int db, int mm, double2* work, long n, int* fail) {
    if (mm > 0 && db != B) return cudaErrorInvalidValue;
    lu_trsm_z_kernel<<<2 * ceil_div(mm, R) + 1, 128, 0, s>>>(F, J, db, mm, work, work + FZ_T, n, fail);
    return cudaGetLastError();
}

cudaError_t launch_lu_restore_z(cudaStream_t s, Z64 F, int J, int db, int mm, double2* work, long n) {
    const long t = 2L * mm * B + B * B;
    lu_restore_z_kernel<<<ceil_div(t, 256), 256, 0, s>>>(F, J, db, mm, work + FZ_T, n);
    return cudaGetLastError();
}

}  // namespace lu_detail
