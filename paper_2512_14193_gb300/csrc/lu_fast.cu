// FP32 LU with the pivots kept on the diagonal while partial pivoting would keep them there.
//
// Partial pivoting (pivot = first index of max |Re| + |Im|) rarely interchanges a row of U33 or of the
// ordinary matrix: the largest candidate below the diagonal is usually 0.5-0.9 of the diagonal entry.
// The pivot search of panel_lc.cu pays a cluster-wide exchange per column (2800-4500 cycles) to find
// that out.  Here a block of 128 columns is factored without a search, every candidate that the
// elimination forms is compared with its pivot, and the first block where one is larger (or a pivot
// is zero or a NaN) stops the sequence: *fail = 2 (J + 1) + stage names the block, later kernels return
// at once, and the host restores that block's columns and rows and continues from it with the pivot
// search (factor_t in lu.cu).  So the pivots are always those of partial pivoting.
//
// Per block of FD_B = 128 columns at J:
//   lu_diag_kernel  one CTA: LU of the diagonal block (stage 0 of the check)
//   lu_trsm_kernel  all SMs: L21 = A21 U11^{-1} by rows (stage 1 of the check) and U12 = L11^{-1} A12
//                   by columns, written to the matrix and packed for the tensor cores; the original
//                   entries are kept in a backup until the next block
//   gemm_tc         A22 -= L21 U12 in 3xTF32: the next diagonal block's tile first, so that the next
//                   lu_diag_kernel runs beside the rest (look-ahead on two streams)
#include "lu_internal.cuh"

namespace lu_detail {
namespace {

constexpr int B = FD_B, PITCH = FD_PITCH, W = 16;  // block, row pitch of the shared block, sub-step width
constexpr int DT = 512;                            // threads of lu_diag_kernel

// Eliminates the 16 x 16 diagonal block at (c0, c0) of the shared block without interchanges: one
// warp, lane = row (lanes 16-31 repeat lanes 0-15), the row in registers.  Returns false if a
// candidate exceeds its pivot.  The chain per column is the pivot's broadcast, its reciprocal and one
// multiply-add (about 90 cycles); sixteen columns keep the unrolled code small.
__device__ __forceinline__ bool diag16(float* Sr, float* Si, int c0, float2* inv_s, float* thr_s) {
    const int lane = threadIdx.x & 31, r = lane & 15;
    float ar[W], ai[W];
    float* pr = Sr + (c0 + r) * PITCH + c0;
    float* pi = Si + (c0 + r) * PITCH + c0;
#pragma unroll
    for (int k = 0; k < W; k += 4) {
        const float4 x = *reinterpret_cast<const float4*>(pr + k), y = *reinterpret_cast<const float4*>(pi + k);
        ar[k] = x.x, ar[k + 1] = x.y, ar[k + 2] = x.z, ar[k + 3] = x.w;
        ai[k] = y.x, ai[k + 1] = y.y, ai[k + 2] = y.z, ai[k + 3] = y.w;
    }
    bool ok = true;
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const float2 u = make_float2(__shfl_sync(0xffffffffu, ar[c], c), __shfl_sync(0xffffffffu, ai[c], c));
        const float un = cnorm1(u);
        const float2 iv = cinv_fast(u);
        const bool below = r > c;
        ok = ok && un > 0.f && (!below || cnorm1(make_float2(ar[c], ai[c])) <= un);
        if (lane == c) {
            inv_s[c0 + c] = iv;
            thr_s[c0 + c] = un;
        }
        const float2 l = below ? cmul(make_float2(ar[c], ai[c]), iv) : make_float2(0.f, 0.f);
#pragma unroll
        for (int k = c + 1; k < W; ++k) {
            const float ur = __shfl_sync(0xffffffffu, ar[k], c), ui = __shfl_sync(0xffffffffu, ai[k], c);
            ar[k] = fmaf(-l.x, ur, fmaf(l.y, ui, ar[k]));
            ai[k] = fmaf(-l.x, ui, fmaf(-l.y, ur, ai[k]));
        }
        if (below) {
            ar[c] = l.x;
            ai[c] = l.y;
        }
    }
    if (lane < W) {
#pragma unroll
        for (int k = 0; k < W; k += 4) {
            *reinterpret_cast<float4*>(pr + k) = make_float4(ar[k], ar[k + 1], ar[k + 2], ar[k + 3]);
            *reinterpret_cast<float4*>(pi + k) = make_float4(ai[k], ai[k + 1], ai[k + 2], ai[k + 3]);
        }
    }
    __syncwarp();
    return ok;
}

// LU of the db x db diagonal block at (J, J) (padded to 128 with the identity), in shared memory in
// sub-steps of 16 columns: the rows below and the columns right of the 16 x 16 block are solved one per
// thread, then the rest takes the rank-16 update (a warp per 16 x 32 tile, 4 x 4 per thread) while warp
// 0 updates and eliminates the next 16 x 16 block.  One SM's FP32 rate bounds the early sub-steps
// (18k cycles of updates in all), the elimination chain the late ones.  The factors go to T for
// lu_trsm_kernel, which also writes them to the matrix: U's and L^T's strict upper triangles as rows
// [p][k], pitch 132, then the reciprocal pivots and the pivots' magnitudes.
__global__ void __launch_bounds__(DT, 1) lu_diag_kernel(C32 F, int J, int db, float* __restrict__ T, int* fail) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float2 inv_s[B];
    __shared__ float thr_s[B];
    __shared__ int bad;
    float* Sr = sm;
    float* Si = sm + B * PITCH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (*reinterpret_cast<volatile int*>(fail) != 0) return;
    if (tid == 0) bad = 0;
    {
        // lane = 8 rows x 4 columns: 32-byte sectors of the matrix, all 32 shared banks
        const int r = warp * 8 + (lane & 7), cs = lane >> 3;
#pragma unroll 8
        for (int q = 0; q < B / 4; ++q) {
            const int c = 4 * q + cs;
            const bool in = r < db && c < db;
            const long o = (long)(J + r) + (long)(J + c) * F.ld;
            Sr[r * PITCH + c] = in ? F.re[o] : (r == c ? 1.f : 0.f);
            Si[r * PITCH + c] = in ? F.im[o] : 0.f;
        }
    }
    __syncthreads();
    bool ok = true;
    if (warp == 0) ok = diag16(Sr, Si, 0, inv_s, thr_s);
    __syncthreads();
#pragma unroll 1
    for (int c0 = 0; c0 + W < B; c0 += W) {
        const int rest = B - c0 - W;
        if (tid < rest) {  // a row of L21
            float* pr = Sr + (c0 + W + tid) * PITCH + c0;
            float* pi = Si + (c0 + W + tid) * PITCH + c0;
            float ar[W], ai[W];
#pragma unroll
            for (int k = 0; k < W; k += 4) {
                const float4 x = *reinterpret_cast<const float4*>(pr + k), y = *reinterpret_cast<const float4*>(pi + k);
                ar[k] = x.x, ar[k + 1] = x.y, ar[k + 2] = x.z, ar[k + 3] = x.w;
                ai[k] = y.x, ai[k + 1] = y.y, ai[k + 2] = y.z, ai[k + 3] = y.w;
            }
#pragma unroll
            for (int c = 0; c < W; ++c) {
                ok = ok && cnorm1(make_float2(ar[c], ai[c])) <= thr_s[c0 + c];
                const float2 l = cmul(make_float2(ar[c], ai[c]), inv_s[c0 + c]);
                ar[c] = l.x;
                ai[c] = l.y;
                const float* ur = Sr + (c0 + c) * PITCH + c0;
                const float* ui = Si + (c0 + c) * PITCH + c0;
#pragma unroll
                for (int k = c + 1; k < W; ++k) {
                    ar[k] = fmaf(-l.x, ur[k], fmaf(l.y, ui[k], ar[k]));
                    ai[k] = fmaf(-l.x, ui[k], fmaf(-l.y, ur[k], ai[k]));
                }
            }
#pragma unroll
            for (int k = 0; k < W; k += 4) {
                *reinterpret_cast<float4*>(pr + k) = make_float4(ar[k], ar[k + 1], ar[k + 2], ar[k + 3]);
                *reinterpret_cast<float4*>(pi + k) = make_float4(ai[k], ai[k + 1], ai[k + 2], ai[k + 3]);
            }
        } else if (tid >= B && tid - B < rest) {  // a column of U12
            float* pr = Sr + c0 * PITCH + c0 + W + (tid - B);
            float* pi = Si + c0 * PITCH + c0 + W + (tid - B);
            float xr[W], xi[W];
#pragma unroll
            for (int k = 0; k < W; ++k) {
                xr[k] = pr[k * PITCH];
                xi[k] = pi[k * PITCH];
            }
#pragma unroll
            for (int c = 0; c < W - 1; ++c) {
#pragma unroll
                for (int k = c + 1; k < W; ++k) {
                    const float lr = Sr[(c0 + k) * PITCH + c0 + c], li = Si[(c0 + k) * PITCH + c0 + c];
                    xr[k] = fmaf(-lr, xr[c], fmaf(li, xi[c], xr[k]));
                    xi[k] = fmaf(-lr, xi[c], fmaf(-li, xr[c], xi[k]));
                }
            }
#pragma unroll
            for (int k = 1; k < W; ++k) {
                pr[k * PITCH] = xr[k];
                pi[k * PITCH] = xi[k];
            }
        }
        __syncthreads();
        const int t0 = c0 + W;  // first row and column of the rest
        if (warp == 0) {
            // the next 16 x 16 block: lane = row x half of the columns
            const int r = lane & 15, h = (lane >> 4) * 8;
            float* pr = Sr + (t0 + r) * PITCH + t0 + h;
            float* pi = Si + (t0 + r) * PITCH + t0 + h;
            float ar[8], ai[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                ar[k] = pr[k];
                ai[k] = pi[k];
            }
#pragma unroll 4
            for (int c = 0; c < W; ++c) {
                const float lr = Sr[(t0 + r) * PITCH + c0 + c], li = Si[(t0 + r) * PITCH + c0 + c];
                const float* ur = Sr + (c0 + c) * PITCH + t0 + h;
                const float* ui = Si + (c0 + c) * PITCH + t0 + h;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    ar[k] = fmaf(-lr, ur[k], fmaf(li, ui[k], ar[k]));
                    ai[k] = fmaf(-lr, ui[k], fmaf(-li, ur[k], ai[k]));
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                pr[k] = ar[k];
                pi[k] = ai[k];
            }
            __syncwarp();
            ok = diag16(Sr, Si, t0, inv_s, thr_s) && ok;
        } else {
            const int nct = (rest + 31) / 32, units = (rest / W) * nct;
            const int rg = lane >> 3, cg = (lane & 7) * 4;
            for (int u = warp - 1; u < units; u += DT / 32 - 1) {
                const int ri = u / nct, col = (u % nct) * 32 + cg;
                if (col >= rest || (ri == 0 && col < W)) continue;  // past the block, or warp 0's tile
                const float* lr0 = Sr + (t0 + ri * W + rg) * PITCH + c0;
                const float* li0 = Si + (t0 + ri * W + rg) * PITCH + c0;
                const float* ur0 = Sr + c0 * PITCH + t0 + col;
                const float* ui0 = Si + c0 * PITCH + t0 + col;
                float* cr0 = Sr + (t0 + ri * W + rg) * PITCH + t0 + col;
                float* ci0 = Si + (t0 + ri * W + rg) * PITCH + t0 + col;
                float4 cr[4], ci[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    cr[a] = *reinterpret_cast<const float4*>(cr0 + 4 * a * PITCH);
                    ci[a] = *reinterpret_cast<const float4*>(ci0 + 4 * a * PITCH);
                }
#pragma unroll 1
                for (int k4 = 0; k4 < W; k4 += 4) {
                    float lr[4][4], li[4][4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const float4 x = *reinterpret_cast<const float4*>(lr0 + 4 * a * PITCH + k4);
                        const float4 y = *reinterpret_cast<const float4*>(li0 + 4 * a * PITCH + k4);
                        lr[a][0] = x.x, lr[a][1] = x.y, lr[a][2] = x.z, lr[a][3] = x.w;
                        li[a][0] = y.x, li[a][1] = y.y, li[a][2] = y.z, li[a][3] = y.w;
                    }
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) {
                        const float4 ur = *reinterpret_cast<const float4*>(ur0 + (k4 + kk) * PITCH);
                        const float4 ui = *reinterpret_cast<const float4*>(ui0 + (k4 + kk) * PITCH);
#pragma unroll
                        for (int a = 0; a < 4; ++a) {
                            const float x = lr[a][kk], y = li[a][kk];
                            cr[a].x = fmaf(-x, ur.x, fmaf(y, ui.x, cr[a].x));
                            cr[a].y = fmaf(-x, ur.y, fmaf(y, ui.y, cr[a].y));
                            cr[a].z = fmaf(-x, ur.z, fmaf(y, ui.z, cr[a].z));
                            cr[a].w = fmaf(-x, ur.w, fmaf(y, ui.w, cr[a].w));
                            ci[a].x = fmaf(-x, ui.x, fmaf(-y, ur.x, ci[a].x));
                            ci[a].y = fmaf(-x, ui.y, fmaf(-y, ur.y, ci[a].y));
                            ci[a].z = fmaf(-x, ui.z, fmaf(-y, ur.z, ci[a].z));
                            ci[a].w = fmaf(-x, ui.w, fmaf(-y, ur.w, ci[a].w));
                        }
                    }
                }
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                    *reinterpret_cast<float4*>(cr0 + 4 * a * PITCH) = cr[a];
                    *reinterpret_cast<float4*>(ci0 + 4 * a * PITCH) = ci[a];
                }
            }
        }
        __syncthreads();
    }
    if (!ok) bad = 1;
    __syncthreads();
    if (bad) {
        if (tid == 0) *reinterpret_cast<volatile int*>(fail) = 2 * (J + 1);
        return;
    }
    FdT t(T);
    for (int e = tid; e < B * (B / 4); e += DT) {  // U's rows
        const int p = e / (B / 4), k = 4 * (e % (B / 4));
        float4 x = *reinterpret_cast<const float4*>(Sr + p * PITCH + k);
        float4 y = *reinterpret_cast<const float4*>(Si + p * PITCH + k);
        if (k <= p) x.x = y.x = 0.f;
        if (k + 1 <= p) x.y = y.y = 0.f;
        if (k + 2 <= p) x.z = y.z = 0.f;
        if (k + 3 <= p) x.w = y.w = 0.f;
        *reinterpret_cast<float4*>(t.Ur + p * PITCH + k) = x;
        *reinterpret_cast<float4*>(t.Ui + p * PITCH + k) = y;
    }
    {  // L^T's rows: 8 columns p x 4 rows k of L per warp access (all banks)
        const int ks = lane & 3, ps = lane >> 2;
        for (int q = warp; q < (B / 8) * (B / 4); q += DT / 32) {
            const int p = 8 * (q / (B / 4)) + ps, k = 4 * (q % (B / 4)) + ks;
            t.Lr[p * PITCH + k] = k > p ? Sr[k * PITCH + p] : 0.f;
            t.Li[p * PITCH + k] = k > p ? Si[k * PITCH + p] : 0.f;
        }
    }
    if (tid < B) {
        t.inv[tid] = inv_s[tid];
        t.piv[tid] = make_float2(Sr[tid * PITCH + tid], Si[tid * PITCH + tid]);
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// L21 = A21 U11^{-1} (rows) and U12 = L11^{-1} A12 (columns): both are x_k = (a_k - sum_{p<k} x_p T[p][k]) s_k
// with T = U, s_k = 1/u_kk for a row and T = L^T, s_k = 1 for a column.  A CTA takes R rows or columns
// with Q = 256 / R threads each; a thread keeps 32 / Q entries of the current chunk of 32 in registers:
// the chunk first takes the products with all earlier entries, then its own entries one after
// another, each broadcast from its owner by shuffles.  FP32 rate and the shuffle chain share the time;
// R = 32 halves both per CTA while the CTAs (one per SM: T takes 135 KB) still fit one wave.
// The last CTA writes the diagonal block's factors to the matrix.  Every CTA saves what it overwrites.
template <int R>
__global__ void __launch_bounds__(256, 1) lu_trsm_kernel(C32 F, int J, int db, int mm, const float* __restrict__ T,
                                                         float* __restrict__ bk, long ldb, float* __restrict__ Lpr,
                                                         float* __restrict__ Lpi, float* __restrict__ Upr,
                                                         float* __restrict__ Upi, long ldk, int* fail) {
    constexpr int Q = 256 / R, CPT = 32 / Q, RW = R / 8, XP = R + 1;
    extern __shared__ __align__(16) float sm[];
    float* Tr = sm;
    float* Ti = Tr + B * PITCH;
    float* Xr = Ti + B * PITCH;  // [k][row]
    float* Xi = Xr + B * XP;
    __shared__ float2 inv_s[B];
    __shared__ float thr_s[B];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const int f = *reinterpret_cast<volatile int*>(fail);
        if (f != 0 && f != 2 * (J + 1) + 1) return;  // (a sibling's check may fail meanwhile: go on)
    }
    const FdT t(const_cast<float*>(T));
    const FdBackup b(bk, ldb);
    const int nr = (mm + R - 1) / R;
    if ((int)blockIdx.x == 2 * nr) {  // the diagonal block
        for (int e = tid; e < B * B; e += 256) {
            const int i = e % B, j = e / B;
            if (i >= db || j >= db) continue;
            const long o = (long)(J + i) + (long)(J + j) * F.ld;
            b.Dr[e] = F.re[o];
            b.Di[e] = F.im[o];
            const float2 p = t.piv[i];
            F.re[o] = i == j ? p.x : (i < j ? t.Ur[i * PITCH + j] : t.Lr[j * PITCH + i]);
            F.im[o] = i == j ? p.y : (i < j ? t.Ui[i * PITCH + j] : t.Li[j * PITCH + i]);
        }
        return;
    }
    const bool rows = (int)blockIdx.x < nr;
    const int x0 = ((int)blockIdx.x - (rows ? 0 : nr)) * R;  // first row or column of this CTA, from J + 128
    {
        const float* sr = rows ? t.Ur : t.Lr;
        const float* si = rows ? t.Ui : t.Li;
        for (int e = tid; e < B * PITCH / 4; e += 256) {
            cp_async16(Tr + 4 * e, sr + 4 * e);
            cp_async16(Ti + 4 * e, si + 4 * e);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    if (tid < B) {
        const float2 p = t.piv[tid];
        inv_s[tid] = rows ? t.inv[tid] : make_float2(1.f, 0.f);
        thr_s[tid] = cnorm1(p);
    }
    if (rows) {
        const int r = tid % R;
#pragma unroll 8
        for (int i = 0; i < B * R / 256; ++i) {
            const int k = tid / R + Q * i;
            float vr = 0.f, vi = 0.f;
            if (x0 + r < mm) {
                const long o = (long)(J + B + x0 + r) + (long)(J + k) * F.ld;
                vr = F.re[o];
                vi = F.im[o];
                b.Lr[x0 + r + (long)k * ldb] = vr;
                b.Li[x0 + r + (long)k * ldb] = vi;
            }
            Xr[k * XP + r] = vr;
            Xi[k * XP + r] = vi;
        }
    } else {
        const int k = tid % B;
#pragma unroll 8
        for (int i = 0; i < B * R / 256; ++i) {
            const int c = tid / B + 2 * i;
            float vr = 0.f, vi = 0.f;
            if (x0 + c < mm) {
                const long o = (long)(J + k) + (long)(J + B + x0 + c) * F.ld;
                vr = F.re[o];
                vi = F.im[o];
                b.Ur[k + (long)(x0 + c) * B] = vr;
                b.Ui[k + (long)(x0 + c) * B] = vi;
            }
            Xr[k * XP + c] = vr;
            Xi[k * XP + c] = vi;
        }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const int rs = lane % RW, q = lane / RW, row = warp * RW + rs;
    bool ok = true;
#pragma unroll 1
    for (int s0 = 0; s0 < B; s0 += 32) {
        const int j0 = s0 + q * CPT;  // this thread's entries j0 .. j0 + CPT - 1
        float ar[CPT], ai[CPT];
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            ar[j] = Xr[(j0 + j) * XP + row];
            ai[j] = Xi[(j0 + j) * XP + row];
        }
#pragma unroll 4
        for (int p = 0; p < s0; ++p) {
            const float xr = Xr[p * XP + row], xi = Xi[p * XP + row];
            const float4* tr = reinterpret_cast<const float4*>(Tr + p * PITCH + j0);
            const float4* ti = reinterpret_cast<const float4*>(Ti + p * PITCH + j0);
#pragma unroll
            for (int j = 0; j < CPT; j += 4) {
                const float4 u = tr[j / 4], v = ti[j / 4];
                ar[j] = fmaf(-xr, u.x, fmaf(xi, v.x, ar[j]));
                ar[j + 1] = fmaf(-xr, u.y, fmaf(xi, v.y, ar[j + 1]));
                ar[j + 2] = fmaf(-xr, u.z, fmaf(xi, v.z, ar[j + 2]));
                ar[j + 3] = fmaf(-xr, u.w, fmaf(xi, v.w, ar[j + 3]));
                ai[j] = fmaf(-xr, v.x, fmaf(-xi, u.x, ai[j]));
                ai[j + 1] = fmaf(-xr, v.y, fmaf(-xi, u.y, ai[j + 1]));
                ai[j + 2] = fmaf(-xr, v.z, fmaf(-xi, u.z, ai[j + 2]));
                ai[j + 3] = fmaf(-xr, v.w, fmaf(-xi, u.w, ai[j + 3]));
            }
        }
#pragma unroll
        for (int g = 0; g < Q; ++g) {
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const int k = s0 + g * CPT + c;
                // the owner scales its entry (a row's entry is the pivot search's candidate first)
                float2 x = make_float2(ar[c], ai[c]);
                if (rows) {
                    if (q == g) ok = ok && cnorm1(x) <= thr_s[k];
                    x = cmul(x, inv_s[k]);
                }
                const float xr = __shfl_sync(0xffffffffu, x.x, g * RW + rs);
                const float xi = __shfl_sync(0xffffffffu, x.y, g * RW + rs);
                // T is zero at and left of the diagonal, so entries up to k stay
                const float4* tr = reinterpret_cast<const float4*>(Tr + k * PITCH + j0);
                const float4* ti = reinterpret_cast<const float4*>(Ti + k * PITCH + j0);
#pragma unroll
                for (int j = 0; j < CPT; j += 4) {
                    const float4 u = tr[j / 4], v = ti[j / 4];
                    ar[j] = fmaf(-xr, u.x, fmaf(xi, v.x, ar[j]));
                    ar[j + 1] = fmaf(-xr, u.y, fmaf(xi, v.y, ar[j + 1]));
                    ar[j + 2] = fmaf(-xr, u.z, fmaf(xi, v.z, ar[j + 2]));
                    ar[j + 3] = fmaf(-xr, u.w, fmaf(xi, v.w, ar[j + 3]));
                    ai[j] = fmaf(-xr, v.x, fmaf(-xi, u.x, ai[j]));
                    ai[j + 1] = fmaf(-xr, v.y, fmaf(-xi, u.y, ai[j + 1]));
                    ai[j + 2] = fmaf(-xr, v.z, fmaf(-xi, u.z, ai[j + 2]));
                    ai[j + 3] = fmaf(-xr, v.w, fmaf(-xi, u.w, ai[j + 3]));
                }
                if (q == g) {
                    ar[c] = x.x;
                    ai[c] = x.y;
                }
            }
        }
#pragma unroll
        for (int j = 0; j < CPT; ++j) {
            Xr[(j0 + j) * XP + row] = ar[j];
            Xi[(j0 + j) * XP + row] = ai[j];
        }
        __syncwarp();  // a row's threads are lanes of one warp
    }
    if (!ok) atomicCAS(fail, 0, 2 * (J + 1) + 1);
    __syncthreads();
    if (rows) {
        const int r = tid % R;
        if (x0 + r < mm)
            for (int k = tid / R; k < B; k += Q) {
                const long o = (long)(J + B + x0 + r) + (long)(J + k) * F.ld;
                F.re[o] = Xr[k * XP + r];
                F.im[o] = Xi[k * XP + r];
            }
    } else {
        const int k = tid % B;
        for (int c = tid / B; c < R && x0 + c < mm; c += 2) {
            const long o = (long)(J + k) + (long)(J + B + x0 + c) * F.ld;
            F.re[o] = Xr[k * XP + c];
            F.im[o] = Xi[k * XP + c];
        }
    }
    // K-major packs, segments [hi | hi | lo] of L21 rows and [hi | lo | hi] of U12 columns
    {
        float* Pr = rows ? Lpr : Upr;
        float* Pi = rows ? Lpi : Upi;
        const int o1 = rows ? B : 2 * B, o2 = rows ? 2 * B : B;  // second hi, lo
        const int k = tid % B;
        for (int r = tid / B; r < R && x0 + r < mm; r += 2) {
            const float vr = Xr[k * XP + r], vi = Xi[k * XP + r];
            const float hr = tf32_rna(vr), hi = tf32_rna(vi);
            float* pr = Pr + (long)(x0 + r) * ldk + k;
            float* pi = Pi + (long)(x0 + r) * ldk + k;
            pr[0] = hr;
            pr[o1] = hr;
            pr[o2] = vr - hr;
            pi[0] = hi;
            pi[o1] = hi;
            pi[o2] = vi - hi;
        }
    }
}

// the entries lu_trsm_kernel overwrote, back into the matrix
__global__ void lu_restore_kernel(C32 F, int J, int db, int mm, float* __restrict__ bk, long ldb) {
    const FdBackup b(bk, ldb);
    const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long nl = (long)mm * B;
    if (e < nl) {
        const long r = e % mm, k = e / mm;
        const long o = (J + B + r) + (J + k) * F.ld;
        F.re[o] = b.Lr[r + k * ldb];
        F.im[o] = b.Li[r + k * ldb];
    } else if (e < 2 * nl) {
        const long k = (e - nl) % B, c = (e - nl) / B;
        const long o = (J + k) + (J + B + c) * F.ld;
        F.re[o] = b.Ur[k + c * B];
        F.im[o] = b.Ui[k + c * B];
    } else if (e - 2 * nl < B * B) {
        const int i = (int)((e - 2 * nl) % B), j = (int)((e - 2 * nl) / B);
        if (i < db && j < db) {
            const long o = (long)(J + i) + (long)(J + j) * F.ld;
            F.re[o] = b.Dr[i + j * B];
            F.im[o] = b.Di[i + j * B];
        }
    }
}

template <int R>
cudaError_t launch_trsm_t(cudaStream_t s, C32 F, int J, int db, int mm, float* T, float* bk, long ldb, float* const* P,
                          long ldk, int* fail) {
    constexpr int smem = (2 * B * PITCH + 2 * B * (R + 1)) * (int)sizeof(float);
    static DeviceFlags attr;
    if (attr.pending()) {
        cudaError_t e = cudaFuncSetAttribute(lu_trsm_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr.done();
    }
    lu_trsm_kernel<R><<<2 * ceil_div(mm, R) + 1, 256, smem, s>>>(F, J, db, mm, T, bk, ldb, P[0], P[1], P[2], P[3], ldk,
                                                                 fail);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_lu_diag(cudaStream_t s, C32 F, int J, int db, float* work, int* fail) {
    constexpr int smem = 2 * B * PITCH * (int)sizeof(float);
    static DeviceFlags attr;
    if (attr.pending()) {
        cudaError_t e = cudaFuncSetAttribute(lu_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr.done();
    }
    lu_diag_kernel<<<1, DT, smem, s>>>(F, J, db, work, fail);
    return cudaGetLastError();
}

cudaError_t launch_lu_trsm(cudaStream_t s, C32 F, int J, int db, int mm, float* work, long n, float* const* packs,
                           long ldk, int num_sms, int* fail) {
    if (mm > 0 && (db != B || ldk < 3 * B)) return cudaErrorInvalidValue;
    if (2 * ceil_div(mm, 32) + 1 <= num_sms)
        return launch_trsm_t<32>(s, F, J, db, mm, work, work + FD_T, n, packs, ldk, fail);
    return launch_trsm_t<64>(s, F, J, db, mm, work, work + FD_T, n, packs, ldk, fail);
}

cudaError_t launch_lu_restore(cudaStream_t s, C32 F, int J, int db, int mm, float* work, long n) {
    const long t = 2L * mm * B + B * B;
    lu_restore_kernel<<<ceil_div(t, 256), 256, 0, s>>>(F, J, db, mm, work + FD_T, n);
    return cudaGetLastError();
}

}  // namespace lu_detail
