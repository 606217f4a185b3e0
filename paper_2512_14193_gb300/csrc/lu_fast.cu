// FP32 LU with the pivots kept on the diagonal while partial pivoting would keep them there.
//
// Partial pivoting (pivot = first index of max |Re| + |Im|) rarely interchanges a row of U33 or of the
// ordinary matrix: the largest candidate below the diagonal is usually 0.5-0.9 of the diagonal entry.
// The pivot search of panel_lc.cu pays a cluster-wide exchange per column (2800-4500 cycles) to find
// that out.  Here a block of 128 columns is factored without a search, every candidate that the
// elimination forms is compared with its pivot, and the first block where one is larger (or a pivot
// is zero or a NaN) stops the sequence: *fail = 2 (J + 1) + stage names the block, later kernels return
// at once, and the host restores that block's columns and rows and continues from it with the pivot
// search (factor_t in lu.cu).  So the pivots are those of partial pivoting up to the rounding of the magnitudes
// compared: below the diagonal block a candidate is formed again from its multiplier and pivot.
//
// Per block of FD_B = 128 columns at J:
//   lu_diag_kernel  one CTA: LU of the diagonal block (stage 0 of the check)
//   lu_trsm_kernel  all SMs: L21 = A21 U11^{-1} by rows (stage 1 of the check) and U12 = L11^{-1} A12
//                   by columns, written to the matrix and packed for the tensor cores; the original
//                   entries are kept in a backup until the next block
//   gemm_tc         A22 -= L21 U12, split FP16 operands (gemm_tc.cu): the next diagonal block's tile first, so that the next
//                   lu_diag_kernel runs beside the rest (look-ahead on two streams)
#include "lu_internal.cuh"

namespace lu_detail {
namespace {

constexpr int B = FD_B, PITCH = FD_PITCH, W = FD_W;  // block, row pitch of the shared block, sub-step
constexpr int DT = 512;                            // threads of lu_diag_kernel

// 1 / a for a != 0, as cinv_fast without its scaling where |a|^2 neither over- nor underflows
__device__ __forceinline__ float2 cinv_near(float2 a) {
    const float d = fmaf(a.x, a.x, a.y * a.y);
    if (!(d > 1e-30f && d < 1e30f)) return cinv_fast(a);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
    r = r * fmaf(-d, r, 2.f);
    return make_float2(a.x * r, -a.y * r);
}
__device__ __forceinline__ float2 shfl2(float2 v, int l) {
    return make_float2(__shfl_sync(0xffffffffu, v.x, l), __shfl_sync(0xffffffffu, v.y, l));
}
// a - b c
__device__ __forceinline__ float2 csubmul(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(-b.x, c.x, fmaf(b.y, c.y, a.x)), fmaf(-b.x, c.y, fmaf(-b.y, c.x, a.y)));
}

// Eliminates the 16 x 16 diagonal block at (c0, c0) of the shared block without interchanges: one
// warp, lane = row (lanes 16-31 repeat lanes 0-15), the row in registers.  Returns false if a
// candidate exceeds its pivot.  The chain per column is one reciprocal: every lane forms the next
// pivot itself from entries shuffled before the reciprocal is known (333 -> 110 cycles per column
// against broadcasting the updated pivot).  Sixteen columns keep the unrolled code small.
__device__ __forceinline__ bool diag16(float* Sr, float* Si, int c0, float2* inv_s, float2* piv_s) {
    const int lane = threadIdx.x & 31, r = lane & 15;
    float2 x[W];
    float* pr = Sr + (c0 + r) * PITCH + c0;
    float* pi = Si + (c0 + r) * PITCH + c0;
#pragma unroll
    for (int k = 0; k < W; k += 4) {
        const float4 u = *reinterpret_cast<const float4*>(pr + k), v = *reinterpret_cast<const float4*>(pi + k);
        x[k] = make_float2(u.x, v.x);
        x[k + 1] = make_float2(u.y, v.y);
        x[k + 2] = make_float2(u.z, v.z);
        x[k + 3] = make_float2(u.w, v.w);
    }
    bool ok = true;
    float2 p = shfl2(x[0], 0);
    float2 iv = cinv_near(p);
#pragma unroll
    for (int c = 0; c < W; ++c) {
        const float un = cnorm1(p);
        const bool below = r > c;
        ok = ok && un > 0.f && (!below || cnorm1(x[c]) <= un);
        if (lane == c) {
            inv_s[c0 + c] = iv;
            piv_s[c0 + c] = p;
        }
        if (c + 1 < W) {
            const float2 ul = shfl2(x[c + 1], c), a0 = shfl2(x[c], c + 1), a1 = shfl2(x[c + 1], c + 1);
            p = csubmul(a1, cmul(a0, iv), ul);  // the next pivot
            const float2 l = below ? cmul(x[c], iv) : make_float2(0.f, 0.f);
            iv = cinv_near(p);
            x[c + 1] = csubmul(x[c + 1], l, ul);
#pragma unroll
            for (int k = c + 2; k < W; ++k) x[k] = csubmul(x[k], l, shfl2(x[k], c));
            if (below) x[c] = l;
        }
    }
    if (lane < W) {
#pragma unroll
        for (int k = 0; k < W; k += 4) {
            *reinterpret_cast<float4*>(pr + k) = make_float4(x[k].x, x[k + 1].x, x[k + 2].x, x[k + 3].x);
            *reinterpret_cast<float4*>(pi + k) = make_float4(x[k].y, x[k + 1].y, x[k + 2].y, x[k + 3].y);
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
// lu_trsm_kernel, which also writes them to the matrix: U and L^T as packed rows of 16-row blocks with
// the 16 x 16 diagonal blocks inverted, and both as they are (see FdT).
__global__ void __launch_bounds__(DT, 1) lu_diag_kernel(C32 F, int J, int db, float* __restrict__ T, int* fail) {
    extern __shared__ __align__(16) float sm[];
    __shared__ float2 inv_s[B], piv_s[B];
    __shared__ int bad;
    float* Sr = sm;
    float* Si = sm + B * PITCH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (*reinterpret_cast<volatile int*>(fail) != 0) return;
    if (tid == 0) bad = 0;
    const int be = (db + W - 1) & ~(W - 1);  // past it the block is the identity's, which needs no elimination
    if (tid >= be && tid < B) inv_s[tid] = piv_s[tid] = make_float2(1.f, 0.f);
    {
        // lane = 8 rows x 4 columns: 32-byte sectors of the matrix, all 32 shared banks
        const int r = warp * 8 + (lane & 7), cs = lane >> 3;
#pragma unroll 16
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
    if (warp == 0) ok = diag16(Sr, Si, 0, inv_s, piv_s);
    __syncthreads();
#pragma unroll 1
    for (int c0 = 0; c0 + W < be; c0 += W) {
        const int rest = be - c0 - W;
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
                ok = ok && cnorm1(make_float2(ar[c], ai[c])) <= cnorm1(piv_s[c0 + c]);
                const float2 l = cmul(make_float2(ar[c], ai[c]), inv_s[c0 + c]);
                ar[c] = l.x;
                ai[c] = l.y;
#pragma unroll
                for (int k4 = (c + 1) & ~3; k4 < W; k4 += 4) {
                    const float4 u = *reinterpret_cast<const float4*>(Sr + (c0 + c) * PITCH + c0 + k4);
                    const float4 v = *reinterpret_cast<const float4*>(Si + (c0 + c) * PITCH + c0 + k4);
                    const float ur[4] = {u.x, u.y, u.z, u.w}, ui[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (k4 + k > c) {
                            ar[k4 + k] = fmaf(-l.x, ur[k], fmaf(l.y, ui[k], ar[k4 + k]));
                            ai[k4 + k] = fmaf(-l.x, ui[k], fmaf(-l.y, ur[k], ai[k4 + k]));
                        }
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
            for (int k = 1; k < W; ++k) {  // x_k -= sum_{c<k} L[k][c] x_c
#pragma unroll
                for (int c4 = 0; c4 < k; c4 += 4) {
                    const float4 u = *reinterpret_cast<const float4*>(Sr + (c0 + k) * PITCH + c0 + c4);
                    const float4 v = *reinterpret_cast<const float4*>(Si + (c0 + k) * PITCH + c0 + c4);
                    const float lr[4] = {u.x, u.y, u.z, u.w}, li[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        if (c4 + c < k) {
                            xr[k] = fmaf(-lr[c], xr[c4 + c], fmaf(li[c], xi[c4 + c], xr[k]));
                            xi[k] = fmaf(-lr[c], xi[c4 + c], fmaf(-li[c], xr[c4 + c], xi[k]));
                        }
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
            ok = diag16(Sr, Si, t0, inv_s, piv_s) && ok;
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
    {
        // inverses of the sixteen 16 x 16 diagonal blocks of U (warps 0-7) and L^T (8-15), a column per
        // lane: x_i = s_i (delta_ij - sum_{k>i} T[i][k] x_k)
        const int b = warp & 7, d0 = W * b, j = lane & 15;
        const bool up = warp < 8;
        float xr[W], xi[W];
#pragma unroll
        for (int i = W - 1; i >= 0; --i) {
            float sr = i == j ? 1.f : 0.f, si = 0.f;
#pragma unroll
            for (int k = i + 1; k < W; ++k) {
                const int o = up ? (d0 + i) * PITCH + d0 + k : (d0 + k) * PITCH + d0 + i;
                const float tr = Sr[o], ti = Si[o];
                sr = fmaf(-tr, xr[k], fmaf(ti, xi[k], sr));
                si = fmaf(-tr, xi[k], fmaf(-ti, xr[k], si));
            }
            const float2 s = up ? inv_s[d0 + i] : make_float2(1.f, 0.f);
            xr[i] = sr * s.x - si * s.y;
            xi[i] = sr * s.y + si * s.x;
        }
        if (lane < W) {
            float* gr = (up ? t.Ur : t.Lr) + fd_row(d0);
            float* gi = (up ? t.Ui : t.Li) + fd_row(d0);
            const int w = B - d0;
#pragma unroll
            for (int i = 0; i < W; ++i) {
                gr[i * w + j] = xr[i];
                gi[i * w + j] = xi[i];
            }
        }
    }
    for (int e = tid; e < B * (B / 4); e += DT) {  // the factors as they are, and U right of the blocks
        const int p = e / (B / 4), k = 4 * (e % (B / 4));
        const float4 x = *reinterpret_cast<const float4*>(Sr + p * PITCH + k);
        const float4 y = *reinterpret_cast<const float4*>(Si + p * PITCH + k);
        *reinterpret_cast<float4*>(t.Fr + p * B + k) = x;
        *reinterpret_cast<float4*>(t.Fi + p * B + k) = y;
        if (k / W > p / W) {
            const int o = fd_row(p) + k - (p & ~(W - 1));
            *reinterpret_cast<float4*>(t.Ur + o) = x;
            *reinterpret_cast<float4*>(t.Ui + o) = y;
        }
    }
    // L^T below the blocks: a lane reads 4 columns p of row k, a warp writes 32 k of each p
    for (int q = warp; q < (B / 4) * (B / 32); q += DT / 32) {
        const int p = 4 * (q % (B / 4)), k = 32 * (q / (B / 4)) + lane;
        if (k / W <= p / W) continue;
        const float4 x = *reinterpret_cast<const float4*>(Sr + k * PITCH + p);
        const float4 y = *reinterpret_cast<const float4*>(Si + k * PITCH + p);
        const int o = fd_row(p) + k - (p & ~(W - 1)), w = B - (p & ~(W - 1));
        t.Lr[o] = x.x, t.Lr[o + w] = x.y, t.Lr[o + 2 * w] = x.z, t.Lr[o + 3 * w] = x.w;
        t.Li[o] = y.x, t.Li[o + w] = y.y, t.Li[o + 2 * w] = y.z, t.Li[o + 3 * w] = y.w;
    }
    if (tid < B) t.piv[tid] = piv_s[tid];
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// L21 = A21 U11^{-1} (rows) and U12 = L11^{-1} A12 (columns): both are x T = a with T = U for a row and
// T = L^T for a column, solved in chunks of 16 entries: y = a_b - sum_{b'<b} x_b' T[b'][b], then
// x_b = y T[b][b]^{-1} with the inverted block.  A CTA takes R = 32 rows or columns, four threads each with
// 4 of a chunk's 16 entries in registers; T (74 KB packed) and the 32 x 128 entries are in shared memory, so
// two CTAs share an SM and one wave covers 4800 rows and columns.  The FP32 rate bounds it (9.2k cycles
// of multiply-adds per CTA).  The pivot search's candidates l_ik u_kk are compared with their pivots.
// The last eight CTAs write the diagonal block's factors to the matrix.  Every CTA saves what it
// overwrites.
constexpr int R = 32, RT = 4 * R, XP = R + 1;
__global__ void __launch_bounds__(RT, 2) lu_trsm_kernel(C32 F, int J, int db, int mm, const float* __restrict__ T,
                                                        float* __restrict__ bk, long ldb, TcPacks packs, int* fail) {
    extern __shared__ __align__(16) float sm[];
    float* Tr = sm;
    float* Ti = Tr + FD_PACK;
    float* Xr = Ti + FD_PACK;  // [k][row]
    float* Xi = Xr + B * XP;
    __shared__ float2 piv_s[B];
    __shared__ float w_s[B];  // inner scale of the packs
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    {
        const int f = *reinterpret_cast<volatile int*>(fail);
        if (f != 0 && f != 2 * (J + 1) + 1) return;  // (a sibling's check may fail meanwhile: go on)
    }
    const FdT t(const_cast<float*>(T));
    const FdBackup b(bk, ldb);
    const int nr = (mm + R - 1) / R;
    if ((int)blockIdx.x >= 2 * nr) {  // 16 columns of the diagonal block, a row of 4 columns at a time
        const int i = tid, j0 = W * ((int)blockIdx.x - 2 * nr);
        float4 x[W / 4], y[W / 4];
#pragma unroll
        for (int q = 0; q < W / 4; ++q) {
            x[q] = *reinterpret_cast<const float4*>(t.Fr + i * B + j0 + 4 * q);
            y[q] = *reinterpret_cast<const float4*>(t.Fi + i * B + j0 + 4 * q);
        }
        if (i < db) {
            float orr[W], oi[W];
#pragma unroll
            for (int j = 0; j < W; ++j)
                if (j0 + j < db) {
                    const long o = (long)(J + i) + (long)(J + j0 + j) * F.ld;
                    orr[j] = F.re[o];
                    oi[j] = F.im[o];
                }
#pragma unroll
            for (int j = 0; j < W; ++j)
                if (j0 + j < db) {
                    const long o = (long)(J + i) + (long)(J + j0 + j) * F.ld;
                    b.Dr[i + (j0 + j) * B] = orr[j];
                    b.Di[i + (j0 + j) * B] = oi[j];
                    const float4 u = x[j / 4], v = y[j / 4];
                    F.re[o] = j % 4 == 0 ? u.x : (j % 4 == 1 ? u.y : (j % 4 == 2 ? u.z : u.w));
                    F.im[o] = j % 4 == 0 ? v.x : (j % 4 == 1 ? v.y : (j % 4 == 2 ? v.z : v.w));
                }
        }
        return;
    }
    const bool rows = (int)blockIdx.x < nr;
    const int x0 = ((int)blockIdx.x - (rows ? 0 : nr)) * R;  // first row or column of this CTA, from J + 128
    {
        const float* sr = rows ? t.Ur : t.Lr;
        const float* si = rows ? t.Ui : t.Li;
        for (int e = tid; e < FD_PACK / 4; e += RT) {
            cp_async16(Tr + 4 * e, sr + 4 * e);
            cp_async16(Ti + 4 * e, si + 4 * e);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    piv_s[tid] = t.piv[tid];
    static_assert(RT == B, "a thread per pivot, row and K index");
    if (rows) {
        const int r = lane;
#pragma unroll 16
        for (int i = 0; i < B / 4; ++i) {
            const int k = warp + 4 * i;
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
#pragma unroll 16
        for (int c = 0; c < R; ++c) {
            float vr = 0.f, vi = 0.f;
            if (x0 + c < mm) {
                const long o = (long)(J + tid) + (long)(J + B + x0 + c) * F.ld;
                vr = F.re[o];
                vi = F.im[o];
                b.Ur[tid + (long)(x0 + c) * B] = vr;
                b.Ui[tid + (long)(x0 + c) * B] = vi;
            }
            Xr[tid * XP + c] = vr;
            Xi[tid * XP + c] = vi;
        }
    }
    {
        const int d = packs.re != nullptr ? inner_exponent(packs.re[J + tid], packs.re[J]) : 0;
        w_s[tid] = tc_pow2(rows ? d : -d);
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();
    const int q = 4 * (lane & 3), row = warp * 8 + (lane >> 2);
    // a -= (or +=) the products of entries p0 .. p0 + 15 with the 16 x 4 entries of T at tr, ti (row pitch w)
    auto mac = [&](float (&ar)[4], float (&ai)[4], int p0, const float* tr, const float* ti, int w, float sign) {
#pragma unroll
        for (int p = 0; p < W; ++p) {
            const float xr = sign * Xr[(p0 + p) * XP + row], xi = sign * Xi[(p0 + p) * XP + row];
            const float4 u = *reinterpret_cast<const float4*>(tr + p * w);
            const float4 v = *reinterpret_cast<const float4*>(ti + p * w);
            ar[0] = fmaf(xr, u.x, fmaf(-xi, v.x, ar[0]));
            ar[1] = fmaf(xr, u.y, fmaf(-xi, v.y, ar[1]));
            ar[2] = fmaf(xr, u.z, fmaf(-xi, v.z, ar[2]));
            ar[3] = fmaf(xr, u.w, fmaf(-xi, v.w, ar[3]));
            ai[0] = fmaf(xr, v.x, fmaf(xi, u.x, ai[0]));
            ai[1] = fmaf(xr, v.y, fmaf(xi, u.y, ai[1]));
            ai[2] = fmaf(xr, v.z, fmaf(xi, u.z, ai[2]));
            ai[3] = fmaf(xr, v.w, fmaf(xi, u.w, ai[3]));
        }
    };
    bool ok = true;
#pragma unroll 1
    for (int j0 = 0; j0 < B; j0 += W) {
        float ar[4], ai[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            ar[j] = Xr[(j0 + q + j) * XP + row];
            ai[j] = Xi[(j0 + q + j) * XP + row];
        }
        int o = j0 + q;  // T[p0 .. p0 + 15][j0 + q ..] in the packed rows
#pragma unroll 1
        for (int p0 = 0; p0 < j0; p0 += W) {
            mac(ar, ai, p0, Tr + o, Ti + o, B - p0, -1.f);
            o += W * (B - p0) - W;
        }
        __syncwarp();  // the chunk's entries have been read
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            Xr[(j0 + q + j) * XP + row] = ar[j];
            Xi[(j0 + q + j) * XP + row] = ai[j];
        }
        __syncwarp();
        float yr[4] = {0.f, 0.f, 0.f, 0.f}, yi[4] = {0.f, 0.f, 0.f, 0.f};
        mac(yr, yi, j0, Tr + o, Ti + o, B - j0, 1.f);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (rows) {
                const float2 u = piv_s[j0 + q + j];
                ok = ok && cnorm1(cmul(make_float2(yr[j], yi[j]), u)) <= cnorm1(u);
            }
            Xr[(j0 + q + j) * XP + row] = yr[j];
            Xi[(j0 + q + j) * XP + row] = yi[j];
        }
        __syncwarp();
    }
    if (!ok) atomicCAS(fail, 0, 2 * (J + 1) + 1);
    __syncthreads();
    if (rows) {
        if (x0 + lane < mm)
#pragma unroll 8
            for (int i = 0; i < B / 4; ++i) {
                const int k = warp + 4 * i;
                const long o = (long)(J + B + x0 + lane) + (long)(J + k) * F.ld;
                F.re[o] = Xr[k * XP + lane];
                F.im[o] = Xi[k * XP + lane];
            }
    } else {
#pragma unroll 8
        for (int c = 0; c < R; ++c)
            if (x0 + c < mm) {
                const long o = (long)(J + tid) + (long)(J + B + x0 + c) * F.ld;
                F.re[o] = Xr[tid * XP + c];
                F.im[o] = Xi[tid * XP + c];
            }
    }
    // packs of the L21 rows and U12 columns and their exponents (the rows' own: with beta far from i / k or a low
    // frequency the ordinary system's lower rows of L21 are small, and a fixed scale would lose them)
    __shared__ float mx_s[RT / 32][R];
    {
        float mx = 0.f;  // of a quarter of row or column `lane`
#pragma unroll 8
        for (int k = warp; k < B; k += RT / 32)
            mx = fmaxf(mx, w_s[k] * fmaxf(fabsf(Xr[k * XP + lane]), fabsf(Xi[k * XP + lane])));
        mx_s[warp][lane] = mx;
        __syncthreads();
    }
    const float w = w_s[tid];
    int* const pe = rows ? packs.Le : packs.Ue;
    __half* Pr = (rows ? packs.Lr : packs.Ur) + tc_pos(tid);
    __half* Pi = (rows ? packs.Li : packs.Ui) + tc_pos(tid);
#pragma unroll 4
    for (int r = 0; r < R; ++r)
        if (x0 + r < mm) {
            const TcRowScale sc(fmaxf(fmaxf(mx_s[0][r], mx_s[1][r]), fmaxf(mx_s[2][r], mx_s[3][r])));
            if (tid == 0) pe[x0 + r] = sc.ex - 15;
            __half* pr = Pr + (long)(x0 + r) * packs.ldk;
            __half* pi = Pi + (long)(x0 + r) * packs.ldk;
            tc_split(sc(w * Xr[tid * XP + r]), pr[0], pr[32]);
            tc_split(sc(w * Xi[tid * XP + r]), pi[0], pi[32]);
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

cudaError_t launch_lu_trsm(cudaStream_t s, C32 F, int J, int db, int mm, float* work, long n, TcPacks packs,
                           int* fail) {
    if (mm > 0 && (db != B || packs.ldk < tc_ldk(B))) return cudaErrorInvalidValue;
    constexpr int smem = (2 * FD_PACK + 2 * B * XP) * (int)sizeof(float);
    static DeviceFlags attr;
    if (attr.pending()) {
        cudaError_t e = cudaFuncSetAttribute(lu_trsm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        attr.done();
    }
    lu_trsm_kernel<<<2 * ceil_div(mm, R) + ceil_div(db, W), RT, smem, s>>>(
        F, J, db, mm, work, work + FD_T, n, packs, fail);
    return cudaGetLastError();
}

cudaError_t launch_lu_restore(cudaStream_t s, C32 F, int J, int db, int mm, float* work, long n) {
    const long t = 2L * mm * B + B * B;
    lu_restore_kernel<<<ceil_div(t, 256), 256, 0, s>>>(F, J, db, mm, work + FD_T, n);
    return cudaGetLastError();
}

}  // namespace lu_detail
