// Dense complex LU with partial pivoting on the GPU (the N x N Schur complement U33 of
// Theorem thm:LU, or the 2N x 2N ordinary matrix of Eq. dis_BM), and the triangular solves.
//
// By default blocks of columns are factored without a pivot search while partial pivoting keeps its pivots on the
// diagonal (lu_fast.cu, lu_fast_z.cu: every candidate is checked); from the first block that needs an interchange
// on, and where a block size or a panel setting asks for it, the search below factors.  Right-looking, with two
// block sizes:
//   for each big panel of NB columns (C32: 256, Z64: 64):
//     for each sub-panel of nbp columns:
//        panel kernel      : unblocked LU with partial pivoting of rows [j, n) x nbp columns on a
//                            cluster of up to 16 CTAs.  C32 panels of at most 4096 rows use the
//                            lane-per-column kernel (panel_c32.cu: nbp = 32, lane k of every warp
//                            holds column k of 4-16 rows, about 64-256 rows per CTA); taller C32
//                            panels and all Z64 panels use the register-row kernel
//                            (lu_internal.cuh: one to four rows per thread, nbp = 32/16/8 for C32,
//                            16/8/4 for Z64).  Each column's pivot candidates (value, index, whole
//                            row) go to every CTA through distributed shared memory; CTA 0 also
//                            builds the row-interchange maps.
//        swap_trsm_kernel  : row interchanges + unit-lower solve for the rest of the big panel
//        gemm (SIMT)       : rank-nbp update of the rest of the big panel
//     swap_trsm_kernel     : interchanges for all other columns, U12 = L11^{-1} A12 (and its
//                            K-major pack for the tensor cores)
//     trailing update      : A22 -= L21 U12  (tensor cores, split FP16 (gemm_tc.cu) for C32, SIMT for Z64)
// Pivot = first row index of max |Re| + |Im| (the LAPACK izamax rule).  An exactly zero pivot
// records the 1-based column in *info and skips the scaling, as LAPACK getrf does.
//
// Solves (getrs): Y = P B, then block forward substitution with the unit L and block back
// substitution with U, each triangle one persistent launch whose items wait for the block rows they need
// (trsv_flow_kernel, trsv_flow_z64_kernel).  The diagonal blocks (64 x 64, FP64: 16 x 16) are inverted once after
// the factorisation so that every step is a small matrix product.  For C32 the off-diagonal tiles of each
// block column are then multiplied by that column's inverted diagonal block (the "G form"), so
// that a step is one product with no dependence on the inverse:
//   forward:  Y[below b] -= (L[below b, b] L_bb^{-1}) Y_b,  Z_b = L_bb^{-1} Y_b
//   backward: Z[above b] -= (U[above b, b] U_bb^{-1}) Z_b,  X_b = U_bb^{-1} Z_b
#include "lu_internal.cuh"

#include <climits>
#include <map>
#include <mutex>

using namespace lu_detail;

namespace {

// Row interchanges (from a swap map) for columns in [a0, a1) u [b0, b1); for columns of the
// second range also X = L11^{-1} X on rows [t0, t0+tb) with the unit-lower L11 at (t0, t0),
// staged in shared memory: whole when it fits, else in chunks of ST_KC columns that the CTA's
// warps step through together.  Optionally writes the solved rows as a K-major tensor-core pack
// (column c -> row c - b0).  One warp per column.
// Asynchronous 4-byte global -> shared copies (cp.async, zero-filled when !full).
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool full) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(full ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Strictly lower part of columns [k0, k0 + kc) of the tb x tb block at (t0, t0) of a planar FP32
// matrix into dst (interleaved complex, leading dimension tb), by cp.async (nthreads threads).
__device__ __forceinline__ void stage_lower_async(float2* dst, const C32& A, long t0, int tb, int k0, int kc,
                                                  int nthreads) {
    const int tot = tb * kc;
    for (int e = threadIdx.x; e < tot; e += nthreads) {
        const int i = e % tb, kk = e / tb;
        const bool in = i > k0 + kk;
        const long off = in ? (t0 + i) + (t0 + k0 + kk) * A.ld : 0;
        cp_async4(&dst[e].x, A.re + off, in);
        cp_async4(&dst[e].y, A.im + off, in);
    }
}

constexpr int ST_WARPS = 16, ST_COLS = 1;
constexpr int ST_KC = 32;  // L11 columns per shared-memory chunk when L11 does not fit whole
template <class V>
__global__ void __launch_bounds__(ST_WARPS * 32) swap_trsm_kernel(V A, const SwapMap* __restrict__ map, int a0, int a1,
                                                                   int b0, int b1, int t0, int tb, __half* Upr,
                                                                   __half* Upi, long ldk, int* Upe, const int* re,
                                                                   const int* perm, int l_in_smem) {
    using CV = typename V::cv;
    using Rl = typename V::real;
    constexpr int QMAX = 8;  // rows per lane: tb <= 256
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smraw[];
    CV* Ls = reinterpret_cast<CV*>(smraw);  // tb x tb, column-major
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int na = a1 - a0, nbc = b1 - b0;
    const int ncols = na + nbc;
    const int cta_col0 = blockIdx.x * ST_WARPS * ST_COLS;
    const bool cta_has_b = (cta_col0 + ST_WARPS * ST_COLS > na) && tb > 0;
    // strictly lower part of L11 columns [k0, k0 + kc) into Ls (leading dimension tb), SB loads in
    // flight per thread at a time
    auto stage = [&](int k0, int kc) {
        constexpr int SB = 8;
        const int tot = tb * kc;
        for (int e0 = 0; e0 < tot; e0 += SB * ST_WARPS * 32) {
            CV v[SB];
#pragma unroll
            for (int m = 0; m < SB; ++m) {
                const int e = e0 + threadIdx.x + m * ST_WARPS * 32;
                const int i = e % tb, kk = e / tb;
                v[m] = (e < tot && i > k0 + kk) ? A.get((long)t0 + i, (long)t0 + k0 + kk) : czero<Rl>();
            }
#pragma unroll
            for (int m = 0; m < SB; ++m) {
                const int e = e0 + threadIdx.x + m * ST_WARPS * 32;
                if (e < tot) Ls[e] = v[m];
            }
        }
    };
    if (cta_has_b && l_in_smem == 1) {
        if constexpr (std::is_same<V, C32>::value) {
            stage_lower_async(Ls, A, t0, tb, 0, tb, ST_WARPS * 32);
            cp_async_commit();
            cp_async_wait<0>();
        } else {
            stage(0, tb);
        }
        __syncthreads();
    }
    static_assert(ST_COLS == 1, "one column per warp");
    const int cnt = map ? map->count : 0;
    const int gw = cta_col0 + warp;
    const bool valid = gw < ncols;
    const bool in_b = valid && gw >= na;
    const long col = in_b ? (long)b0 + (gw - na) : (long)a0 + gw;
    if (valid && cnt > 0) {
        CV v[MAP_MAX / 32];
#pragma unroll
        for (int q = 0; q < MAP_MAX / 32; ++q) {
            int t = lane + 32 * q;
            if (t < cnt) v[q] = A.get(map->src[t], col);
        }
        __syncwarp();
#pragma unroll
        for (int q = 0; q < MAP_MAX / 32; ++q) {
            int t = lane + 32 * q;
            if (t < cnt) A.set(map->dst[t], col, v[q]);
        }
        __syncwarp();
    }
    const bool do_trsm = in_b && tb > 0;
    CV x[QMAX];
#pragma unroll
    for (int q = 0; q < QMAX; ++q) {
        int i = lane + 32 * q;
        x[q] = (do_trsm && i < tb) ? A.get((long)t0 + i, col) : czero<Rl>();
    }
    // x -= L11 columns k in [kb, ke), all in one group of 32 (k = 32 QK + l); lk(i, k) reads
    // L(t0 + i, t0 + k) from wherever it is staged.  With the group a compile-time constant, the
    // value x_k comes straight from register x[QK] of lane l, and only rows of groups >= QK are
    // touched, without per-row predicates beyond the diagonal group.
    auto steps_q = [&](auto qc, int kb, int ke, auto lk) {
        constexpr int QK = decltype(qc)::value;
        for (int k = kb; k < ke; ++k) {
            const int l = k & 31;
            CV nx;
            nx.x = -__shfl_sync(0xffffffffu, x[QK].x, l);
            nx.y = -__shfl_sync(0xffffffffu, x[QK].y, l);
            if (lane > l && lane + 32 * QK < tb) cfma(x[QK], lk(lane + 32 * QK, k), nx);
#pragma unroll
            for (int q = QK + 1; q < QMAX; ++q) {
                if (32 * q >= tb) break;  // warp-uniform: groups past tb issue nothing
                const int i = lane + 32 * q;
                if (i < tb) cfma(x[q], lk(i, k), nx);
            }
        }
    };
    auto steps = [&](int kb, int ke, auto lk) {
        for (int g0 = kb; g0 < ke;) {
            const int g1 = min(ke, (g0 & ~31) + 32);
            switch (g0 >> 5) {
                case 0: steps_q(std::integral_constant<int, 0>{}, g0, g1, lk); break;
                case 1: steps_q(std::integral_constant<int, 1>{}, g0, g1, lk); break;
                case 2: steps_q(std::integral_constant<int, 2>{}, g0, g1, lk); break;
                case 3: steps_q(std::integral_constant<int, 3>{}, g0, g1, lk); break;
                case 4: steps_q(std::integral_constant<int, 4>{}, g0, g1, lk); break;
                case 5: steps_q(std::integral_constant<int, 5>{}, g0, g1, lk); break;
                case 6: steps_q(std::integral_constant<int, 6>{}, g0, g1, lk); break;
                default: steps_q(std::integral_constant<int, 7>{}, g0, g1, lk); break;
            }
            g0 = g1;
        }
    };
    static_assert(QMAX == 8, "one case per group of 32 rows");
    if (l_in_smem == 2) {
        // L11 larger than the shared-memory budget: stage it ST_KC columns at a time, the whole
        // CTA stepping through the chunks together (warps without a column to solve only help)
        if constexpr (!std::is_same<V, C32>::value) {  // FP64: L11 (NB <= 64) always fits whole
            if (cta_has_b)
                for (int k0 = 0; k0 < tb; k0 += ST_KC) {
                    const int kc = min(ST_KC, tb - k0);
                    __syncthreads();
                    stage(k0, kc);
                    __syncthreads();
                    if (do_trsm) steps(k0, k0 + kc, [&](int i, int kk) { return Ls[i + (kk - k0) * tb]; });
                }
        } else if (cta_has_b) {
            // two buffers of ST_KC / 2 columns: the next chunk's cp.async copies run while the
            // warps step through the current one
            constexpr int KC = ST_KC / 2;
            CV* const buf1 = Ls + tb * KC;
            stage_lower_async(Ls, A, t0, tb, 0, min(KC, tb), ST_WARPS * 32);
            cp_async_commit();
            for (int k0 = 0, c = 0; k0 < tb; k0 += KC, ++c) {
                const int kc = min(KC, tb - k0);
                if (k0 + KC < tb) {
                    stage_lower_async((c & 1) ? Ls : buf1, A, t0, tb, k0 + KC, min(KC, tb - k0 - KC), ST_WARPS * 32);
                    cp_async_commit();
                    cp_async_wait<1>();
                } else {
                    cp_async_wait<0>();
                }
                __syncthreads();  // chunk c is in shared memory for every warp
                const CV* cur = (c & 1) ? buf1 : Ls;
                if (do_trsm) steps(k0, k0 + kc, [&](int i, int kk) { return cur[i + (kk - k0) * tb]; });
                __syncthreads();  // every warp is done with chunk c before its buffer is refilled
            }
        }
    } else if (do_trsm) {
        if (l_in_smem)
            steps(0, tb, [&](int i, int kk) { return Ls[i + kk * tb]; });
        else
            steps(0, tb, [&](int i, int kk) { return A.get((long)t0 + i, (long)t0 + kk); });
    }
    if (do_trsm) {
#pragma unroll
        for (int q = 0; q < QMAX; ++q) {
            int i = lane + 32 * q;
            if (i < tb) A.set((long)t0 + i, col, x[q]);
        }
        if (Upr != nullptr) {
            // pack row col - b0 (tb is a multiple of 32: the last panel has no pack) and its exponent
            const long rowp = col - b0;
            float mx = 0.f, w[QMAX];
#pragma unroll
            for (int q = 0; q < QMAX; ++q)
                if (lane + 32 * q < tb) {
                    w[q] = re != nullptr ? tc_pow2(-inner_exponent(re[perm[t0 + lane + 32 * q]], re[perm[t0]])) : 1.f;
                    mx = fmaxf(mx, w[q] * fmaxf(fabsf((float)x[q].x), fabsf((float)x[q].y)));
                }
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            const TcRowScale sc(mx);
            if (lane == 0) Upe[rowp] = sc.ex - 15;
            __half* pr = Upr + rowp * ldk + lane;
            __half* pi = Upi + rowp * ldk + lane;
#pragma unroll
            for (int q = 0; q < QMAX; ++q)
                if (lane + 32 * q < tb) {
                    tc_split(sc(w[q] * (float)x[q].x), pr[64 * q], pr[64 * q + 32]);
                    tc_split(sc(w[q] * (float)x[q].y), pi[64 * q], pi[64 * q + 32]);
                }
        }
    }
}

// L21 pack: rows [r0, r0+m) x columns [c0, c0+kb) of A (kb a multiple of 32) -> pack rows and their exponents: the
// maxima of 32 rows, then the pack through 32 x 32 tiles (the second reads come from L2).
__global__ void pack_L_kernel(C32 A, long r0, long c0, int m, int kb, __half* Pr, __half* Pi, long ldk, int* Le,
                              const int* re, const int* perm) {
    __shared__ float2 t[32][33];
    auto w = [&](int k) { return re != nullptr ? tc_pow2(inner_exponent(re[perm[c0 + k]], re[perm[c0]])) : 1.f; };
    __shared__ float top[8][32];
    const int i0 = blockIdx.x * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;
    const bool in = i0 + tx < m;
    float mx = 0.f;
#pragma unroll 8
    for (int k = ty; k < kb; k += 8) {
        const float2 v = in ? A.get(r0 + i0 + tx, c0 + k) : make_float2(0.f, 0.f);
        mx = fmaxf(mx, w(k) * fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    top[ty][tx] = mx;
    for (int k0 = 0; k0 < kb; k0 += 32) {
        __syncthreads();  // the maxima are there; the tile before has been packed
        for (int q = ty; q < 32; q += 8) t[q][tx] = in ? A.get(r0 + i0 + tx, c0 + k0 + q) : make_float2(0.f, 0.f);
        __syncthreads();
        const float wk = w(k0 + tx);
        for (int q = ty; q < 32; q += 8) {
            const int i = i0 + q;
            if (i >= m) continue;
            float mi = 0.f;
#pragma unroll
            for (int w = 0; w < 8; ++w) mi = fmaxf(mi, top[w][q]);
            const TcRowScale sc(mi);
            if (k0 == 0 && tx == 0) Le[i] = sc.ex - 15;
            const float2 v = t[tx][q];
            __half* pr = Pr + (long)i * ldk + 2 * k0 + tx;
            __half* pi = Pi + (long)i * ldk + 2 * k0 + tx;
            tc_split(sc(wk * v.x), pr[0], pr[32]);
            tc_split(sc(wk * v.y), pi[0], pi[32]);
        }
    }
}

__global__ void iota_kernel(int* p, int* q, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = q[i] = i;
}

// A ROWS x COLS tile of view A at (r0, c0) into shared memory (column-major, leading dimension
// ROWS), zero outside nr x nc.  Each thread issues all its global loads before its first shared
// store, so one memory latency covers the whole tile (256 threads).
template <int ROWS, int COLS, class V>
__device__ __forceinline__ void load_tile(typename V::cv* dst, const V& A, long r0, long c0, int nr, int nc) {
    using CV = typename V::cv;
    using Rl = typename V::real;
    static_assert(ROWS * COLS % 256 == 0, "tile must split evenly over 256 threads");
    constexpr int PER = ROWS * COLS / 256;
    CV v[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) {
        const int e = threadIdx.x + 256 * m;
        const int i = e % ROWS, j = e / ROWS;
        v[m] = (i < nr && j < nc) ? A.get(r0 + i, c0 + j) : czero<Rl>();
    }
#pragma unroll
    for (int m = 0; m < PER; ++m) dst[threadIdx.x + 256 * m] = v[m];
}

// The same for a dense column-major B x B block (leading dimension B), zero outside n x n.
template <int B, class CV>
__device__ __forceinline__ void load_block(CV* dst, const CV* __restrict__ src, int nb) {
    static_assert(B * B % 256 == 0, "block must split evenly over 256 threads");
    constexpr int PER = B * B / 256;
    CV v[PER];
#pragma unroll
    for (int m = 0; m < PER; ++m) {
        const int e = threadIdx.x + 256 * m;
        const int i = e % B, j = e / B;
        v[m] = (i < nb && j < nb) ? src[e] : CV{};
    }
#pragma unroll
    for (int m = 0; m < PER; ++m) dst[threadIdx.x + 256 * m] = v[m];
}

// Inverse of each 64 x 64 diagonal block (unit lower L or upper U) of the LU factor, by a
// column sweep over X = I: for k in order (L: 0..rb-1; U: rb-1..0, row k first divided by U_kk),
// every later row i takes X_i -= T_ik X_k.  Thread t holds X[t % 64, t / 64 + 4 m] (m < 16) in
// registers; row k goes through a double-buffered shared row, so each step needs one barrier
// (the reciprocals 1 / U_kk are formed before the sweep).
// Entries outside the rb x rb leading block are zero.
constexpr int TI_B = 64;
template <bool UPPER>
__global__ void __launch_bounds__(256) tri_inv_kernel(C32 F, int n, float2* __restrict__ out, const int* fail) {
    using CV = float2;
    using Rl = float;
    if (*fail != 0) return;  // the factorisation stopped (lu_fast.cu) and is continued first
    constexpr int B = TI_B, M = B * B / 256;
    extern __shared__ __align__(16) unsigned char sm[];
    CV* T = reinterpret_cast<CV*>(sm);  // [B][B] column-major
    CV* buf = T + B * B;                // [2][B]
    CV* dg = buf + 2 * B;               // [B] 1 / U_kk
    const int t = threadIdx.x, i = t % B, c0 = t / B;
    const long r0 = (long)blockIdx.x * B;
    const int rb = (int)min((long)B, n - r0);
    load_tile<B, B>(T, F, r0, r0, rb, rb);
    if (UPPER && t < rb) dg[t] = cinv(F.get(r0 + t, r0 + t));
    CV x[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        x[m] = czero<Rl>();
        if (i == c0 + 4 * m && i < rb) x[m].x = (Rl)1;
    }
    __syncthreads();
    for (int s = 0; s < rb; ++s) {
        const int k = UPPER ? rb - 1 - s : s;
        CV* bk = buf + (s & 1) * B;
        if (i == k) {
            if (UPPER) {
                const CV d = dg[k];
#pragma unroll
                for (int m = 0; m < M; ++m) x[m] = cmul(x[m], d);
            }
#pragma unroll
            for (int m = 0; m < M; ++m) bk[c0 + 4 * m] = x[m];
        }
        __syncthreads();
        if (UPPER ? i < k : (i > k && i < rb)) {
            CV tik = T[i + k * B];
            tik.x = -tik.x;
            tik.y = -tik.y;
#pragma unroll
            for (int m = 0; m < M; ++m) cfma(x[m], tik, bk[c0 + 4 * m]);
        }
    }
    CV* o = out + (long)blockIdx.x * B * B;
#pragma unroll
    for (int m = 0; m < M; ++m) o[i + (c0 + 4 * m) * B] = x[m];
}

constexpr int TS_BM = 64;
// G form of the factors (C32): every off-diagonal bs x bs tile F[it, b] (it != b) becomes
// F[it, b] T_b with T_b = L_bb^{-1} below the diagonal and U_bb^{-1} above it.  One CTA per tile,
// in place (each CTA reads its whole tile before writing it).  bs == TS_BM == 64.
__global__ void __launch_bounds__(256) g_form_kernel(C32 F, int n, const float2* __restrict__ dinvL,
                                                     const float2* __restrict__ dinvU, const int* fail) {
    using CV = float2;
    using Rl = float;
    constexpr int B = TS_BM;
    const int it = blockIdx.x, b = blockIdx.y;
    if (it == b || *fail != 0) return;
    extern __shared__ __align__(16) unsigned char sm[];
    CV* Ft = reinterpret_cast<CV*>(sm);  // [B][B] column-major tile of F
    CV* Ts = Ft + B * B;                 // [B][B] column-major T_b
    const int t = threadIdx.x;
    const long r0 = (long)it * B, c0 = (long)b * B;
    const int tm = (int)min((long)B, n - r0), rb = (int)min((long)B, n - c0);
    const CV* T = (it > b ? dinvL : dinvU) + (long)b * B * B;
    load_tile<B, B>(Ft, F, r0, c0, tm, rb);
    load_block<B>(Ts, T, rb);
    __syncthreads();
    const int tx = t % 16, ty = t / 16;  // rows tx + 16 a, columns ty + 16 c
    CV acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[a][c] = czero<Rl>();
    for (int k = 0; k < rb; ++k) {
        CV fv[4], tv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) fv[a] = Ft[k * B + tx + 16 * a];
#pragma unroll
        for (int c = 0; c < 4; ++c) tv[c] = Ts[k + (ty + 16 * c) * B];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) cfma(acc[a][c], fv[a], tv[c]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int i = tx + 16 * a;
        if (i >= tm) continue;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int j = ty + 16 * c;
            if (j < rb) F.set(r0 + i, c0 + j, acc[a][c]);
        }
    }
}

// Waits for a flag (bounded: 1 s by the global timer, then *err is raised).
__device__ __forceinline__ void flow_wait(const int* flag, int* err) {
    if (*reinterpret_cast<volatile int*>(err) != 0) return;  // an earlier wait gave up: no more waiting
    uint64_t t0 = 0;
    for (int it = 0;; ++it) {
        int v;
        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v != 0) return;
        if (it == 0) t0 = gtime();
        else if (gtime() - t0 > 1000000000ull) {
            atomicExch(err, 1);
            return;
        }
    }
}
// Persistent blocked triangular solve in G form (C32): the block steps and the diagonal blocks of
// one triangle (forward: lower, backward: upper) in a single cooperative launch.  Work item (i, j)
// is tile row i (64 rows) of column tile j (8 right-hand sides).  It accumulates
// sum_b G[i, b] Y[b, j] over the tile rows b before i (lower) or after i (upper), each as soon as item
// (b, j) has published its final rows, publishes Y[i, j] minus that sum and writes
// Z[i, j] = T_i Y[i, j] with T_i the inverted diagonal block.
// The chain of tile rows bounds the launch, so a link is kept short: the published rows are their own flag
// (xch starts as FL_UNSET words, a bit pattern that arithmetic never produces; a reader polls the 16 bytes it
// needs, one trip to L2 instead of a flag, a fence and a read), and the tiles of G arrive by cp.async in two
// buffers while the step before is multiplied, with one barrier per step.  65 right-hand sides, one triangle,
// n = 4096: 305 -> 193 us; n = 8192: 990 -> 583 us; 8 right-hand sides, n = 2048: 123 -> 57 us (1.8 us a link)
// against flags, fences and single-buffered tiles.
// CTA q takes items q, q + grid, ... in dependency order, so the earliest unfinished item never waits; with
// every CTA resident (cooperative launch) no wait can deadlock.  Waits are bounded (1 s by the global timer): a
// timeout raises *err and the item goes on with what it has.
constexpr int FL_BN = FLOW_BN, FL_T = 256, FL_TILE = 2 * TS_BM * TS_BM;  // threads; floats of a tile of G or T
static_assert(TS_BM * FL_BN == 2 * FL_T, "a thread per pair of entries of an item");
static_assert(FLOW_ITEM_BYTES == FL_T * sizeof(float4), "an item's rows in xch: [pair of columns][row] float4");
constexpr uint32_t FL_UNSET = 0xffffffffu;
__device__ __forceinline__ bool flow_load(const float4* p, float4& v) {
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p)
                 : "memory");
    return __float_as_uint(v.x) != FL_UNSET && __float_as_uint(v.y) != FL_UNSET && __float_as_uint(v.z) != FL_UNSET &&
           __float_as_uint(v.w) != FL_UNSET;
}
__device__ __forceinline__ float4 flow_take(const float4* p, int* err) {
    float4 v;
    if (flow_load(p, v)) return v;
    const uint64_t t0 = gtime();
    for (int it = 1;; ++it) {
        if (flow_load(p, v)) return v;
        if ((it & 31) == 0) {
            if (*reinterpret_cast<volatile int*>(err) != 0) return v;  // an earlier wait gave up: no more waiting
            if (gtime() - t0 > 1000000000ull) {
                atomicExch(err, 1);
                return v;
            }
        }
    }
}
__device__ __forceinline__ float flow_word(float v) { return __float_as_uint(v) == FL_UNSET ? __int_as_float(0x7fffffff) : v; }
__device__ __forceinline__ void flow_publish(float4* p, float4 v) {
    asm volatile("st.relaxed.gpu.global.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(flow_word(v.x)),
                 "f"(flow_word(v.y)), "f"(flow_word(v.z)), "f"(flow_word(v.w))
                 : "memory");
}
// 16 bytes global -> shared, the last 16 - bytes of them zeros
__device__ __forceinline__ void cp_async16z(void* dst, const void* src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
// acc[c] += sum_k M[r, k] V[k, c] over this thread's 16 k from k0: M column-major 64 x 64, planar (G) or
// interleaved (T); V [pair of columns][row]
template <bool PLANAR>
__device__ __forceinline__ void flow_mac(float2 (&acc)[FL_BN], const float* M, const float4* V, int r, int k0) {
#pragma unroll 4
    for (int k = k0; k < k0 + TS_BM / 4; ++k) {
        const float2 g = PLANAR ? make_float2(M[k * TS_BM + r], M[FL_TILE / 2 + k * TS_BM + r])
                                : reinterpret_cast<const float2*>(M)[k * TS_BM + r];
#pragma unroll
        for (int c2 = 0; c2 < FL_BN / 2; ++c2) {
            const float4 y = V[c2 * TS_BM + k];
            cfma(acc[2 * c2], g, make_float2(y.x, y.y));
            cfma(acc[2 * c2 + 1], g, make_float2(y.z, y.w));
        }
    }
}
template <bool UPPER>
__global__ void __launch_bounds__(FL_T, 3) trsv_flow_kernel(C32 F, C32 Y, C32 Z, int n, int nrhs,
                                                            const float2* __restrict__ Tinv, float4* xch, int* err,
                                                            const float4* never, const int* hook) {
    constexpr int B = TS_BM, BN = FL_BN;
    extern __shared__ __align__(16) unsigned char sm[];
    float* const Gs = reinterpret_cast<float*>(sm);                 // [2] tiles of G, the last one T_i
    float4* const Ys = reinterpret_cast<float4*>(Gs + 2 * FL_TILE);  // [2] Y[b, j], the last one Y[i, j]
    const int t = threadIdx.x;
    const int nblk = (n + B - 1) / B, ct = (nrhs + BN - 1) / BN;
    const int items = nblk * ct;
    // this thread: row r; columns 2 ks, 2 ks + 1 of the item's rows, k in [16 ks, 16 ks + 16) of the products
    const int r = t % B, ks = t / B, k0 = ks * (B / 4);
    const bool hooked = never != nullptr && *hook != 0;  // test hook (set at assembly)
    for (int q = blockIdx.x; q < items; q += gridDim.x) {
        __syncthreads();  // the previous item is done with the shared buffers
        const int i = UPPER ? nblk - 1 - q / ct : q / ct, j = q % ct;
        const long r0 = (long)i * B;
        const int tm = (int)min((long)B, n - r0);
        const int j0 = j * BN;
        const int nsteps = UPPER ? nblk - 1 - i : i;
        // step st's tile (the last one: T_i) into buffer st & 1, zeros outside the matrix
        auto fetch = [&](int st) {
            float* dst = Gs + (st & 1) * FL_TILE;
            if (st == nsteps) {
                const float2* T = Tinv + (long)i * B * B;
#pragma unroll
                for (int m = 0; m < FL_TILE / 4 / FL_T; ++m) {
                    const int e = t + FL_T * m, k = e / (B / 2), x = 2 * (e % (B / 2));
                    const int bytes = k < tm ? 8 * min(max(tm - x, 0), 2) : 0;
                    cp_async16z(dst + 4 * e, T + k * B + x, bytes);
                }
            } else {
                const long c0 = (long)(UPPER ? nblk - 1 - st : st) * B;
                const int rb = (int)min((long)B, n - c0);
#pragma unroll
                for (int m = 0; m < FL_TILE / 8 / FL_T; ++m) {
                    const int e = t + FL_T * m, k = e / (B / 4), x = 4 * (e % (B / 4));
                    const int bytes = k < rb ? 4 * min(max(tm - x, 0), 4) : 0;
                    const long o = bytes > 0 ? r0 + x + (c0 + k) * F.ld : 0;
                    cp_async16z(dst + 4 * e, F.re + o, bytes);
                    cp_async16z(dst + FL_TILE / 2 + 4 * e, F.im + o, bytes);
                }
            }
            cp_async_commit();
        };
        fetch(0);
        // this item's own right-hand-side rows (zeros outside)
        float2 own[2];
#pragma unroll
        for (int c = 0; c < 2; ++c)
            own[c] = r < tm && j0 + 2 * ks + c < nrhs ? Y.get(r0 + r, (long)j0 + 2 * ks + c) : make_float2(0.f, 0.f);
        float2 acc[BN];
#pragma unroll
        for (int c = 0; c < BN; ++c) acc[c] = make_float2(0.f, 0.f);
        for (int st = 0; st < nsteps; ++st) {
            const int b = UPPER ? nblk - 1 - st : st;
            // (test hook: the last item's first wait is on rows that nothing publishes)
            const float4* from = (hooked && q == items - 1 && st == 0) ? never : xch + (long)(b * ct + j) * FL_T;
            Ys[(st & 1) * FL_T + t] = flow_take(from + t, err);
            cp_async_wait<0>();
            __syncthreads();  // this step's operands are there; the step before has been multiplied
            fetch(st + 1);
            flow_mac<true>(acc, Gs + (st & 1) * FL_TILE, Ys + (st & 1) * FL_T, r, k0);
        }
        // sums over the four k ranges through the buffer of G that is free, [k range][pair of columns][row]
        float4* const Red = reinterpret_cast<float4*>(Gs + ((nsteps + 1) & 1) * FL_TILE);
        auto reduce = [&]() {
#pragma unroll
            for (int c2 = 0; c2 < BN / 2; ++c2)
                Red[(ks * (BN / 2) + c2) * B + r] =
                    make_float4(acc[2 * c2].x, acc[2 * c2].y, acc[2 * c2 + 1].x, acc[2 * c2 + 1].y);
            __syncthreads();
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2) {
                const float4 p = Red[(q2 * (BN / 2) + ks) * B + r];
                v.x += p.x, v.y += p.y, v.z += p.z, v.w += p.w;
            }
            return v;
        };
        __syncthreads();  // the last step has been multiplied
        float4 y = reduce();
        y = make_float4(own[0].x - y.x, own[0].y - y.y, own[1].x - y.z, own[1].y - y.w);
        flow_publish(xch + (long)(i * ct + j) * FL_T + t, y);
        Ys[(nsteps & 1) * FL_T + t] = y;
        cp_async_wait<0>();
        __syncthreads();  // T_i and Y[i, j]
        // Z[i, j] = T_i Y[i, j]
#pragma unroll
        for (int c = 0; c < BN; ++c) acc[c] = make_float2(0.f, 0.f);
        flow_mac<false>(acc, Gs + (nsteps & 1) * FL_TILE, Ys + (nsteps & 1) * FL_T, r, k0);
        const float4 z = reduce();
        if (r < tm) {
            if (j0 + 2 * ks < nrhs) Z.set(r0 + r, (long)j0 + 2 * ks, make_float2(z.x, z.y));
            if (j0 + 2 * ks + 1 < nrhs) Z.set(r0 + r, (long)j0 + 2 * ks + 1, make_float2(z.z, z.w));
        }
    }
}

// Inverses of the 16 x 16 diagonal blocks of the FP64 factors: a block per half warp, lane = column,
// the unit lower triangles for blockIdx.y = 0, the upper ones for 1.  Rows and columns past n are the
// identity's.  out: column-major 16 x 16 blocks.
constexpr int FZ_B = 16, FZ_NC = 4;
__global__ void __launch_bounds__(32) tri_inv16_kernel(Z64 F, int n, double2* __restrict__ outL,
                                                       double2* __restrict__ outU, const int* fail) {
    if (*fail != 0) return;
    const int lane = threadIdx.x & 31, j = lane & 15, blk = (int)blockIdx.x * 2 + (lane >> 4);
    const long r0 = (long)blk * FZ_B;
    const bool upper = blockIdx.y == 1;
    double2 x[FZ_B];
    auto at = [&](int i, int k) {
        return r0 + max(i, k) < n ? F.get(r0 + i, r0 + k) : (i == k ? make_double2(1.0, 0.0) : make_double2(0.0, 0.0));
    };
    if (upper) {
        const double2 dinv = cinv(at(j, j));
#pragma unroll
        for (int i = FZ_B - 1; i >= 0; --i) {
            double2 s = make_double2(i == j ? 1.0 : 0.0, 0.0);
#pragma unroll
            for (int k = i + 1; k < FZ_B; ++k) {
                const double2 t = at(i, k);
                cfma(s, make_double2(-t.x, -t.y), x[k]);
            }
            const int src = (lane & 16) + i;
            x[i] = cmul(s, make_double2(__shfl_sync(0xffffffffu, dinv.x, src), __shfl_sync(0xffffffffu, dinv.y, src)));
        }
    } else {
#pragma unroll
        for (int i = 0; i < FZ_B; ++i) {
            double2 s = make_double2(i == j ? 1.0 : 0.0, 0.0);
#pragma unroll
            for (int k = 0; k < i; ++k) {
                const double2 t = at(i, k);
                cfma(s, make_double2(-t.x, -t.y), x[k]);
            }
            x[i] = s;
        }
    }
    if (r0 >= n) return;
    double2* o = (upper ? outU : outL) + (long)blk * FZ_B * FZ_B + j * FZ_B;
#pragma unroll
    for (int i = 0; i < FZ_B; ++i) o[i] = x[i];
}

// The FP64 triangular solve as one persistent cooperative launch per triangle (the scheme of
// trsv_flow_kernel).  Work item (i, j): tile row i of 16 rows, 4 right-hand sides; it takes
// Y[i, j] - sum_b F[i, b] X[b, j] over the tile rows before it, each as soon as ready[b, j] is set, then
// X[i, j] = T_i (that) with the inverted 16 x 16 diagonal block, and publishes.  An SM does two FP64
// multiply-adds a cycle, so a link of the chain costs its two 16 x 16 x 4 products (2 us) besides the flag
// and the loads; 64-row block steps cost 77 us per block instead (each CTA recomputed the diagonal block's
// product, padded to 16 columns).  N = 1000, four right-hand sides: 2.46 -> 0.6 ms.  Thread: row t % 16,
// column, half of the k range.
template <bool UPPER>
__global__ void __launch_bounds__(128, 8) trsv_flow_z64_kernel(Z64 F, Z64 Y, Z64 X, int n, int nrhs,
                                                               const double2* __restrict__ Tinv, int* ready, int* err) {
    constexpr int B = FZ_B, NC = FZ_NC, KH = B / 2;
    __shared__ double2 red[2][NC][B];
    __shared__ double2 ys[NC][B];
    const int t = threadIdx.x, r = t % B, c = (t / B) % NC, ks = t / (B * NC), k0 = ks * KH;
    const int nblk = (n + B - 1) / B, ct = (nrhs + NC - 1) / NC, items = nblk * ct;
    pdl_wait();
    pdl_trigger();
    for (int q = blockIdx.x; q < items; q += gridDim.x) {
        const int i = UPPER ? nblk - 1 - q / ct : q / ct, j = q % ct;
        const long r0 = (long)i * B, row = r0 + r;
        const int col = j * NC + c;
        const bool in = row < n && col < nrhs;
        double2 f[KH], ti[KH];
        auto load_f = [&](int b) {
#pragma unroll
            for (int k = 0; k < KH; ++k) {
                const long fc = (long)b * B + k0 + k;
                f[k] = (row < n && fc < n) ? F.get(row, fc) : make_double2(0.0, 0.0);
            }
        };
        const int nsteps = UPPER ? nblk - 1 - i : i;
        if (nsteps > 0) load_f(UPPER ? nblk - 1 : 0);
        const double2 y0 = in ? Y.get(row, col) : make_double2(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < KH; ++k) ti[k] = Tinv[(long)i * B * B + (k0 + k) * B + r];
        double2 acc = make_double2(0.0, 0.0);
        for (int st = 0; st < nsteps; ++st) {
            const int b = UPPER ? nblk - 1 - st : st;
            double2 g[KH];
#pragma unroll
            for (int k = 0; k < KH; ++k) g[k] = f[k];
            if (st + 1 < nsteps) load_f(UPPER ? b - 1 : b + 1);  // the next tile, while this one waits
            flow_wait(ready + b * ct + j, err);
            double2 x[KH];
#pragma unroll
            for (int k = 0; k < KH; ++k) {
                const long xr = (long)b * B + k0 + k;
                x[k] = (xr < n && col < nrhs) ? __ldcg(X.p + xr + (long)col * X.ld) : make_double2(0.0, 0.0);
            }
#pragma unroll
            for (int k = 0; k < KH; ++k) cfma(acc, g[k], x[k]);
        }
        red[ks][c][r] = acc;
        __syncthreads();
        if (ks == 0) ys[c][r] = csub(y0, cadd(red[0][c][r], red[1][c][r]));
        __syncthreads();
        double2 z = make_double2(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < KH; ++k) cfma(z, ti[k], ys[c][k0 + k]);
        red[ks][c][r] = z;
        __syncthreads();
        if (ks == 0 && in) X.set(row, col, cadd(red[0][c][r], red[1][c][r]));
        __syncthreads();  // orders every thread's rows before the release (cumulative at gpu scope)
        if (t == 0) asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(ready + i * ct + j), "r"(1) : "memory");
    }
}

__global__ void gather_rows_z64_kernel(const int* __restrict__ perm, int n, int nrhs, const double2* __restrict__ B,
                                       long ldb, double2* __restrict__ Y, long ldy) {
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)n * nrhs) return;
    int c = (int)(idx / n), i = (int)(idx % n);
    Y[i + (long)c * ldy] = B[perm[i] + (long)c * ldb];
}
__global__ void gather_rows_c32_kernel(const int* __restrict__ perm, int n, int nrhs, const float* __restrict__ Br,
                                       const float* __restrict__ Bi, long ldb, float* __restrict__ Yr,
                                       float* __restrict__ Yi, long ldy) {
    long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)n * nrhs) return;
    int c = (int)(idx / n), i = (int)(idx % n);
    Yr[i + (long)c * ldy] = Br[perm[i] + (long)c * ldb];
    Yi[i + (long)c * ldy] = Bi[perm[i] + (long)c * ldb];
}

// ------------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------------
#define LU_CUDA(expr)                                                                                  \
    do {                                                                                               \
        cudaError_t _e = (expr);                                                                       \
        if (_e != cudaSuccess) {                                                                       \
            bm_set_error(std::string("lu: ") + #expr + ": " + cudaGetErrorString(_e));                 \
            return BM_ECUDA;                                                                           \
        }                                                                                              \
    } while (0)

template <class V>
cudaError_t launch_swap_trsm(cudaStream_t s, V A, const SwapMap* map, int a0, int a1, int b0, int b1, int t0, int tb,
                             __half* Upr, __half* Upi, long ldk, int* Upe, const int* re = nullptr,
                             const int* perm = nullptr) {
    using CV = typename V::cv;
    long ncols = (long)(a1 - a0) + (b1 - b0);
    if (ncols <= 0) return cudaSuccess;
    // L11 staging: whole (1) when it fits 160 KB, else in ST_KC-column chunks (2)
    size_t lbytes = (size_t)tb * tb * sizeof(CV);
    int l_in_smem = tb <= 0 ? 0 : (lbytes <= 160 * 1024 ? 1 : 2);
    size_t smem = l_in_smem == 1 ? lbytes : (l_in_smem == 2 ? (size_t)tb * ST_KC * sizeof(CV) : 0);
    auto kern = swap_trsm_kernel<V>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    int grid = ceil_div(ncols, ST_WARPS * ST_COLS);
    return launch_pdl(kern, dim3(grid), dim3(ST_WARPS * 32), smem, s, A, map, a0, a1, b0, b1, t0, tb, Upr, Upi, ldk,
                      Upe, re, perm, l_in_smem);
}

cudaError_t gemm_any(cudaStream_t s, int m, int n, int k, Z64 A, Z64 B, Z64 C) {
    return gemm_z64(s, m, n, k, -1.0, A, B, 1.0, C);
}
cudaError_t gemm_any(cudaStream_t s, int m, int n, int k, C32 A, C32 B, C32 C) {
    return gemm_c32(s, m, n, k, -1.0f, A, B, 1.0f, C);
}

// Exponents of the rows of the factored matrix for the inner scale of its updates: the ordinary system's, whose
// block rows differ (the Schur complement's rows do not).
const int* row_exponents(const bm_ctx* c) { return c->form == BM_ORDINARY ? c->d_dge[0] : nullptr; }

// What the solves need besides the factors: the inverted diagonal blocks and (FP32) the G form.
bm_status finish_t(bm_ctx* c, Z64 F, cudaStream_t s) {
    BM_PROF(c, "tri_inv16_kernel");
    tri_inv16_kernel<<<dim3(ceil_div(ceil_div(c->n, FZ_B), 2), 2), 32, 0, s>>>(
        F, c->n, reinterpret_cast<double2*>(c->d_dinvL), reinterpret_cast<double2*>(c->d_dinvU), c->d_info + 4);
    LU_CUDA(cudaGetLastError());
    return BM_OK;
}
bm_status finish_t(bm_ctx* c, C32 F, cudaStream_t s) {
    const int n = c->n, nblk = ceil_div(n, TI_B);
    const int* const fail = c->d_info + 4;
    float2* const dinvL = reinterpret_cast<float2*>(c->d_dinvL);
    float2* const dinvU = reinterpret_cast<float2*>(c->d_dinvU);
    static_assert(TI_B == TS_BM, "one block size for the inverses and the G form");
    constexpr int smem = (TI_B * TI_B + 3 * TI_B) * (int)sizeof(float2), gsm = 2 * TS_BM * TS_BM * (int)sizeof(float2);
    LU_CUDA(cudaFuncSetAttribute(tri_inv_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LU_CUDA(cudaFuncSetAttribute(tri_inv_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    {
        BM_PROF(c, "tri_inv_kernel");
        tri_inv_kernel<false><<<nblk, 256, smem, s>>>(F, n, dinvL, fail);
        tri_inv_kernel<true><<<nblk, 256, smem, s>>>(F, n, dinvU, fail);
        LU_CUDA(cudaGetLastError());
    }
    if (nblk > 1) {
        BM_PROF(c, "g_form_kernel");
        LU_CUDA(cudaFuncSetAttribute(g_form_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, gsm));
        g_form_kernel<<<dim3(nblk, nblk), 256, gsm, s>>>(F, n, dinvL, dinvU, fail);
        LU_CUDA(cudaGetLastError());
    }
    return BM_OK;
}

// The FP32 LU in blocks of FD_B columns without a pivot search (lu_fast.cu).  Two streams: the chain
// diagonal block -> solves -> next diagonal block's tile, and the rest of each trailing update beside
// the next diagonal block.
bm_status factor_fast(bm_ctx* c, C32 F) {
    const int n = c->n;
    int* const fail = c->d_info + 4;
    const bool la = !c->prof && n > 2 * FD_B && c->la_hi != nullptr;
    cudaStream_t s = la ? c->la_hi : c->stream;
    cudaStream_t s2 = c->la_lo;
    cudaEvent_t ev_start = c->la_ev[0], ev_fork = c->la_ev[1], ev_join = c->la_ev[2], ev_done = c->la_ev[3];
    if (la) {
        LU_CUDA(cudaEventRecord(ev_start, c->stream));
        LU_CUDA(cudaStreamWaitEvent(s, ev_start, 0));
    }
    {
        BM_PROF(c, "iota");
        iota_kernel<<<ceil_div(n, 256), 256, 0, s>>>(c->d_perm, c->d_ipiv, n);
        LU_CUDA(cudaGetLastError());
    }
    const TcPacks packs{c->d_Lp_r, c->d_Lp_i, c->d_Up_r, c->d_Up_i, c->d_Lpe, c->d_Upe, row_exponents(c), c->ldk_lu};
    bool rest = false;  // a trailing update is under way on s2
    for (int J = 0; J < n; J += FD_B) {
        const int db = std::min(FD_B, n - J), mm = n - J - db;
        {
            // (the profile keeps one name for the kernels that eliminate the panels)
            BM_PROF(c, "panel_lc_kernel");
            LU_CUDA(launch_lu_diag(s, F, J, db, c->d_fd, fail));
        }
        if (rest) LU_CUDA(cudaStreamWaitEvent(s, ev_join, 0));
        {
            BM_PROF(c, "lu_trsm_kernel");
            LU_CUDA(launch_lu_trsm(s, F, J, db, mm, c->d_fd, n, packs, fail));
        }
        rest = false;
        if (mm == 0) break;
        BM_PROF(c, "cgemm_tc_kernel (trailing update)");
        const C32 C = F.sub(J + FD_B, J + FD_B);
        // (persistent CTAs on all SMs but one, which the next diagonal block takes meanwhile)
        TcGate gate{fail, J + 1, 0};
        auto update = [&](cudaStream_t st, int m) {
            return gemm_tc_upd(st, c->tm_lu[0], c->tm_lu[1], c->tm_lu[2], c->tm_lu[3], C.re, C.im, C.ld, m, m, FD_B,
                               TcScale{c->d_Lpe, c->d_Upe, 0}, c->num_sms - 1, c->d_err, gate);
        };
        if (!la || mm <= FD_B) {
            LU_CUDA(update(s, mm));
            continue;
        }
        LU_CUDA(cudaEventRecord(ev_fork, s));
        LU_CUDA(update(s, FD_B));
        LU_CUDA(cudaStreamWaitEvent(s2, ev_fork, 0));
        gate.first_tile = 1;
        LU_CUDA(update(s2, mm));
        LU_CUDA(cudaEventRecord(ev_join, s2));
        rest = true;
    }
    BM_TRY(finish_t(c, F, s));
    if (la) {  // join the handle's stream
        LU_CUDA(cudaEventRecord(ev_done, s));
        LU_CUDA(cudaStreamWaitEvent(c->stream, ev_done, 0));
    }
    return BM_OK;
}

// the inner scale of the product of the columns and rows from J on (rows in place: no interchange so far)
RtShift inner_z(const bm_ctx* c, int J) {
    RtShift sh;
    if (const int* re = row_exponents(c)) sh.re = re + J;
    return sh;
}

// A[e:, e:] -= A[e:, J:e] A[J:e, e:], by digits on the tensor cores where that is the faster (dg_bytes) and the
// workspace is there, else on the FP64 pipe.
bm_status update_z(bm_ctx* c, Z64 F, int J, int c1, int e, const int* stop) {
    const int m = c->n - e, k = c1 - J;
    const size_t need = dg_bytes(m, m, k, c->num_sms);
    const bool digits = need > 0 && need <= c->dgw_bytes;
    BM_PROF(c, digits ? "resid_tc_kernel (trailing update)" : "cgemm_simt_kernel (trailing update)");
    if (digits)
        return gemm_z64_dg(c->stream, c->d_dgw, c->num_sms, m, m, k, -1.0, F.sub(e, J), F.sub(J, e), F.sub(e, e), c->d_err,
                           nullptr, inner_z(c, J), stop);
    LU_CUDA(gemm_z64(c->stream, m, m, k, -1.0, F.sub(e, J), F.sub(J, e), 1.0, F.sub(e, e), stop));
    return BM_OK;
}

// The FP64 LU in blocks of FZ_BLOCK columns without a pivot search (lu_fast_z.cu), outer blocks of FZ_OUTER:
// inside one, each block updates the rest of the outer block's columns and rows on the FP64 pipe; then the
// trailing matrix takes the outer block's product.
bm_status factor_fast_z(bm_ctx* c, Z64 F) {
    const int n = c->n;
    cudaStream_t s = c->stream;
    int* const fail = c->d_info + 4;
    double2* const work = reinterpret_cast<double2*>(c->d_fd);
    {
        BM_PROF(c, "iota");
        iota_kernel<<<ceil_div(n, 256), 256, 0, s>>>(c->d_perm, c->d_ipiv, n);
        LU_CUDA(cudaGetLastError());
    }
    for (int J = 0; J < n; J += FZ_OUTER) {
        const int je = std::min(J + FZ_OUTER, n);
        for (int j = J; j < je; j += FZ_BLOCK) {
            const int db = std::min(FZ_BLOCK, n - j), e = j + db, mm = n - e;
            {
                BM_PROF(c, "lu_diag_z_kernel");
                LU_CUDA(launch_lu_diag_z(s, F, j, db, work, fail));
            }
            {
                BM_PROF(c, "lu_trsm_z_kernel");
                LU_CUDA(launch_lu_trsm_z(s, F, j, db, mm, work, n, fail));
            }
            if (mm == 0 || e >= je) continue;
            BM_PROF(c, "cgemm_simt_kernel (panel update)");
            LU_CUDA(gemm_z64(s, mm, je - e, db, -1.0, F.sub(e, j), F.sub(j, e), 1.0, F.sub(e, e), fail));
            if (je < n)
                LU_CUDA(gemm_z64(s, je - e, n - je, db, -1.0, F.sub(e, j), F.sub(j, je), 1.0, F.sub(e, je), fail));
        }
        if (je == n) break;
        BM_TRY(update_z(c, F, J, je, je, fail));
    }
    return finish_t(c, F, s);
}

// The LU with the pivot search, from column J0 on (the columns before it are factored, their
// interchanges and trailing updates applied).
template <class V>
bm_status factor_t(bm_ctx* c, V F, bool tc, int J0 = 0) {
    const int n = c->n;
    const int NB = c->nb;
    const int cl_max = c->panel_cluster;
    SwapMap* const maps = reinterpret_cast<SwapMap*>(c->d_maps);
    SwapMap* const d_map2 = maps + 1;  // sub-panel map (register-row panels)
    // Look-ahead (FP32 with tensor-core trailing updates): after big panel J, the interchanges,
    // U12 solve and trailing update of the next big panel's columns run first on the high-priority
    // stream, which then factors that panel while the low-priority stream finishes the rest of the
    // trailing update; the next block step waits for it.  Profiling keeps the serial order.
    const bool la = std::is_same<V, C32>::value && tc && !c->prof && n - J0 > 2 * NB && c->la_hi != nullptr;
    cudaStream_t s = la ? c->la_hi : c->stream;
    cudaStream_t s2 = c->la_lo;
    cudaEvent_t ev_start = c->la_ev[0], ev_fork = c->la_ev[1], ev_join = c->la_ev[2], ev_done = c->la_ev[3];
    if (la) {
        LU_CUDA(cudaEventRecord(ev_start, c->stream));
        LU_CUDA(cudaStreamWaitEvent(s, ev_start, 0));
        LU_CUDA(cudaStreamWaitEvent(s2, ev_start, 0));
    }
    if (J0 == 0) {
        BM_PROF(c, "iota");
        iota_kernel<<<ceil_div(n, 256), 256, 0, s>>>(c->d_perm, c->d_ipiv, n);
        LU_CUDA(cudaGetLastError());
    }
    for (int J = J0, blk = 0; J < n; J += NB, ++blk) {
        const int jb = std::min(NB, n - J);
        SwapMap* const d_map = (blk & 1) ? maps + 2 : maps;  // this big panel's map (two in flight)
        for (int j = J; j < J + jb;) {
            PanelShape ps;
            if (!panel_shape<V>(n - j, cl_max, c->panel_lane_col, ps)) {
                bm_set_error("lu: system too large for the panel kernel");
                return BM_EINVAL;
            }
            const int ib = std::min(ps.nbp, J + jb - j);
            // the lane-per-column kernel (FP32) also applies the sub-panel's interchanges to the
            // big panel's other columns and solves L11 against its columns on the right
            bool fused = false;
            if constexpr (std::is_same<V, C32>::value) {
                if (ps.RPW > 0) {
                    BM_PROF(c, "panel_lc_kernel");
                    LcParams lp{F, j, n - j, ib, J, jb, c->d_ipiv, c->d_info, c->d_info + 1, d_map, c->d_perm};
                    LU_CUDA(launch_panel_lc(s, ps, lp));
                    fused = true;
                }
            }
            if (!fused) {
                BM_PROF(c, "panel_kernel");
                LU_CUDA(launch_panel(s, F, ps, j, n - j, ib, c->d_ipiv, c->d_info, J, jb, d_map2, d_map, c->d_perm));
            }
            if (jb > ib) {
                if (!fused) {
                    BM_PROF(c, "swap_trsm_kernel (sub-panel)");
                    LU_CUDA(launch_swap_trsm<V>(s, F, d_map2, J, j, j + ib, J + jb, j, ib, nullptr, nullptr, 0, nullptr));
                }
                if (j + ib < J + jb) {
                    BM_PROF(c, "cgemm_simt_kernel (panel update)");
                    LU_CUDA(gemm_any(s, n - j - ib, J + jb - j - ib, ib, F.sub(j + ib, j), F.sub(j, j + ib),
                                     F.sub(j + ib, j + ib)));
                }
            }
            j += ib;
        }
        const bool pack = tc && (J + jb < n);
        const int mm = n - J - jb;          // trailing rows and columns
        const int nnext = la ? std::min(NB, mm) : mm;  // trailing columns updated on s
        // the rest of the previous trailing update (columns this block row touches) is done
        if (la && blk > 0) LU_CUDA(cudaStreamWaitEvent(s, ev_join, 0));
        {
            BM_PROF(c, "swap_trsm_kernel (block row)");
            // on s: the next big panel's columns (all trailing columns without look-ahead), and the
            // columns left of this panel unless the rest stream takes them
            LU_CUDA(launch_swap_trsm<V>(s, F, d_map, 0, la ? 0 : J, J + jb, J + jb + nnext, J, jb,
                                        pack ? c->d_Up_r : nullptr, pack ? c->d_Up_i : nullptr, c->ldk_lu, c->d_Upe,
                                        row_exponents(c), c->d_perm));
        }
        if (mm > 0) {
            if (tc) {
                if constexpr (std::is_same<V, C32>::value) {
                    {
                        BM_PROF(c, "pack_L_kernel");
                        pack_L_kernel<<<ceil_div(mm, 32), dim3(32, 8), 0, s>>>(F, J + jb, J, mm, jb, c->d_Lp_r, c->d_Lp_i,
                                                                               c->ldk_lu, c->d_Lpe, row_exponents(c), c->d_perm);
                        LU_CUDA(cudaGetLastError());
                    }
                    C32 Cv = F.sub(J + jb, J + jb);
                    {
                        // (a CTA per tile: the panels' clusters need SMs that come free beside the rest)
                        BM_PROF(c, "cgemm_tc_kernel (trailing update)");
                        LU_CUDA(gemm_tc_upd(s, c->tm_lu[0], c->tm_lu[1], c->tm_lu[2], c->tm_lu[3], Cv.re, Cv.im, Cv.ld, mm,
                                        nnext, jb, TcScale{c->d_Lpe, c->d_Upe, 0}, INT_MAX, c->d_err));
                    }
                    if (la) {
                        // the rest on s2: interchanges of the columns left of this panel and right of
                        // the next one, their U12 rows (packed from pack row NB on) and their update
                        LU_CUDA(cudaEventRecord(ev_fork, s));
                        LU_CUDA(cudaStreamWaitEvent(s2, ev_fork, 0));
                        LU_CUDA(launch_swap_trsm<V>(s2, F, d_map, 0, J, J + jb + nnext, n, J, jb,
                                                    c->d_Up_r + (long)NB * c->ldk_lu, c->d_Up_i + (long)NB * c->ldk_lu,
                                                    c->ldk_lu, c->d_Upe + NB, row_exponents(c), c->d_perm));
                        if (mm > nnext) {
                            C32 Cr = F.sub(J + jb, J + jb + nnext);
                            LU_CUDA(gemm_tc_upd(s2, c->tm_lu[0], c->tm_lu[1], c->tm_lu[4], c->tm_lu[5], Cr.re, Cr.im, Cr.ld,
                                            mm, mm - nnext, jb, TcScale{c->d_Lpe, c->d_Upe + NB, 0}, INT_MAX,
                                                c->d_err));
                        }
                        LU_CUDA(cudaEventRecord(ev_join, s2));
                    }
                }
            } else {
                BM_PROF(c, "cgemm_simt_kernel (trailing update)");
                LU_CUDA(gemm_any(s, mm, mm, jb, F.sub(J + jb, J), F.sub(J, J + jb), F.sub(J + jb, J + jb)));
            }
        }
    }
    if (la) LU_CUDA(cudaStreamWaitEvent(s, ev_join, 0));
    BM_TRY(finish_t(c, F, s));
    if (la) {  // join the handle's stream
        LU_CUDA(cudaEventRecord(ev_done, s));
        LU_CUDA(cudaStreamWaitEvent(c->stream, ev_done, 0));
    }
    return BM_OK;
}

// one cooperative launch of a persistent triangular solve: as many CTAs as the items, at most the number the
// device keeps resident (queried once per process, device and kernel)
template <class... KArgs, class... Args>
cudaError_t launch_flow(cudaStream_t s, void (*kern)(KArgs...), int threads, int smem, int items, int num_sms,
                        Args... args) {
    cudaError_t e = cudaSuccess;
    if (smem > 0) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> per_sm_cache;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        const std::pair<const void*, int> key{reinterpret_cast<const void*>(kern), dev};
        auto it = per_sm_cache.find(key);
        if (it == per_sm_cache.end()) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
            if (e != cudaSuccess) return e;
            it = per_sm_cache.emplace(key, per_sm).first;
        }
        per_sm = it->second;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(std::max(1, std::min(items, std::max(per_sm, 1) * std::max(num_sms, 1))), 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Solve L U X = Y in place (Y holds P B); Zw is an n x nrhs work buffer.
template <class V>
bm_status getrs_t(bm_ctx* c, V F, V Y, V Zw, int nrhs, const typename V::cv* dinvL, const typename V::cv* dinvU) {
    cudaStream_t s = c->stream;
    const int n = c->n;
    if constexpr (std::is_same<V, C32>::value) {  // factors in G form
        const int items = ceil_div(n, TS_BM) * ceil_div(nrhs, FL_BN);
        if (c->d_flowx == nullptr || 2L * items > c->flow_len) {
            bm_set_error("lu: the triangular solve's exchange buffer is missing");
            return BM_EINVAL;
        }
        // one persistent launch per triangle (block steps and diagonal blocks); a timed-out wait raises the
        // handle's device-wait word, which the refinement loop reads back with every backward error
        // (BM_ETIMEOUT).  (Test hook: with d_info[3] set at assembly, one wait of the forward sweep is on the
        // never-written item after the others.)
        BM_PROF(c, "trsv_flow_kernel");
        float4* const x = reinterpret_cast<float4*>(c->d_flowx);
        LU_CUDA(cudaMemsetAsync(x, 0xff, 2 * items * FLOW_ITEM_BYTES, s));
        const int smem = 2 * FL_TILE * (int)sizeof(float) + 2 * (int)FLOW_ITEM_BYTES;
        LU_CUDA(launch_flow(s, trsv_flow_kernel<false>, FL_T, smem, items, c->num_sms, F, Y, Zw, n, nrhs, dinvL, x,
                            c->d_err, x + c->flow_len * FL_T, c->d_info + 3));
        LU_CUDA(launch_flow(s, trsv_flow_kernel<true>, FL_T, smem, items, c->num_sms, F, Zw, Y, n, nrhs, dinvU,
                            x + (long)items * FL_T, c->d_err, nullptr, c->d_info + 3));
    } else {
        const int items = ceil_div(n, FZ_B) * ceil_div(nrhs, FZ_NC);
        if (c->d_flow == nullptr || 2L * items > c->flow_len) {
            bm_set_error("lu: the triangular solve's flags are missing");
            return BM_EINVAL;
        }
        BM_PROF(c, "trsv_flow_z64_kernel");
        LU_CUDA(cudaMemsetAsync(c->d_flow, 0, (size_t)2 * items * sizeof(int), s));
        LU_CUDA(launch_flow(s, trsv_flow_z64_kernel<false>, 128, 0, items, c->num_sms, F, Y, Zw, n, nrhs, dinvL,
                            c->d_flow, c->d_err));
        LU_CUDA(launch_flow(s, trsv_flow_z64_kernel<true>, 128, 0, items, c->num_sms, F, Zw, Y, n, nrhs, dinvU,
                            c->d_flow + items, c->d_err));
    }
    return BM_OK;
}

}  // namespace

// Panel launch configuration of the handle: the largest cluster the device co-schedules (queried
// once), capped by bm_opts.panel_cluster_max (fewer CTAs put more rows on each thread, which selects
// the narrower sub-panel variants), and the panel kernel bm_opts.panel_kernel selects.
bm_status lu_setup(bm_ctx* c, int cluster_cap, int panel_kernel) {
    // the occupancy query is a property of the device and kernel: asked once per process and device
    static std::mutex mu;
    static std::map<int, int> cache[2];
    int& dev_max = (c->prec == BM_FP64) ? c->panel_cluster_z64 : c->panel_cluster_c32;
    if (dev_max == 0) {
        const int kind = (c->prec == BM_FP64) ? 1 : 0;
        std::lock_guard<std::mutex> lock(mu);
        auto it = cache[kind].find(c->device);
        if (it == cache[kind].end())
            it = cache[kind].emplace(c->device, kind ? query_cluster_max_z64() : query_cluster_max_c32()).first;
        dev_max = it->second;
    }
    c->panel_cluster = dev_max;
    if (cluster_cap >= 1 && cluster_cap <= MAX_CLUSTER) c->panel_cluster = std::min(c->panel_cluster, cluster_cap);
    c->panel_lane_col = panel_kernel == 0;
    // the look-ahead's streams (panel chain at the device's highest priority, the rest of the
    // trailing updates at its lowest) and events, created once per handle
    if (c->prec != BM_FP64 && c->la_hi == nullptr) {
        int least = 0, greatest = 0;
        if (cudaDeviceGetStreamPriorityRange(&least, &greatest) != cudaSuccess ||
            cudaStreamCreateWithPriority(&c->la_hi, cudaStreamNonBlocking, greatest) != cudaSuccess ||
            cudaStreamCreateWithPriority(&c->la_lo, cudaStreamNonBlocking, least) != cudaSuccess) {
            bm_set_error("lu: cannot create the factorisation's streams");
            return BM_ECUDA;
        }
        for (cudaEvent_t& e : c->la_ev)
            if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) {
                bm_set_error("lu: cannot create the factorisation's events");
                return BM_ECUDA;
            }
    }
    return BM_OK;
}

bm_status lu_factor_enqueue(bm_ctx* c) {
    if (c->prec == BM_FP64) {
        Z64 F{c->d_F64, c->ldF};
        return c->lu_fast ? factor_fast_z(c, F) : factor_t<Z64>(c, F, false);
    }
    C32 F{c->d_F32r, c->d_F32i, c->ldF};
    if (c->lu_fast) return factor_fast(c, F);
    return factor_t<C32>(c, F, true);
}

bm_status lu_resume_enqueue(bm_ctx* c, int stop) {
    const int J = (stop >> 1) - 1;
    LU_CUDA(cudaMemsetAsync(c->d_info + 4, 0, sizeof(int), c->stream));
    if (c->prec == BM_FP64) {
        const Z64 F{c->d_F64, c->ldF};
        const int db = std::min(FZ_BLOCK, c->n - J), o = J / FZ_OUTER * FZ_OUTER, oe = std::min(o + FZ_OUTER, c->n);
        if (stop & 1)
            LU_CUDA(launch_lu_restore_z(c->stream, F, J, db, c->n - J - db, reinterpret_cast<double2*>(c->d_fd), c->n));
        // what lies past the outer block still lacks the products of its blocks before this one
        if (J > o && oe < c->n) BM_TRY(update_z(c, F, o, J, oe, nullptr));
        return factor_t<Z64>(c, F, false, J);
    }
    C32 F{c->d_F32r, c->d_F32i, c->ldF};
    const int db = std::min(FD_B, c->n - J);
    if (stop & 1) LU_CUDA(launch_lu_restore(c->stream, F, J, db, c->n - J - db, c->d_fd, c->n));
    return factor_t<C32>(c, F, true, J);
}

size_t lu_fast_bytes(int n) { return fd_work_floats(n) * sizeof(float); }
size_t lu_fast_z_bytes(int n) { return fz_work(n) * sizeof(double2); }

// Y holds P B already (rows gathered with d_perm); solves L U X = Y in place.
bm_status getrs_z64(bm_ctx* c, double2* Y, long ldy, int nrhs) {
    Z64 F{c->d_F64, c->ldF};
    Z64 Yv{Y, ldy};
    Z64 Zv{c->d_Zw64, (long)c->n};
    return getrs_t<Z64>(c, F, Yv, Zv, nrhs, reinterpret_cast<const double2*>(c->d_dinvL),
                        reinterpret_cast<const double2*>(c->d_dinvU));
}

bm_status getrs_c32(bm_ctx* c, float* Yr, float* Yi, long ldy, int nrhs) {
    C32 F{c->d_F32r, c->d_F32i, c->ldF};
    C32 Yv{Yr, Yi, ldy};
    C32 Zv{c->d_Zwr, c->d_Zwi, (long)c->n};
    return getrs_t<C32>(c, F, Yv, Zv, nrhs, reinterpret_cast<const float2*>(c->d_dinvL),
                        reinterpret_cast<const float2*>(c->d_dinvU));
}

cudaError_t launch_gather_rows_z64(cudaStream_t s, const int* perm, int n, int nrhs, const double2* B, long ldb,
                                   double2* Y, long ldy) {
    long total = (long)n * nrhs;
    gather_rows_z64_kernel<<<ceil_div(total, 256), 256, 0, s>>>(perm, n, nrhs, B, ldb, Y, ldy);
    return cudaGetLastError();
}
cudaError_t launch_gather_rows_c32(cudaStream_t s, const int* perm, int n, int nrhs, const float* Br, const float* Bi,
                                   long ldb, float* Yr, float* Yi, long ldy) {
    long total = (long)n * nrhs;
    gather_rows_c32_kernel<<<ceil_div(total, 256), 256, 0, s>>>(perm, n, nrhs, Br, Bi, ldb, Yr, Yi, ldy);
    return cudaGetLastError();
}

size_t swap_map_bytes() { return sizeof(SwapMap); }
