// Refinement residual r = r + alpha A x to FP64-level accuracy on the tensor cores.
//
// Iterative refinement needs the residual b - A x of the FP32 iterate far more accurately than
// FP32 arithmetic gives (the backward-error target is 1e-9 and the iterate is already at ~1e-7),
// and GB300 runs FP64 at ~1.2 TFLOP/s.  The product is therefore formed from exact integer
// products on the bf16 tensor cores (a splitting in the manner of Ozaki et al.):
//   * every row i of A is scaled by a power of two, 2^-e_i, so that its entries (real and imaginary
//     parts) lie in (-1/2, 1/2), and written as seven base-128 digits
//         A_ij 2^-e_i = sum_{d=1..7} a_ij,d 128^-d,   a_ij,d integers in [-64, 64]
//     (exact to 2^-50 of the row's largest entry); every column c of x likewise with 2^-f_c;
//   * each digit is an integer of at most 7 bits, so bf16 holds it exactly and every product of
//     two digits is an exact integer below 2^12;
//   * the pairs (d, d') with d + d' <= 8 are grouped by level l = d + d' - 2 (weight 128^-l), one
//     FP32 accumulator per level in tensor memory.  Over a K chunk of 256 the level sums stay below
//     2^24 (at most 7 pairs x 2 real products per complex term x 256 x 2^12), so every partial sum
//     is an integer that FP32 represents exactly: nothing is rounded inside a chunk, whatever order
//     the hardware adds in;
//   * after each chunk the level sums are added to two 64-bit integers per output, the upper levels and the
//     lower ones, each weighted by its power of 128: nothing is rounded until the end, where the two are
//     added in FP64 (pairs of FP32 per output, the form before, round near 2^-48 in every chunk: errors of FP64
//     solutions were three times as large).  The dropped pairs of one term add up to below 2^-48 (seven
//     digits) or 2^-62 (nine) of the row's and column's scales.
// The x digit tiles sit one after another in shared memory and the levels' accumulators one after
// another in tensor memory, so one MMA multiplies A digit d by all the x digits it pairs with and
// lands each pair in its level.  Seven digits (32 right-hand sides per CTA): four MMAs of width
// 32 (7 - d) per A digit and 16-wide K step, the A-negate bit of the instruction descriptor giving
// -Im A Im x.  Nine digits (16 right-hand sides): the real and imaginary parts of a level share an
// accumulator, [Re | Im], and x is staged as two stacks per digit, [Re x | Im x] for Re A and
// [-Im x | Re x] for Im A, so each A tile is read from shared memory once per K step by two MMAs of width
// 32 (9 - d) instead of four half as wide: the narrow ones left the tensor pipe waiting for A.
// The digits of A are taken from the last to the first: digit d reaches levels d and up, so the next
// chunk's products start on level D - 1 as soon as it has been read while the readers go on with the lower
// levels (reading all of them first left the tensor pipe idle for a third of the time).
//
// CTA: 128 output rows x up to 32 (16) right-hand sides, K range [kbeg, kend) (split K, deterministic
// reduction afterwards when there is more than one split).  Warp 0 issues TMA loads (per 64-wide
// K block: the digit planes of x, then the digit tiles of A one stage at a time), warp 1 issues the
// MMAs, warps 2-9 read the level sums from tensor memory after each chunk (warps 2-5 the real parts,
// 6-9 the imaginary parts, one output row per thread) and keep the running sums.  All waits are
// bounded (2 s); a timeout sets *err and the CTA drains what it issued.
#include "common.cuh"
#include "kernels.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

namespace {

constexpr int RT_BM = 128;   // output rows per CTA
constexpr int RT_BK = 64;    // K elements per stage: bf16 rows of 128 bytes (one swizzle span)
constexpr int RT_TILE_A = RT_BM * RT_BK * 2;  // one digit plane of A: 16 KB
constexpr int RT_THREADS = 320;
constexpr uint64_t RT_WAIT_NS = 2000000000ull;
// D digits per operand (7: pairs to level 6, 2^-50; 9: to level 8, 2^-64) and NT right-hand sides
// per CTA (32 for D = 7, 16 for D = 9).  Level sums over a chunk stay below 2^24: D pairs x 2
// products x 4096 x chunk K, so the chunk is 256 for D = 7 and 192 for D = 9.
template <int D>
struct RtCfg {
    static constexpr bool STACK = D > 7;                // [Re | Im] levels, two x stacks, single-plane A stages
    static constexpr int NT = STACK ? 16 : 32;          // right-hand sides per CTA
    static constexpr int TILE_X = NT * RT_BK * 2;       // one digit plane of x
    static constexpr int KB_CHUNK = STACK ? 3 : 4;      // K blocks of 64 per exact chunk
    static constexpr int X_STACK = 2 * D * TILE_X;      // one stack: all digits, two planes each
    static constexpr int X_BUF = (STACK ? 2 : 1) * X_STACK;
    static constexpr int A_PL = STACK ? 1 : 2;          // A planes per stage
    static constexpr int A_STAGE = A_PL * RT_TILE_A;
    static constexpr int AST = STACK ? 5 : 3;           // A stages
    static constexpr int USES = 2 * D / A_PL;           // stage uses per K block
    static constexpr int LH = D / 2;                    // last of the upper levels
    static constexpr int SMEM = AST * A_STAGE + 2 * X_BUF + 1024 + 256;
    static_assert(2 * D * NT <= 512, "the level accumulators fit tensor memory");
    static_assert(D * NT <= 256, "the widest single MMA has N <= 256");
    static_assert(D * 2 * 4096L * 64 * KB_CHUNK <= (1L << 24), "chunk sums stay exact in FP32");
    // |upper levels' sum| < 2^14 K 128^LH, |lower levels'| < 2^(14 + 1) D K 128^(D - 2 - LH): K below 2^20
    static_assert(14 + 7 * LH + 20 < 63 && 19 + 7 * (D - 2 - LH) + 20 < 63, "the integer sums do not overflow");
    static_assert(SMEM <= 232448, "shared memory");
};

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gtimer() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; false on timeout or when another thread already gave up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (gtimer() - t0 > RT_WAIT_NS) {
            *abort_flag = 1;
            return false;
        }
    }
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "r"(z)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y, int z, int w) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D += A B (acc: a literal 0 or 1) from the low words of the two shared-memory descriptors, issued by the
// lanes with `leader` set.  The operands are warp-uniform, so that they live in uniform registers and a
// product costs a handful of instructions: one thread's issue rate bounds the narrow products otherwise.
__device__ __forceinline__ void mma_bf16(bool leader, uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc,
                                         uint32_t acc) {
    if (leader)
        asm volatile(
            "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %4, 0;\n mov.b64 a, {%1, %5};\n mov.b64 b, {%2, %5};\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n}\n" ::"r"(d),
            "r"(alo), "r"(blo), "r"(idesc), "r"(acc), "n"(DESC_HI)
            : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 consecutive FP32 accumulator columns of this thread's tensor-memory lane
__device__ __forceinline__ void tmem_ld16(uint32_t ta, float* v) {
    uint32_t a[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]),
          "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15])
        : "r"(ta)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(a[i]);
}
// Instruction descriptor, kind::f16: D = F32, A = B = BF16, both K-major, M = 128, N = n.
__device__ constexpr uint32_t idesc_bf16(uint32_t neg_a, uint32_t n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (neg_a << 13) | ((n >> 3) << 17) | ((uint32_t)(RT_BM >> 4) << 24);
}
struct RtProd {
    CUtensorMap tmA;   // the A digit planes (3-D: K, rows, 14 planes)
    CUtensorMap tmX[2];  // the x digit planes: 3-D (K, columns, 14 planes), or the two stacks (4-D)
    const int* eA;     // row exponents of A
    const int* fX;     // column exponents of x
    double2* C;        // output (FP64 complex), C += alpha A x
    long ldc;
    double* Wr;        // split-K workspace (S > 1): S planes of m x n, Re and Im
    double* Wi;
    int m, K, S;       // rows, K, K splits
};
struct RtJob {
    RtProd p[2];
    int nprod, n, ntile_n;  // right-hand sides, column tiles
    double alpha;
    int first_unit[3];
    const int* stop;  // the launch does nothing when this word is not zero
};
__device__ __forceinline__ bool stopped(const int* stop) { return stop != nullptr && *stop != 0; }

template <int D>
__global__ void __launch_bounds__(RT_THREADS, 1) resid_tc_kernel(const __grid_constant__ RtJob J, int* __restrict__ err) {
    using Cfg = RtCfg<D>;
    constexpr int RT_D = D, RT_KB_CHUNK = Cfg::KB_CHUNK, RT_X_BUF = Cfg::X_BUF, RT_AST = Cfg::AST;
    constexpr int RT_NT = Cfg::NT, RT_TILE_X = Cfg::TILE_X, RT_A_STAGE = Cfg::A_STAGE, USES = Cfg::USES;
    constexpr bool STACK = Cfg::STACK;
    if (stopped(J.stop)) return;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;                               // RT_AST stages of digit tiles of A
    uint8_t* sX = smem + RT_AST * RT_A_STAGE;         // 2 buffers of all digit tiles of x
    uint64_t* bars = reinterpret_cast<uint64_t*>(sX + 2 * RT_X_BUF);
    // afull[AST], aempty[AST], xfull[2], xempty[2], accfull, drain, levfree[D]
    const uint32_t afull = su32(bars), aempty = afull + 8 * RT_AST, xfull = aempty + 8 * RT_AST;
    const uint32_t xempty = xfull + 16, accfull = xempty + 16, drain = accfull + 8, levfree = drain + 8;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * RT_AST + 6 + RT_D);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    // ---- work unit: product q, row tile, K split z, column tile ----
    const int q = (int)blockIdx.x >= J.first_unit[1] ? 1 : 0;
    const RtProd& P = J.p[q];
    int u = (int)blockIdx.x - J.first_unit[q];
    const int tn = u % J.ntile_n;
    u /= J.ntile_n;
    const int z = u % P.S, it = u / P.S;
    const int nkb_all = (P.K + RT_BK - 1) / RT_BK;
    const int kb0 = (int)((long)z * nkb_all / P.S), kb1 = (int)((long)(z + 1) * nkb_all / P.S);
    const int nkb = kb1 - kb0;
    const int nchunks = (nkb + RT_KB_CHUNK - 1) / RT_KB_CHUNK;
    const int row0 = it * RT_BM, col0 = tn * RT_NT;
    const int ncols = min(RT_NT, J.n - col0);
    // (the shuffle tells the compiler that the warp index is uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        for (int s = 0; s < RT_AST; ++s) {
            mbar_init(afull + 8 * s, 1);
            mbar_init(aempty + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(xfull + 8 * s, 1);
            mbar_init(xempty + 8 * s, 1);
        }
        mbar_init(accfull, 1);
        mbar_init(drain, 1);
        for (int l = 0; l < RT_D; ++l) mbar_init(levfree + 8 * l, 8);  // the eight reading warps
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int a_issued = 0, x_issued = 0;
        for (int kb = 0; kb < nkb && !*abort_flag; ++kb) {
            const int xb = kb & 1;
            if (kb >= 2 && !mbar_wait(xempty + 8 * xb, (uint32_t)((kb >> 1) - 1) & 1u, abort_flag)) break;
            const int kx = (kb0 + kb) * RT_BK;
            mbar_expect_tx(xfull + 8 * xb, RT_X_BUF);
            uint8_t* xbuf = sX + xb * RT_X_BUF;
            if constexpr (STACK) {
                tma_load_4d(su32(xbuf), &P.tmX[0], xfull + 8 * xb, kx, col0, 0, 0);
                tma_load_4d(su32(xbuf + Cfg::X_STACK), &P.tmX[1], xfull + 8 * xb, kx, col0, 0, 0);
            } else {
                // shared layout: the real-part digit tiles, then the imaginary-part ones
                for (int pl = 0; pl < 2 * RT_D; ++pl)
                    tma_load_3d(su32(xbuf + ((pl & 1) * RT_D + (pl >> 1)) * RT_TILE_X), &P.tmX[0], xfull + 8 * xb, kx,
                                col0, pl);
            }
            x_issued = kb + 1;
            for (int u2 = 0; u2 < USES; ++u2) {
                const int idx = kb * USES + u2, s = idx % RT_AST;
                if (idx >= RT_AST && !mbar_wait(aempty + 8 * s, (uint32_t)(idx / RT_AST - 1) & 1u, abort_flag)) break;
                uint8_t* as = sA + s * RT_A_STAGE;
                mbar_expect_tx(afull + 8 * s, RT_A_STAGE);
                const int d = RT_D - 1 - u2 * Cfg::A_PL / 2;  // from the last digit to the first
                if constexpr (STACK) {
                    tma_load_3d(su32(as), &P.tmA, afull + 8 * s, kx, row0, 2 * d + (u2 & 1));
                } else {
                    tma_load_3d(su32(as), &P.tmA, afull + 8 * s, kx, row0, 2 * d);
                    tma_load_3d(su32(as + RT_TILE_A), &P.tmA, afull + 8 * s, kx, row0, 2 * d + 1);
                }
                a_issued = idx + 1;
            }
        }
        if (*abort_flag) {
            // copies already in flight land before shared memory is released
            for (int idx = (a_issued > RT_AST ? a_issued - RT_AST : 0); idx < a_issued; ++idx) {
                const uint64_t t0 = gtimer();
                while (!mbar_try(afull + 8 * (idx % RT_AST), (uint32_t)(idx / RT_AST) & 1u) && gtimer() - t0 < RT_WAIT_NS) {
                }
            }
            for (int kb = (x_issued > 2 ? x_issued - 2 : 0); kb < x_issued; ++kb) {
                const uint64_t t0 = gtimer();
                while (!mbar_try(xfull + 8 * (kb & 1), (uint32_t)(kb >> 1) & 1u) && gtimer() - t0 < RT_WAIT_NS) {
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (the whole warp walks the loop, lane 0 issues) ----------------
        const bool leader = lane == 0;
        const uint32_t xlo0 = desc_lo(su32(sX)), alo0 = desc_lo(su32(sA));
        bool ok = true;
        int s = 0;             // stage
        uint32_t sph = 0;      // its phase
        for (int kb = 0; kb < nkb && ok; ++kb) {
            const int ch = kb / RT_KB_CHUNK;
            const int xb = kb & 1;
            if (!mbar_wait(xfull + 8 * xb, (uint32_t)(kb >> 1) & 1u, abort_flag)) break;
            fence_after();
            const uint32_t xlo = xlo0 + (uint32_t)xb * (RT_X_BUF >> 4);
            // one K block; FIRST: of a chunk.  The first products of a chunk overwrite level d (and add to
            // the levels above, which the digits before have overwritten), once the readers have taken it
            // out of tensor memory.
            auto block = [&](auto first) {
                constexpr bool FIRST = decltype(first)::value;
#pragma unroll
                for (int u2 = 0; u2 < USES; ++u2) {
                    const int d = RT_D - 1 - u2 * Cfg::A_PL / 2;
                    const bool fresh = FIRST && (!STACK || (u2 & 1) == 0);
                    if ((fresh && ch > 0 && !mbar_wait(levfree + 8 * d, (uint32_t)(ch - 1) & 1u, abort_flag)) ||
                        !mbar_wait(afull + 8 * s, sph, abort_flag)) {
                        ok = false;
                        return;
                    }
                    fence_after();
                    const uint32_t alo = alo0 + (uint32_t)s * (RT_A_STAGE >> 4);
                    if constexpr (STACK) {
                        // x digits 0 .. D - 1 - d (both parts) into levels d .. D - 1
                        const uint32_t blo = xlo + (uint32_t)(u2 & 1) * (Cfg::X_STACK >> 4);
                        const uint32_t Dl = tmem + (uint32_t)(2 * RT_NT * d);
                        const uint32_t n1 = 2 * RT_NT, nw = n1 * (uint32_t)(RT_D - d);
#pragma unroll
                        for (int kk = 0; kk < RT_BK / 16; ++kk) {
                            const uint32_t off = kk * 2;  // 16 bf16 = 32 bytes along K inside the swizzle span
                            const bool over = fresh && kk == 0;
                            if (over || nw > 256) {
                                mma_bf16(leader, Dl, alo + off, blo + off, idesc_bf16(0, n1), over ? 0u : 1u);
                                if (nw > n1)
                                    mma_bf16(leader, Dl + n1, alo + off, blo + (2 * RT_TILE_X >> 4) + off,
                                             idesc_bf16(0, nw - n1), 1u);
                            } else {
                                mma_bf16(leader, Dl, alo + off, blo + off, idesc_bf16(0, nw), 1u);
                            }
                        }
                    } else {
                        const uint32_t ail = alo + (RT_TILE_A >> 4);
                        const uint32_t nw = (uint32_t)(RT_NT * (RT_D - d));
                        const uint32_t idp = idesc_bf16(0, nw), idn = idesc_bf16(1, nw);
                        const uint32_t Dr = tmem + (uint32_t)(d * RT_NT), Di = Dr + RT_D * RT_NT;
                        const uint32_t xr = xlo, xi = xlo + (RT_D * RT_TILE_X >> 4);
#pragma unroll
                        for (int kk = 0; kk < RT_BK / 16; ++kk) {
                            const uint32_t off = kk * 2;
                            if (fresh && kk == 0) {
                                const uint32_t id1 = idesc_bf16(0, RT_NT), idw = idesc_bf16(0, nw - RT_NT);
                                mma_bf16(leader, Dr, alo, xr, id1, 0u);
                                mma_bf16(leader, Di, alo, xi, id1, 0u);
                                if (nw > RT_NT) {
                                    mma_bf16(leader, Dr + RT_NT, alo, xr + (RT_TILE_X >> 4), idw, 1u);
                                    mma_bf16(leader, Di + RT_NT, alo, xi + (RT_TILE_X >> 4), idw, 1u);
                                }
                            } else {
                                mma_bf16(leader, Dr, alo + off, xr + off, idp, 1u);
                                mma_bf16(leader, Di, alo + off, xi + off, idp, 1u);
                            }
                            mma_bf16(leader, Dr, ail + off, xi + off, idn, 1u);
                            mma_bf16(leader, Di, ail + off, xr + off, idp, 1u);
                        }
                    }
                    if (leader) mma_commit(aempty + 8 * s);
                    if (++s == RT_AST) {
                        s = 0;
                        sph ^= 1u;
                    }
                }
            };
            if (kb % RT_KB_CHUNK == 0)
                block(std::true_type{});
            else
                block(std::false_type{});
            if (!ok) break;
            if (leader) {
                mma_commit(xempty + 8 * xb);
                if ((kb % RT_KB_CHUNK) == RT_KB_CHUNK - 1 || kb == nkb - 1) mma_commit(accfull);
            }
        }
        if (*abort_flag && leader) {
            // products already issued finish before tensor memory and shared memory are released
            mma_commit(drain);
            const uint64_t t0 = gtimer();
            while (!mbar_try(drain, 0u) && gtimer() - t0 < RT_WAIT_NS) {
            }
        }
        __syncwarp();
    } else if (warp >= 2) {
        // ---------------- level-sum readers: warps 2-5 real parts, 6-9 imaginary parts ----------------
        const int qw = warp & 3;  // tensor-memory lane quarter this warp may read
        const int part = warp >= 6 ? 1 : 0;
        const uint32_t lane_off = (uint32_t)(qw * 32) << 16;
        long long hi[RT_NT], lo[RT_NT];  // running sums of this row's outputs: levels up to LH, and past it
#pragma unroll
        for (int j = 0; j < RT_NT; ++j) hi[j] = lo[j] = 0;
        // level lev of every output times w onto acc, then released to the next chunk's products
        auto add_level = [&](long long (&acc)[RT_NT], int lev, int w) {
#pragma unroll
            for (int g = 0; g < RT_NT / 16; ++g) {
                float v[16];
                tmem_ld16(tmem + lane_off + (uint32_t)(STACK ? 2 * RT_NT * lev + RT_NT * part + g * 16
                                                             : part * RT_D * RT_NT + lev * RT_NT + g * 16), v);
                if (g == RT_NT / 16 - 1) {
                    fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(levfree + 8 * lev);
                }
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[g * 16 + j] += (long long)__float2int_rn(v[j]) * w;
            }
        };
        for (int ch = 0; ch < nchunks; ++ch) {
            if (!mbar_wait(accfull, (uint32_t)ch & 1u, abort_flag)) break;
            fence_after();
            // (the last level first: the order in which the next chunk's products need them)
#pragma unroll 1
            for (int lev = RT_D - 1; lev > Cfg::LH; --lev) add_level(lo, lev, 1 << (7 * (RT_D - 1 - lev)));
#pragma unroll 1
            for (int lev = Cfg::LH; lev >= 0; --lev) add_level(hi, lev, 1 << (7 * (Cfg::LH - lev)));
        }
        if (!*abort_flag) {
            const int row = row0 + qw * 32 + lane;
            if (row < P.m) {
                // value = 128^-2 2^(e_row + f_col) (hi 128^-LH + lo 128^-(D - 1))  (digits carry 128^-d each)
                constexpr int EH = -14 - 7 * Cfg::LH;
                constexpr double LO = 1.0 / (double)(1ll << (7 * (RT_D - 1 - Cfg::LH)));
                const int er = P.eA[row];
#pragma unroll
                for (int j = 0; j < RT_NT; ++j) {
                    if (j >= ncols) break;
                    const int col = col0 + j;
                    const int fc = P.fX[col];
                    const double v = er == RT_NONFINITE || fc == RT_NONFINITE
                                         ? __longlong_as_double(0x7FF8000000000000ll)
                                         : ldexp(fma((double)lo[j], LO, (double)hi[j]), er + fc + EH);
                    if (P.S == 1) {
                        double* o = reinterpret_cast<double*>(P.C + row + (long)col * P.ldc) + part;
                        *o += J.alpha * v;
                    } else {
                        double* W = part ? P.Wi : P.Wr;
                        W[((long)z * J.n + col) * P.m + row] = v;
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
    if (threadIdx.x == 0 && *abort_flag) atomicExch(err, 1);
}

// C += alpha sum_z W[z]  (z in order; W: S planes of n columns of m rows, Re and Im)
__global__ void rt_reduce_kernel(const double* __restrict__ Wr, const double* __restrict__ Wi, int S, int m, int n,
                                 double alpha, double2* __restrict__ C, long ldc, const int* stop) {
    if (stopped(stop)) return;
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long zs = (long)m * n;
    if (idx >= zs) return;
    const int j = (int)(idx / m), i = (int)(idx % m);
    double re = 0.0, im = 0.0;
    for (int z = 0; z < S; ++z) {
        re += Wr[idx + z * zs];
        im += Wi[idx + z * zs];
    }
    double2& c = C[i + (long)j * ldc];
    c.x += alpha * re;
    c.y += alpha * im;
}

// Row maxima of A (rows x K, column-major FP64 complex) over max(|Re|, |Im|): each thread a row and
// 256 columns, combined by an atomic maximum on the bit patterns (non-negative doubles order as
// their bits).  mx must start at zero.
__global__ void row_max_kernel(const double2* __restrict__ A, long lda, int rows, int K,
                               unsigned long long* __restrict__ mx, RtShift sh, const int* stop) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows || stopped(stop)) return;
    const int j0 = blockIdx.y * 256, j1 = min(K, j0 + 256);
    // (integer maxima: FP64 compares run on the narrow FP64 pipe)
    unsigned long long m = 0;
    auto take = [&](double2 v, int j) { m = max(m, scaled_mag(max(mag_bits(v.x), mag_bits(v.y)), -sh.at(j))); };
    const double2* a = A + i;
    int j = j0;
    for (; j + 8 <= j1; j += 8) {
        double2 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = a[(long)(j + u) * lda];
#pragma unroll
        for (int u = 0; u < 8; ++u) take(v[u], j + u);
    }
    for (; j < j1; ++j) take(a[(long)j * lda], j);
    atomicMax(mx + i, m);
}
// e_i with max_j max(|Re|, |Im|) < 2^(e_i - 1) (0 for a zero row)
__global__ void row_exponent_kernel(const unsigned long long* __restrict__ mx, int rows, int* __restrict__ e) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= rows) return;
    e[i] = row_exponent(mx[i]);
}

// The ND base-128 digits of v 2^-ex (|v 2^-ex| < 1/2), each an integer in [-64, 64]: v 2^(7 ND - ex) rounded
// to the nearest integer M (|M| <= 2^(7 ND - 1)), written as M = sum_d a_d 128^(ND - 1 - d) with balanced
// digits in [-64, 63] but for the most significant one (which may be +64).  M + sum_d 64 128^d has the digits
// a_d + 64, so they are plain 7-bit fields without carries; digit_word returns that sum.
// Integer arithmetic on the FP64 bit pattern only (FP64 arithmetic and conversions are slow here).
template <int ND>
__device__ __forceinline__ unsigned long long digit_word(double v, int ex) {
    constexpr unsigned long long BIAS = 64ull * (((1ull << (7 * ND - 7)) - 1) / 127 + (1ull << (7 * ND - 7)));
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int E = (int)((bits >> 52) & 0x7FF);
    unsigned long long M = 0;
    // zero and subnormals (below any row scale used here) give zero digits; so does a value that does not fit
    // its scale (only in a row or column with a non-finite entry, whose outputs are NaN: RT_NONFINITE)
    if (E != 0 && E != 0x7FF) {
        const unsigned long long mant = (bits & 0xFFFFFFFFFFFFFull) | (1ull << 52);
        const int sh = E - 1075 + 7 * ND - ex;  // v 2^(7 ND - ex) = mant 2^sh, mant in [2^52, 2^53)
        if (sh > 7 * ND - 54)                   // |v 2^-ex| >= 1/2: does not fit the scale
            M = 0;
        else if (sh >= 0)
            M = mant << sh;
        else if (sh > -62)
            M = (mant + (1ull << (-sh - 1))) >> (-sh);  // round half up
        if (bits >> 63) M = 0ull - M;
    }
    return M + BIAS;
}
// Digit d (most significant first) as a float: the field's bits in the last places of 1.5 2^23, so that no
// conversion instruction is needed; its upper half is the digit's bf16 (at most 8 significant bits).
constexpr float DIGIT_ONE = 12582912.f;
template <int ND>
__device__ __forceinline__ float digit_raw(unsigned long long w, int d) {
    const unsigned u = (unsigned)(w >> (7 * (ND - 1 - d)));
    return __uint_as_float(0x4B400000u | (d == 0 ? u & 255u : u & 127u));
}
// the bf16 of two floats that bf16 holds exactly, the first in the lower half
__device__ __forceinline__ unsigned bf16_pair(float a, float b) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
}

// Digit planes of A: plane 2d + part holds digit d of the real (part 0) or imaginary (1) parts, K-major
// ([row][ldk]); through a 32-row x 64-column shared tile so that both sides are coalesced, a lane taking two
// columns and writing 4 bytes per plane.  Integer work bounded it when each digit was peeled off with its
// carry and built bit by bit: N = 4096, both operators, 1.39 -> 0.65 ms (3.5 GB read and written: 5.3 TB/s).
template <int ND>
__global__ void __launch_bounds__(256) digits_a_kernel(const double2* __restrict__ A, long lda, int rows, int K,
                                                       const int* __restrict__ e, unsigned* __restrict__ D, long ldk,
                                                       long plane, RtShift sh, const int* stop) {
    if (stopped(stop)) return;
    __shared__ double2 t[32][65];
    const int k0 = blockIdx.x * 64, r0 = blockIdx.y * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int q = ty; q < 64; q += 8) {
        const int r = r0 + tx, k = k0 + q;
        t[tx][q] = (r < rows && k < K) ? A[r + (long)k * lda] : make_double2(0.0, 0.0);
    }
    __syncthreads();
    const int k = k0 + 2 * tx;
    if (k >= K) return;
    const int sa = sh.at(k), sb = sh.at(k + 1);
#pragma unroll 1
    for (int q = ty; q < 32; q += 8) {
        const int r = r0 + q;
        if (r >= rows) return;
        const double2 a = t[q][2 * tx], b = t[q][2 * tx + 1];  // (zero past K)
        const int ex = e[r];
        unsigned* o = D + ((long)r * ldk + k) / 2;
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const unsigned long long wa = digit_word<ND>(part ? a.y : a.x, ex + sa),
                                     wb = digit_word<ND>(part ? b.y : b.x, ex + sb);
#pragma unroll
            for (int d = 0; d < ND; ++d)
                o[(2 * d + part) * (plane / 2)] =
                    bf16_pair(digit_raw<ND>(wa, d) - (DIGIT_ONE + 64.f), digit_raw<ND>(wb, d) - (DIGIT_ONE + 64.f));
        }
    }
}

// Column exponents of x over rows [r0, r0 + K) for the n columns (one block per column).
__global__ void col_exponent_kernel(const double2* __restrict__ X, long ldx, int r0, int K, int* __restrict__ f,
                                    RtShift sh, const int* stop) {
    if (stopped(stop)) return;
    const int c = blockIdx.x;
    unsigned long long mx = 0;
    for (int i = threadIdx.x; i < K; i += blockDim.x) {
        const double2 v = X[r0 + i + (long)c * ldx];
        mx = max(mx, scaled_mag(max(mag_bits(v.x), mag_bits(v.y)), sh.at(i)));
    }
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __shared__ unsigned long long sm[32];
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, sm[w]);
        f[c] = row_exponent(mx);
    }
}

// Digit planes of x rows [r0, r0 + K) (columns c < n; columns up to npad are zero), layout [col][ldk]:
// plane 2 d + part, or (nine digits: stacks) planes 3 d .. 3 d + 2 = -Im, Re, Im.  A thread takes two rows.
template <int ND>
__global__ void digits_x_kernel(const double2* __restrict__ X, long ldx, int r0, int K, int n, int npad,
                                const int* __restrict__ f, unsigned* __restrict__ D, long ldk, long plane,
                                RtShift sh, const int* stop) {
    if (stopped(stop)) return;
    constexpr bool STACK = ND > 7;
    const int Kp = (K + 1) / 2;
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (long)npad * Kp) return;
    const int c = (int)(idx / Kp), k = 2 * (int)(idx % Kp);
    unsigned* o = D + ((long)c * ldk + k) / 2;
    const long pl = plane / 2;
    if (c >= n) {
        for (int p = 0; p < (STACK ? 3 : 2) * ND; ++p) o[p * pl] = 0u;
        return;
    }
    const double2* x = X + r0 + k + (long)c * ldx;
    const double2 a = x[0], b = k + 1 < K ? x[1] : make_double2(0.0, 0.0);
    const int ea = f[c] - sh.at(k), eb = f[c] - sh.at(k + 1);
    constexpr float Z = DIGIT_ONE + 64.f;
    const unsigned long long ra = digit_word<ND>(a.x, ea), rb = digit_word<ND>(b.x, eb);
    const unsigned long long ia = digit_word<ND>(STACK ? -a.y : a.y, ea), ib = digit_word<ND>(STACK ? -b.y : b.y, eb);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const float va = digit_raw<ND>(ia, d), vb = digit_raw<ND>(ib, d);
        const unsigned re = bf16_pair(digit_raw<ND>(ra, d) - Z, digit_raw<ND>(rb, d) - Z);
        if (STACK) {
            o[3 * d * pl] = bf16_pair(va - Z, vb - Z);
            o[(3 * d + 1) * pl] = re;
            o[(3 * d + 2) * pl] = bf16_pair(Z - va, Z - vb);
        } else {
            o[2 * d * pl] = re;
            o[(2 * d + 1) * pl] = bf16_pair(va - Z, vb - Z);
        }
    }
}

PFN_cuTensorMapEncodeTiled_v12000 rt_encode() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (fn == nullptr) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

}  // namespace

// 3-D tensor map over 14 bf16 digit planes, each [rows][ldk] (K-major): dims {K, rows, 14},
// box {64, box_rows, 1}, 128-byte swizzle; reads outside {K, rows} return zeros.
bm_status rt_make_map(void* tmap, const void* base, long rows, long K, long ldk, long plane_elems, int box_rows,
                      int nd) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = rt_encode();
    if (enc == nullptr) {
        bm_set_error("cuTensorMapEncodeTiled is unavailable from the driver");
        return BM_ECUDA;
    }
    if ((reinterpret_cast<uintptr_t>(base) & 15) != 0 || (ldk * 2) % 16 != 0 || (plane_elems * 2) % 16 != 0) {
        bm_set_error("digit-plane tensor map: base or stride not 16-byte aligned");
        return BM_EINVAL;
    }
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)(2 * nd)};
    cuuint64_t strides[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)plane_elems * 2};
    cuuint32_t box[3] = {(cuuint32_t)RT_BK, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = enc(reinterpret_cast<CUtensorMap*>(tmap), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base),
                     dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        bm_set_error("cuTensorMapEncodeTiled (digit planes) failed with code " + std::to_string((int)r));
        return BM_ECUDA;
    }
    return BM_OK;
}

// Tensor maps of the x digit planes (two blobs): the 3-D map of seven digits, or the two stacks of nine,
// [Re | Im] and [-Im | Re] per digit (4-D: K, columns, two consecutive planes, digits three planes apart).
bm_status rt_make_map_x(void* tmaps, const void* base, long cols, long K, long ldk, int nd) {
    const long plane = cols * ldk;
    if (nd <= 7) return rt_make_map(tmaps, base, cols, K, ldk, plane, rt_col_tile(nd), nd);
    PFN_cuTensorMapEncodeTiled_v12000 enc = rt_encode();
    if (enc == nullptr) {
        bm_set_error("cuTensorMapEncodeTiled is unavailable from the driver");
        return BM_ECUDA;
    }
    if ((reinterpret_cast<uintptr_t>(base) & 15) != 0 || (ldk * 2) % 16 != 0) {
        bm_set_error("digit-plane tensor map: base or stride not 16-byte aligned");
        return BM_EINVAL;
    }
    for (int q = 0; q < 2; ++q) {
        cuuint64_t dims[4] = {(cuuint64_t)K, (cuuint64_t)cols, 2, (cuuint64_t)nd};
        cuuint64_t strides[3] = {(cuuint64_t)ldk * 2, (cuuint64_t)plane * 2, (cuuint64_t)plane * 6};
        cuuint32_t box[4] = {(cuuint32_t)RT_BK, (cuuint32_t)rt_col_tile(nd), 2, (cuuint32_t)nd};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        // q = 0: planes Re, Im of each digit; q = 1: planes -Im, Re
        unsigned char* from = const_cast<unsigned char*>(static_cast<const unsigned char*>(base)) + (q == 0 ? plane * 2 : 0);
        CUresult r = enc(reinterpret_cast<CUtensorMap*>(static_cast<unsigned char*>(tmaps) + 128 * q),
                         CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, from, dims, strides, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            bm_set_error("cuTensorMapEncodeTiled (digit stacks) failed with code " + std::to_string((int)r));
            return BM_ECUDA;
        }
    }
    return BM_OK;
}

long rt_ldk(long K) { return (K + RT_BK - 1) / RT_BK * RT_BK; }
int rt_digit_planes(int nd) { return 2 * nd; }
int rt_x_planes(int nd) { return nd <= 7 ? 2 * nd : 3 * nd; }
int rt_col_tile(int nd) { return nd <= 7 ? RtCfg<7>::NT : RtCfg<9>::NT; }

// Row exponents (unless rowmax is null: they are there) and digit planes of A.
cudaError_t launch_digits_a(cudaStream_t s, const double2* A, long lda, int rows, int K, int* e, void* D, long ldk,
                            void* rowmax, int nd, RtShift sh, const int* stop) {
    if (rows <= 0 || K <= 0) return cudaSuccess;
    unsigned long long* mx = reinterpret_cast<unsigned long long*>(rowmax);
    if (mx != nullptr) {
        cudaError_t err = cudaMemsetAsync(mx, 0, (size_t)rows * 8, s);
        if (err != cudaSuccess) return err;
        row_max_kernel<<<dim3(ceil_div(rows, 128), ceil_div(K, 256)), 128, 0, s>>>(A, lda, rows, K, mx, sh, stop);
        row_exponent_kernel<<<ceil_div(rows, 128), 128, 0, s>>>(mx, rows, e);
    }
    const dim3 grid(ceil_div(K, 64), ceil_div(rows, 32));
    auto kern = nd <= 7 ? digits_a_kernel<7> : digits_a_kernel<9>;
    kern<<<grid, 256, 0, s>>>(A, lda, rows, K, e, reinterpret_cast<unsigned*>(D), ldk, (long)rows * ldk, sh, stop);
    return cudaGetLastError();
}

cudaError_t launch_digits_x(cudaStream_t s, const double2* X, long ldx, int r0, int K, int n, int npad, int* f,
                            void* D, long ldk, long plane, int nd, RtShift sh, const int* stop) {
    if (n <= 0 || K <= 0) return cudaSuccess;
    col_exponent_kernel<<<n, 256, 0, s>>>(X, ldx, r0, K, f, sh, stop);
    const long t = (long)npad * ((K + 1) / 2);
    auto kern = nd <= 7 ? digits_x_kernel<7> : digits_x_kernel<9>;
    kern<<<ceil_div(t, 256L), 256, 0, s>>>(X, ldx, r0, K, n, npad, f, reinterpret_cast<unsigned*>(D), ldk, plane, sh,
                                           stop);
    return cudaGetLastError();
}

// K splits of the products of one residual launch.  A CTA holds a whole SM (its shared memory
// and all 512 tensor-memory columns), so the launch aims at one CTA per SM: every CTA covers
// ceil(work / SMs) K blocks of 64, at least 4 (the set-up and the x digit loads amortised) and at
// most 32, where work counts the K blocks of every row and column tile of the launch.  Large
// systems land on 32 (N = 4096: two and four splits); small ones split further, so that, e.g., a
// 1024-point mixed system with 16 right-hand sides runs 128 CTAs instead of 24.  Every split keeps
// at least one K block (S <= K blocks).
void rt_plan_splits(int nprod, const long* m, const long* K, int n, int nd, int num_sms, int* S) {
    auto cdiv = [](long a, long b) { return (a + b - 1) / b; };
    const long ntn = cdiv(n, rt_col_tile(nd));
    long work = 0;
    for (int q = 0; q < nprod; ++q) work += cdiv(m[q], RT_BM) * ntn * cdiv(K[q], RT_BK);
    const long per = std::min(32L, std::max(4L, cdiv(work, std::max(num_sms, 1))));
    for (int q = 0; q < nprod; ++q) {
        const long kb = cdiv(K[q], RT_BK);
        S[q] = (int)std::max(1L, std::min(std::min(16L, kb), cdiv(kb, per)));
    }
}

// The products of one residual (at most two, sharing n and alpha): C += alpha A x each.  A product
// with S > 1 K splits writes S m n doubles (Re and Im) to its workspace, reduced in order afterwards.
cudaError_t gemm_rt(cudaStream_t s, const RtArgs* prods, int nprod, int n, double alpha, int* d_err, int* launched,
                    int nd, const int* stop) {
    if (nprod < 1 || nprod > 2 || n <= 0 || (nd != 7 && nd != 9)) return cudaSuccess;
    static DeviceFlags attr7, attr9;
    if (nd == 7 && attr7.pending()) {
        cudaError_t e = cudaFuncSetAttribute(resid_tc_kernel<7>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             RtCfg<7>::SMEM);
        if (e != cudaSuccess) return e;
        attr7.done();
    }
    if (nd == 9 && attr9.pending()) {
        cudaError_t e = cudaFuncSetAttribute(resid_tc_kernel<9>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             RtCfg<9>::SMEM);
        if (e != cudaSuccess) return e;
        attr9.done();
    }
    RtJob J{};
    J.nprod = nprod;
    J.n = n;
    J.ntile_n = ceil_div(n, rt_col_tile(nd));
    J.alpha = alpha;
    J.stop = stop;
    int u = 0;
    for (int q = 0; q < 2; ++q) {
        J.first_unit[q] = u;
        if (q < nprod) {
            const RtArgs& a = prods[q];
            RtProd& p = J.p[q];
            std::memcpy(&p.tmA, a.tmA, sizeof(CUtensorMap));
            std::memcpy(p.tmX, a.tmX, (nd <= 7 ? 1 : 2) * sizeof(CUtensorMap));
            p.eA = a.eA;
            p.fX = a.fX;
            p.C = a.C;
            p.ldc = a.ldc;
            p.Wr = a.Wr;
            p.Wi = a.Wi;
            p.m = a.m;
            p.K = a.K;
            p.S = a.S;
            if (a.m > 0 && a.K > 0) u += ceil_div(a.m, RT_BM) * a.S * J.ntile_n;
        }
    }
    J.first_unit[2] = u;
    if (nprod == 1) J.first_unit[1] = u;
    if (u == 0) return cudaSuccess;
    if (nd == 7)
        resid_tc_kernel<7><<<u, RT_THREADS, RtCfg<7>::SMEM, s>>>(J, d_err);
    else
        resid_tc_kernel<9><<<u, RT_THREADS, RtCfg<9>::SMEM, s>>>(J, d_err);
    *launched += 1;
    for (int q = 0; q < nprod; ++q) {
        const RtArgs& a = prods[q];
        if (a.S > 1 && a.m > 0 && a.K > 0) {
            const long t = (long)a.m * n;
            rt_reduce_kernel<<<ceil_div(t, 256L), 256, 0, s>>>(a.Wr, a.Wi, a.S, a.m, n, alpha, a.C, a.ldc, stop);
            *launched += 1;
        }
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// FP64 products C += alpha A B (column-major, C initialised) from nine-digit products: the Schur
// complement and the trailing updates of the FP64 precision.  A product of two entries is good to about 2^-61 of
// the scales of its row of A and column of B (the last digits, and the dropped pairs), its sum over K is exact and
// rounded once.  The scales have to fit the entries that matter: the Schur complement's blocks are balanced
// (balance_kernel), the LU's columns and rows scaled against each other (inner_exponent).  Solution errors against extended
// precision over N = 256 .. 1024, four curves: 0.29 times those with FP64 multiply-adds (geometric mean; 0.64 at
// most).  N = 1000 Schur complement 14.0 -> 0.9 ms; the FP64 pipe runs 304 multiply-adds a cycle on the whole chip.
// The operands' digit planes are made per call in the workspace, in chunks of rows and columns when it
// does not hold them all.
// ------------------------------------------------------------------------------------------------
namespace {
constexpr int DG_ND = 9;
struct DgPlan {
    int mr, nc;       // rows and columns per chunk
    size_t a, x, w;   // bytes: A planes with exponents and row maxima, X planes with exponents, K-split sums
};
size_t al256(size_t v) { return (v + 255) / 256 * 256; }
size_t dg_a_bytes(int mr, int K) { return al256((size_t)2 * DG_ND * mr * rt_ldk(K) * 2) + al256((size_t)mr * 4) + al256((size_t)mr * 8); }
size_t dg_x_bytes(int nc, int K) { return al256((size_t)rt_x_planes(DG_ND) * nc * rt_ldk(K) * 2) + al256((size_t)nc * 4); }
DgPlan dg_plan(int m, int n, int K, int num_sms) {
    constexpr size_t CAP = (size_t)512 << 20;  // per operand
    DgPlan p{};
    const int nt = rt_col_tile(DG_ND);
    const long ar = (long)(CAP / ((size_t)4 * DG_ND * rt_ldk(K))) / RT_BM * RT_BM;
    const long xc = (long)(CAP / ((size_t)2 * rt_x_planes(DG_ND) * rt_ldk(K))) / nt * nt;
    p.mr = (int)std::min<long>(m, std::max<long>(ar, RT_BM));
    p.nc = (int)std::min<long>(ceil_div(n, nt) * (long)nt, std::max<long>(xc, nt));
    p.a = dg_a_bytes(p.mr, K);
    p.x = dg_x_bytes(p.nc, K);
    const long mq = p.mr, kq = K;
    int S = 1;
    rt_plan_splits(1, &mq, &kq, std::min(p.nc, n), DG_ND, num_sms, &S);
    p.w = S > 1 ? al256((size_t)2 * S * p.mr * std::min(p.nc, n) * 8) : 0;
    return p;
}
}  // namespace

// Workspace one product needs, and whether it is worth it: below about 60 us of FP64 multiply-adds the
// digit conversions cost more than they save.
size_t dg_bytes(int m, int n, int K, int num_sms) {
    if ((double)m * n * K < 9e6) return 0;
    const DgPlan p = dg_plan(m, n, K, num_sms);
    return p.a + p.x + p.w;
}

bm_status gemm_z64_dg(cudaStream_t s, void* work, int num_sms, int m, int n, int K, double alpha, Z64 A, Z64 B, Z64 C,
                      int* d_err, int* eA, RtShift sh, const int* stop) {
    const DgPlan p = dg_plan(m, n, K, num_sms);
    const int nt = rt_col_tile(DG_ND);
    const long ldk = rt_ldk(K);
    unsigned char* w = static_cast<unsigned char*>(work);
    void* ap = w;
    int* ea = reinterpret_cast<int*>(w + al256((size_t)2 * DG_ND * p.mr * ldk * 2));
    void* rmax = reinterpret_cast<unsigned char*>(ea) + al256((size_t)p.mr * 4);
    unsigned char* xp = w + p.a;
    int* fx = reinterpret_cast<int*>(xp + al256((size_t)rt_x_planes(DG_ND) * p.nc * ldk * 2));
    double* ws = reinterpret_cast<double*>(xp + p.x);
    alignas(64) unsigned char tma[128], tmx[256];
    BM_TRY(rt_make_map_x(tmx, xp, p.nc, K, ldk, DG_ND));
    for (int i0 = 0; i0 < m; i0 += p.mr) {
        const int mr = std::min(p.mr, m - i0);
        int* const er = eA != nullptr ? eA + i0 : ea;
        BM_CUDA_TRY(launch_digits_a(s, A.p + i0, A.ld, mr, K, er, ap, ldk, eA != nullptr ? nullptr : rmax, DG_ND, sh, stop));
        BM_TRY(rt_make_map(tma, ap, mr, K, ldk, (long)mr * ldk, RT_BM, DG_ND));
        for (int j0 = 0; j0 < n; j0 += p.nc) {
            const int nc = std::min(p.nc, n - j0);
            BM_CUDA_TRY(launch_digits_x(s, B.p + (long)j0 * B.ld, B.ld, 0, K, nc, ceil_div(nc, nt) * nt, fx, xp, ldk,
                                        (long)p.nc * ldk, DG_ND, sh, stop));
            const long mq = mr, kq = K;
            int S = 1, nl = 0;
            rt_plan_splits(1, &mq, &kq, nc, DG_ND, num_sms, &S);
            while (S > 1 && (size_t)2 * S * mr * nc * 8 > p.w) --S;
            RtArgs a{tma, tmx, er, fx, C.p + i0 + (long)j0 * C.ld, C.ld, nullptr, nullptr, mr, K, S};
            if (S > 1) {
                a.Wr = ws;
                a.Wi = ws + (size_t)S * mr * nc;
            }
            BM_CUDA_TRY(gemm_rt(s, &a, 1, nc, alpha, d_err, &nl, DG_ND, stop));
        }
    }
    return BM_OK;
}
