// Complex GEMM on the 5th-generation tensor cores (sm_103a): C = beta C + alpha A B^T with
// A (m x K) and B (n x K) given as K-major planar packs.  This is the contraction of Theorem thm:LU
// (U33 = -[M31 M32][M13; M23]), of every LU trailing update A22 -= L21 U12 and of the skinny products of
// the solve.
//
// Operand split: every entry is an FP32 value scaled by a power of two of its row (A) or of its column
// (rows of B) to below 2^15, and held as two FP16 numbers hi + lo (11 + 11 significant bits; entries below
// 2^-18 of their row's largest keep 2^-40 of that one).  The product is A_hi B_hi + A_hi B_lo + A_lo B_hi,
// the terms and significands of a 3xTF32 product, at twice its rate and from a third of its bytes: hi
// and lo of 32 consecutive K are adjacent, [32 hi | 32 lo], one 128-byte shared row, so each is loaded
// once for the three products.  Exponents: TcScale.  Schur complement N = 4096 (per-launch times):
// 3.50 -> 1.58 ms against the same kernel on three-segment TF32 packs.
//
// Complex product with planar operands and one accumulator [Dr | Di] (128 lanes x 256 columns of TMEM):
//     [Dr | Di] += Ar [Br; Bi]^T,  Dr -= Ai Bi^T,  Di += Ai Br^T
// The real and imaginary tiles of B lie one after another in shared memory, so the first is one MMA of
// width 256 (a narrower MMA reads A again: shared-memory bandwidth bounds 128 x 128 FP16 products); the
// minus sign is the A-negate bit of the instruction descriptor.
//
// CTA tile 128 x 128, 32 K elements per stage (64 KB), 3-stage TMA -> shared-memory pipeline with
// mbarriers.  Warp 0 lane 0 issues TMA loads, warp 1 the tcgen05.mma (the whole warp walks the loop so
// that the operands live in uniform registers, lane 0 issues); all four warps
// then read the accumulators (tcgen05.ld 32x32b, warp w owns TMEM lanes 32(w mod 4) .. +31 = rows)
// and update C with coalesced column-major stores; the LU trailing updates have a persistent form
// (cgemm_tc_upd_kernel).  Every mbarrier wait is bounded (2 s by the global timer); a timeout
// sets *err, skips the epilogue, waits for issued copies and products and frees TMEM.  err[1] is
// a test hook: when it is set the MMA warp first waits on a barrier that nothing completes, gives
// up after 1 ms and takes that timeout path without issuing any product.
#include "common.cuh"
#include "kernels.cuh"
#include "tc_pack.cuh"

#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <vector>

namespace {

constexpr int BM = TC_BM, BN = TC_BN;
constexpr int BKE = 32;  // K elements per stage: 32 hi and 32 lo halves, a 128-byte row (one swizzle span)
constexpr int STAGES = 3;
constexpr int TILE_A = BM * 2 * BKE * 2;
constexpr int TILE_B = BN * 2 * BKE * 2;
constexpr int STAGE_BYTES = 2 * TILE_A + 2 * TILE_B;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr uint32_t TMEM_COLS = 2 * BN;  // Dr, Di
constexpr uint64_t WAIT_NS = 2000000000ull;
constexpr uint64_t TEST_WAIT_NS = 1000000ull;  // the test hook's wait limit

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups 1024 bytes apart.
constexpr uint32_t DESC_HI = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

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
// bounded wait; returns false on timeout or when another thread already gave up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
    if (mbar_try(bar, parity)) return true;
    const uint64_t t0 = gtimer();
    while (true) {
        if (mbar_try(bar, parity)) return true;
        if (*abort_flag) return false;
        if (gtimer() - t0 > WAIT_NS) {
            *abort_flag = 1;
            return false;
        }
    }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, uint32_t bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar), "r"(x), "r"(y)
        : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (+)= A B from the low words of the two shared-memory descriptors, issued by the lanes with `leader` set;
// the operands are warp-uniform.
__device__ __forceinline__ void mma_f16(bool leader, uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc,
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

// 16 consecutive fp32 accumulator columns of this thread's TMEM lane, of two accumulators (real
// and imaginary part), one wait for both
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, float* va, float* vb) {
    uint32_t a[16], b[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, "
        "[%33];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(a[8]),
          "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]), "=r"(a[14]), "=r"(a[15]), "=r"(b[0]),
          "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]),
          "=r"(b[10]), "=r"(b[11]), "=r"(b[12]), "=r"(b[13]), "=r"(b[14]), "=r"(b[15])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        va[i] = __uint_as_float(a[i]);
        vb[i] = __uint_as_float(b[i]);
    }
}

// Instruction descriptor, kind::f16: D = F32, A = B = F16, both K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc_f16(uint32_t neg_a, uint32_t n) {
    return (1u << 4) | (neg_a << 13) | ((n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

// The products of one stage (its descriptor's low word ar: A re, A im, B re, B im tiles) into [Dr | Di], issued
// by the lanes with `leader` set; acc = 0 overwrites.
__device__ __forceinline__ void tc_stage_products(bool leader, uint32_t Dr, uint32_t Di, uint32_t ar, uint32_t acc) {
    constexpr uint32_t IDW = idesc_f16(0, 2 * BN), IDP = idesc_f16(0, BN), IDN = idesc_f16(1, BN);
    const uint32_t ai = ar + (TILE_A >> 4), br = ar + (2 * TILE_A >> 4), bi = br + (TILE_B >> 4);
    // [Dr | Di] (+)= A B^T at offsets oa and ob (16-byte units) of the 128-byte rows
    auto product = [&](uint32_t oa, uint32_t ob, uint32_t ac) {
        mma_f16(leader, Dr, ar + oa, br + ob, IDW, ac);
        mma_f16(leader, Dr, ai + oa, bi + ob, IDN, 1u);
        mma_f16(leader, Di, ai + oa, br + ob, IDP, 1u);
    };
#pragma unroll
    for (uint32_t kk = 0; kk < BKE / 16; ++kk) {
        const uint32_t hi = 2 * kk, lo = hi + 4;  // 16 halves = 32 bytes; lo 64 bytes after hi
        product(hi, hi, kk > 0 ? 1u : acc);
        product(hi, lo, 1u);
        product(lo, hi, 1u);
    }
}

// Output modes: OUT_C32 C (FP32 planar) = beta C + alpha D; OUT_Z64 C64 (FP64) = beta C64 + alpha D;
// OUT_PART the D of this K split to a workspace slice (split-K partial sums).
enum { OUT_C32 = 0, OUT_Z64 = 1, OUT_PART = 2 };

// The body of one CTA: tile (tm, tn) of C, K split z of S.  The four tensor maps are param-space
// copies (single product) or global-memory entries of a batch.
template <int OUT>
__device__ __forceinline__ void cgemm_tc_body(const CUtensorMap& tmAr, const CUtensorMap& tmAi, const CUtensorMap& tmBr,
                                              const CUtensorMap& tmBi, float* __restrict__ Cr, float* __restrict__ Ci,
                                              double2* __restrict__ C64, long ldc, long zstride, int m, int n, int K,
                                              int S, int zsplit, float alpha, float beta, const TcScale& sc,
                                              int* __restrict__ err) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // full[S], empty[S], done, never (the test hook's barrier: initialised, never arrived on)
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    // (the shuffle tells the compiler that the warp index is uniform)
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int tm = blockIdx.x, tn = blockIdx.y;
    // this CTA's K split: k-blocks [kb_begin, kb_begin + nkb)
    const int nkb_all = (K + BKE - 1) / BKE;
    const int kb_begin = (int)((long)zsplit * nkb_all / S);
    const int nkb = (int)((long)(zsplit + 1) * nkb_all / S) - kb_begin;
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES), done = smem_u32(bars + 2 * STAGES);
    const uint32_t never = smem_u32(bars + 2 * STAGES + 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(done, 1);
        mbar_init(never, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), TMEM_COLS);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t Dr = tmem, Di = tmem + BN;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int issued = 0;
        for (int kb = 0; kb < nkb; ++kb) {
            const int s = kb % STAGES;
            const uint32_t ph = (uint32_t)(kb / STAGES) & 1u;
            if (kb >= STAGES && !mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag)) break;
            uint8_t* st = smem + s * STAGE_BYTES;
            const uint32_t fb = full0 + 8 * s;
            mbar_expect_tx(fb, STAGE_BYTES);
            const int kx = (kb_begin + kb) * 2 * BKE;
            tma_load_2d(smem_u32(st), &tmAr, fb, kx, tm * BM);
            tma_load_2d(smem_u32(st + TILE_A), &tmAi, fb, kx, tm * BM);
            tma_load_2d(smem_u32(st + 2 * TILE_A), &tmBr, fb, kx, tn * BN);
            tma_load_2d(smem_u32(st + 2 * TILE_A + TILE_B), &tmBi, fb, kx, tn * BN);
            issued = kb + 1;
        }
        if (*abort_flag) {
            // let copies already in flight land before shared memory is released
            for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb) {
                const uint64_t t0 = gtimer();
                while (!mbar_try(full0 + 8 * (kb % STAGES), (uint32_t)(kb / STAGES) & 1u) && gtimer() - t0 < WAIT_NS) {
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (the whole warp walks the loop, lane 0 issues) ----------------
        const bool leader = lane == 0;
        if (err[1] != 0) {
            // test hook: a wait that nothing ends, bounded like every other wait
            const uint64_t t0 = gtimer();
            while (!mbar_try(never, 0u) && gtimer() - t0 < TEST_WAIT_NS) {
            }
            *abort_flag = 1;
        }
        const uint32_t lo0 = desc_lo(smem_u32(smem));
        int s = 0;
        uint32_t ph = 0;
        for (int kb = 0; kb < nkb && !*abort_flag; ++kb) {
            if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) break;
            fence_after();
            const uint32_t ar = lo0 + (uint32_t)s * (STAGE_BYTES >> 4);
            tc_stage_products(leader, Dr, Di, ar, kb > 0 ? 1u : 0u);
            if (leader) mma_commit(empty0 + 8 * s);
            if (++s == STAGES) {
                s = 0;
                ph ^= 1u;
            }
        }
        __syncwarp();
        if (leader) {
            mma_commit(done);
            if (*abort_flag) {
                // the products already issued finish (and the commit lands) before TMEM and shared
                // memory are released
                const uint64_t t0 = gtimer();
                while (!mbar_try(done, 0u) && gtimer() - t0 < WAIT_NS) {
                }
            }
        }
    }
    __syncwarp();
    // ---------------- epilogue: all four warps ----------------
    mbar_wait(done, 0, abort_flag);
    fence_before();
    __syncthreads();  // the abort decision below must be uniform: tcgen05.ld is warp-synchronous
    fence_after();
    if (!*abort_flag) {
        const long row = (long)tm * BM + warp * 32 + lane;
        const uint32_t lane_off = (uint32_t)(warp * 32) << 16;
        const long col0 = (long)tn * BN;
        const int er = sc.e0 + (sc.eA != nullptr && row < m ? __ldg(sc.eA + row) : 0);
#pragma unroll 1
        for (int c0 = 0; c0 < BN && col0 + c0 < n; c0 += 16) {  // (few right-hand sides: few chunks)
            float vr[16], vi[16];
            tmem_ld16x2(Dr + lane_off + c0, Di + lane_off + c0, vr, vi);
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const long col = col0 + c0 + q;
                const int e = er + (col < n ? __ldg(sc.eB + col) : 0);
                const float f = tc_pow2(e >> 1), g = tc_pow2(e - (e >> 1));  // e may exceed one factor's range
                vr[q] = vr[q] * f * g;
                vi[q] = vi[q] * f * g;
            }
            if (OUT == OUT_PART && row < m) {
                // slice z of the workspace: m x n column-major, leading dimension ldc (= m)
                float* Pr = Cr + (long)zsplit * zstride;
                float* Pi = Ci + (long)zsplit * zstride;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const long col = col0 + c0 + q;
                    if (col < n) {
                        Pr[row + col * ldc] = vr[q];
                        Pi[row + col * ldc] = vi[q];
                    }
                }
            } else if (OUT == OUT_Z64 && row < m) {
                double2 cz[16];
                if (beta != 0.f) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const long col = col0 + c0 + q;
                        cz[q] = (col < n) ? C64[row + col * ldc] : make_double2(0.0, 0.0);
                    }
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const long col = col0 + c0 + q;
                    if (col < n) {
                        double r = (double)alpha * (double)vr[q], im = (double)alpha * (double)vi[q];
                        if (beta != 0.f) {
                            r = fma((double)beta, cz[q].x, r);
                            im = fma((double)beta, cz[q].y, im);
                        }
                        C64[row + col * ldc] = make_double2(r, im);
                    }
                }
            } else if (OUT == OUT_C32 && row < m) {
                // issue every load of this 16-column chunk before any store, so the chunk costs
                // one memory round trip instead of sixteen
                float cr[16], ci[16];
                if (beta != 0.f) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const long col = col0 + c0 + q;
                        cr[q] = (col < n) ? __ldg(Cr + row + col * ldc) : 0.f;
                        ci[q] = (col < n) ? __ldg(Ci + row + col * ldc) : 0.f;
                    }
                }
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const long col = col0 + c0 + q;
                    if (col < n) {
                        const long o = row + col * ldc;
                        float r = alpha * vr[q], im = alpha * vi[q];
                        if (beta != 0.f) {
                            r = fmaf(beta, cr[q], r);
                            im = fmaf(beta, ci[q], im);
                        }
                        Cr[o] = r;
                        Ci[o] = im;
                    }
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicExch(err, 1);
}

template <int OUT>
__global__ void __launch_bounds__(128, 1)
    cgemm_tc_kernel(const __grid_constant__ CUtensorMap tmAr, const __grid_constant__ CUtensorMap tmAi,
                    const __grid_constant__ CUtensorMap tmBr, const __grid_constant__ CUtensorMap tmBi,
                    float* __restrict__ Cr, float* __restrict__ Ci, double2* __restrict__ C64, long ldc, long zstride,
                    int m, int n, int K, int S, float alpha, float beta, int* __restrict__ err, TcScale sc) {
    cgemm_tc_body<OUT>(tmAr, tmAi, tmBr, tmBi, Cr, Ci, C64, ldc, zstride, m, n, K, S, (int)blockIdx.z, alpha, beta,
                       sc, err);
}

// C -= A B^T for the LU trailing updates: few K (128 of them), so loading and storing C sets the time.  One
// persistent CTA per SM walks the 128 x 128 tiles (numbers first, first + grid, ...; row tiles fastest).  Warp 0
// loads the operands ahead across tiles, warp 1 issues into the two accumulators in turn, and sixteen warps
// take a tile's C into registers (64 loads in flight per thread, a quarter of the columns each) while its
// products run, then subtract and store while the next tile's do.  Against one CTA per tile with the C tile
// staged through tensor memory by four warps, 8064 x 8064 (63 x 63 tiles): 477 -> 206 us (5.0 TB/s of C), one tile
// alone 18.4 -> 11.6 us; the next tile prefetched into L2 makes 10 % of it.  An entry takes one product with its
// row's factor and one multiply-add with its column's, which is uniform in the warp (a factor per entry from both
// exponents: 10 % slower).
constexpr int UPD_WARPS = 16, UPD_THREADS = 64 + 32 * UPD_WARPS;
constexpr int UPD_COLS = BN / (UPD_WARPS / 4);  // columns per warp
static_assert(UPD_COLS == 32, "a lane per column");
__device__ __forceinline__ void tmem_ld8x2(uint32_t ta, uint32_t tb, float* va, float* vb) {
    uint32_t a[8], b[8];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]), "=r"(a[7]), "=r"(b[0]),
          "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]), "=r"(b[6]), "=r"(b[7])
        : "r"(ta), "r"(tb)
        : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        va[i] = __uint_as_float(a[i]);
        vb[i] = __uint_as_float(b[i]);
    }
}

__global__ void __launch_bounds__(UPD_THREADS, 1)
    cgemm_tc_upd_kernel(const __grid_constant__ CUtensorMap tmAr, const __grid_constant__ CUtensorMap tmAi,
                        const __grid_constant__ CUtensorMap tmBr, const __grid_constant__ CUtensorMap tmBi,
                        float* __restrict__ Cr, float* __restrict__ Ci, long ldc, int m, int n, int K,
                        int* __restrict__ err, TcScale sc, TcGate gate) {
    if (gate.fail) {  // a factorisation that stopped before this product's block (lu_fast.cu)
        const int f = *reinterpret_cast<const volatile int*>(gate.fail);
        if (f != 0 && (f >> 1) <= gate.block) return;
    }
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    // full[S], empty[S], accfull[2], accempty[2], drain, never (the test hook's)
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 6);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    const int ntm = (m + BM - 1) / BM, ntiles = ntm * ((n + BN - 1) / BN);
    const int nkb = (K + BKE - 1) / BKE;
    const int first = gate.first_tile + (int)blockIdx.x, step = (int)gridDim.x;
    const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * STAGES, accfull = empty0 + 8 * STAGES;
    const uint32_t accempty = accfull + 16, drain = accempty + 16, never = drain + 8;
    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(accfull + 8 * s, 1);
            mbar_init(accempty + 8 * s, UPD_WARPS);
        }
        mbar_init(drain, 1);
        mbar_init(never, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) tmem_alloc(smem_u32(tmem_slot), 2 * TMEM_COLS);
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer ----------------
        int it = 0;  // stages issued
        for (int t = first; t < ntiles && !*abort_flag; t += step) {
            const int tm = t % ntm, tn = t / ntm;
            for (int kb = 0; kb < nkb; ++kb, ++it) {
                const int s = it % STAGES;
                if (it >= STAGES && !mbar_wait(empty0 + 8 * s, (uint32_t)(it / STAGES - 1) & 1u, abort_flag)) break;
                uint8_t* st = smem + s * STAGE_BYTES;
                const uint32_t fb = full0 + 8 * s;
                mbar_expect_tx(fb, STAGE_BYTES);
                const int kx = kb * 2 * BKE;
                tma_load_2d(smem_u32(st), &tmAr, fb, kx, tm * BM);
                tma_load_2d(smem_u32(st + TILE_A), &tmAi, fb, kx, tm * BM);
                tma_load_2d(smem_u32(st + 2 * TILE_A), &tmBr, fb, kx, tn * BN);
                tma_load_2d(smem_u32(st + 2 * TILE_A + TILE_B), &tmBi, fb, kx, tn * BN);
            }
        }
        if (*abort_flag) {
            // copies already in flight land before shared memory is released
            for (int i = (it > STAGES ? it - STAGES : 0); i < it; ++i) {
                const uint64_t t0 = gtimer();
                while (!mbar_try(full0 + 8 * (i % STAGES), (uint32_t)(i / STAGES) & 1u) && gtimer() - t0 < WAIT_NS) {
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (the whole warp walks the loop, lane 0 issues) ----------------
        const bool leader = lane == 0;
        if (err[1] != 0) {  // test hook: as in cgemm_tc_body
            const uint64_t t0 = gtimer();
            while (!mbar_try(never, 0u) && gtimer() - t0 < TEST_WAIT_NS) {
            }
            *abort_flag = 1;
        }
        const uint32_t lo0 = desc_lo(smem_u32(smem));
        int s = 0, j = 0;  // stage, tile of this CTA
        uint32_t ph = 0;
        bool ok = true;
        for (int t = first; t < ntiles && ok && !*abort_flag; t += step, ++j) {
            const int buf = j & 1;
            if (j >= 2 && !mbar_wait(accempty + 8 * buf, (uint32_t)((j >> 1) - 1) & 1u, abort_flag)) break;
            fence_after();
            const uint32_t Dr = tmem + (uint32_t)buf * TMEM_COLS, Di = Dr + BN;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) {
                    ok = false;
                    break;
                }
                fence_after();
                const uint32_t ar = lo0 + (uint32_t)s * (STAGE_BYTES >> 4);
                tc_stage_products(leader, Dr, Di, ar, kb > 0 ? 1u : 0u);
                if (leader) mma_commit(empty0 + 8 * s);
                if (++s == STAGES) {
                    s = 0;
                    ph ^= 1u;
                }
            }
            if (ok && leader) mma_commit(accfull + 8 * buf);
        }
        __syncwarp();
        if (leader) {
            // the products already issued finish before TMEM and shared memory are released
            mma_commit(drain);
            const uint64_t t0 = gtimer();
            while (!mbar_try(drain, 0u) && gtimer() - t0 < WAIT_NS) {
            }
        }
    } else if (warp >= 2) {
        // ---------------- C (sixteen warps) ----------------
        const int qw = warp & 3, cg = (warp - 2) >> 2;  // TMEM lane quarter this warp may access; column group
        const uint32_t lane_off = (uint32_t)(qw * 32) << 16;
        int j = 0;
        for (int t = first; t < ntiles; t += step, ++j) {
            const int tm = t % ntm, tn = t / ntm, buf = j & 1;
            const long row = (long)tm * BM + qw * 32 + lane;
            const int col0 = tn * BN + cg * UPD_COLS;
            const int nc = row < m ? min(UPD_COLS, n - col0) : 0;  // columns of this thread inside C
            // minus the row's factor; it and the columns' are normal numbers (TcRowScale), and a product times the
            // first is about L21's entry times 2^15
            const float rf = -tc_pow2(row < m ? __ldg(sc.eA + row) : 0);
            float* pr = Cr + row + (long)col0 * ldc;
            float* pi = Ci + row + (long)col0 * ldc;
            const int ld = (int)ldc;  // (32 columns of it fit an int)
            if (t + step < ntiles) {  // the next tile's C into L2: a lane per column, its 32 rows of this warp a line
                const long r2 = (long)((t + step) % ntm) * BM + qw * 32;
                const int c2 = (t + step) / ntm * BN + cg * UPD_COLS + lane;
                if (r2 < m && c2 < n) {
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(Cr + r2 + (long)c2 * ldc));
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(Ci + r2 + (long)c2 * ldc));
                }
            }
            float cr[UPD_COLS], ci[UPD_COLS];
#pragma unroll
            for (int q = 0; q < UPD_COLS; ++q) {
                cr[q] = q < nc ? __ldcg(pr + q * ld) : 0.f;
                ci[q] = q < nc ? __ldcg(pi + q * ld) : 0.f;
            }
            const bool got = mbar_wait(accfull + 8 * buf, (uint32_t)(j >> 1) & 1u, abort_flag);
            if (!__all_sync(0xffffffffu, got)) break;
            fence_after();
            const uint32_t D = tmem + (uint32_t)buf * TMEM_COLS + lane_off + cg * UPD_COLS;
#pragma unroll
            for (int c0 = 0; c0 < UPD_COLS; c0 += 8) {
                float vr[8], vi[8];
                tmem_ld8x2(D + c0, D + BN + c0, vr, vi);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float cf = tc_pow2(col0 + c0 + q < n ? __ldg(sc.eB + col0 + c0 + q) : 0);
                    cr[c0 + q] = fmaf(vr[q] * rf, cf, cr[c0 + q]);
                    ci[c0 + q] = fmaf(vi[q] * rf, cf, ci[c0 + q]);
                }
            }
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(accempty + 8 * buf);
#pragma unroll
            for (int q = 0; q < UPD_COLS; ++q)
                if (q < nc) {
                    pr[q * ld] = cr[q];
                    pi[q * ld] = ci[q];
                }
        }
    }
    __syncwarp();  // the roles' lanes meet again: the barrier below is warp-aligned
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        tmem_dealloc(tmem, 2 * TMEM_COLS);
    }
    if (threadIdx.x == 0 && *abort_flag) atomicExch(err, 1);
}

// One product per blockIdx.z: C_z = beta C_z + alpha A_z B_z^T for a batch of equal-shape products
// (the contour points' Schur complements), maps and outputs read from global memory.
struct alignas(64) TcBatchEntry {
    CUtensorMap map[4];  // A re, A im, B re, B im
    float* Cr;
    float* Ci;
    long ldc;
    TcScale sc;
};
__global__ void __launch_bounds__(128, 1)
    cgemm_tc_batch_kernel(const TcBatchEntry* __restrict__ E, int m, int n, int K, float alpha, int* __restrict__ err) {
    const TcBatchEntry& e = E[blockIdx.z];
    cgemm_tc_body<OUT_C32>(e.map[0], e.map[1], e.map[2], e.map[3], e.Cr, e.Ci, nullptr, e.ldc, 0, m, n, K, 1, 0,
                           alpha, 0.f, e.sc, err);
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
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

// 2-D tensor map over a row-major [rows][ldk] pack of K entries a row (tc_ldk): dims {2 K rounded to 64,
// rows} halves, box {64, box_rows}, 128-byte swizzle; reads outside return zeros.
bm_status tc_make_map(void* tmap, const __half* base, long rows, long K, long ldk, int box_rows) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode();
    if (enc == nullptr) {
        bm_set_error("cuTensorMapEncodeTiled is unavailable from the driver");
        return BM_ECUDA;
    }
    if ((reinterpret_cast<uintptr_t>(base) & 15) != 0 || (ldk * 2) % 16 != 0) {
        bm_set_error("tensor map: base or stride not 16-byte aligned");
        return BM_EINVAL;
    }
    cuuint64_t dims[2] = {(cuuint64_t)tc_ldk(K), (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ldk * 2};
    cuuint32_t box[2] = {(cuuint32_t)(2 * BKE), (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(reinterpret_cast<CUtensorMap*>(tmap), CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base),
                     dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
        bm_set_error("cuTensorMapEncodeTiled failed with code " + std::to_string((int)r));
        return BM_ECUDA;
    }
    return BM_OK;
}

namespace {

template <int OUT>
cudaError_t launch_tc(cudaStream_t s, dim3 grid, const void* tAr, const void* tAi, const void* tBr, const void* tBi,
                      float* Cr, float* Ci, double2* C64, long ldc, long zstride, int m, int n, int K, int S,
                      float alpha, float beta, int* d_err, TcScale sc) {
    static DeviceFlags attr_set;
    if (attr_set.pending()) {
        cudaError_t e =
            cudaFuncSetAttribute(cgemm_tc_kernel<OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        if (e != cudaSuccess) return e;
        attr_set.done();
    }
    cgemm_tc_kernel<OUT><<<grid, 128, SMEM_BYTES, s>>>(
        *reinterpret_cast<const CUtensorMap*>(tAr), *reinterpret_cast<const CUtensorMap*>(tAi),
        *reinterpret_cast<const CUtensorMap*>(tBr), *reinterpret_cast<const CUtensorMap*>(tBi), Cr, Ci, C64, ldc,
        zstride, m, n, K, S, alpha, beta, d_err, sc);
    return cudaGetLastError();
}

// C = beta C + alpha sum_z P[z]  (P: S slices of m x n column-major, leading dimension m)
__global__ void splitk_reduce_c32_kernel(const float* __restrict__ Pr, const float* __restrict__ Pi, int S, int m,
                                         int n, float alpha, float beta, float* __restrict__ Cr,
                                         float* __restrict__ Ci, long ldc) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long zs = (long)m * n;
    if (idx >= zs) return;
    const int j = (int)(idx / m), i = (int)(idx % m);
    float r = 0.f, im = 0.f;
    for (int z = 0; z < S; ++z) {
        r += __ldg(Pr + idx + z * zs);
        im += __ldg(Pi + idx + z * zs);
    }
    const long o = i + (long)j * ldc;
    float cr = alpha * r, ci = alpha * im;
    if (beta != 0.f) {
        cr = fmaf(beta, Cr[o], cr);
        ci = fmaf(beta, Ci[o], ci);
    }
    Cr[o] = cr;
    Ci[o] = ci;
}

// C64 = beta C64 + alpha sum_z P[z], the slice sum in FP32 (it is an FP32 product)
__global__ void splitk_reduce_z64_kernel(const float* __restrict__ Pr, const float* __restrict__ Pi, int S, int m,
                                         int n, float alpha, float beta, double2* __restrict__ C, long ldc) {
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long zs = (long)m * n;
    if (idx >= zs) return;
    const int j = (int)(idx / m), i = (int)(idx % m);
    float r = 0.f, im = 0.f;
    for (int z = 0; z < S; ++z) {
        r += __ldg(Pr + idx + z * zs);
        im += __ldg(Pi + idx + z * zs);
    }
    double2& c = C[i + (long)j * ldc];
    double cr = (double)alpha * (double)r, ci = (double)alpha * (double)im;
    if (beta != 0.f) {
        cr = fma((double)beta, c.x, cr);
        ci = fma((double)beta, c.y, ci);
    }
    c = make_double2(cr, ci);
}

// B operand of a skinny product: V (K x nrhs FP32 planar, column-major) -> row c of a [nrhs][ldk] pack and
// its exponent eB[c], the entries from `half` on times 2^*shift (balance_kernel).  One CTA per column, which it reads twice
// (the second time from L2).
struct PlanarCol {
    const float *re, *im;
    int half;
    float w;
    __device__ __forceinline__ float2 operator()(long k) const {
        const float f = k < half ? 1.f : w;
        return make_float2(__ldg(re + k) * f, __ldg(im + k) * f);
    }
};
__global__ void __launch_bounds__(TC_PACK_THREADS) pack_b_kernel(const float* __restrict__ Vr,
                                                                 const float* __restrict__ Vi, long ldv, int K, int half,
                                                                 const int* __restrict__ shift, __half* __restrict__ Br, __half* __restrict__ Bi,
                                                                 long ldk, int* __restrict__ eB) {
    const long c = blockIdx.x;
    const float w = shift != nullptr ? tc_pow2(*shift) : 1.f;
    tc_pack_column(PlanarCol{Vr + c * ldv, Vi + c * ldv, half, w}, K, Br + c * ldk, Bi + c * ldk, eB + c);
}

}  // namespace

// C = alpha A B^T, C FP32 planar column-major (m x n, ld ldc); one K range per CTA.
cudaError_t gemm_tc(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, float* Cr,
                    float* Ci, long ldc, int m, int n, int K, float alpha, TcScale sc, int* d_err) {
    if (m <= 0 || n <= 0 || K <= 0) return cudaSuccess;
    return launch_tc<OUT_C32>(s, dim3(ceil_div(m, BM), ceil_div(n, BN), 1), tAr, tAi, tBr, tBi, Cr, Ci, nullptr, ldc, 0,
                              m, n, K, 1, alpha, 0.f, d_err, sc);
}

// C -= A B^T by at most `ctas` CTAs.
cudaError_t gemm_tc_upd(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, float* Cr,
                        float* Ci, long ldc, int m, int n, int K, TcScale sc, int ctas, int* d_err, TcGate gate) {
    if (m <= 0 || n <= 0 || K <= 0) return cudaSuccess;
    static DeviceFlags attr_set;
    if (attr_set.pending()) {
        cudaError_t e = cudaFuncSetAttribute(cgemm_tc_upd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
        if (e != cudaSuccess) return e;
        attr_set.done();
    }
    const int tiles = ceil_div(m, BM) * ceil_div(n, BN) - gate.first_tile;
    if (tiles <= 0) return cudaSuccess;
    cgemm_tc_upd_kernel<<<std::min(tiles, std::max(ctas, 1)), UPD_THREADS, SMEM_BYTES, s>>>(
        *reinterpret_cast<const CUtensorMap*>(tAr), *reinterpret_cast<const CUtensorMap*>(tAi),
        *reinterpret_cast<const CUtensorMap*>(tBr), *reinterpret_cast<const CUtensorMap*>(tBi), Cr, Ci, ldc, m, n, K,
        d_err, sc, gate);
    return cudaGetLastError();
}

// Number of K splits for a product with few output tiles: about three waves of CTAs over the
// SMs (one CTA per SM fits), at most 32 splits and at least one 32-wide K step per split.
int tc_split_k(int m, int n, int K, int num_sms) {
    const long tiles = (long)ceil_div(m, BM) * ceil_div(n, BN);
    const int nkb = ceil_div(K, BKE);
    long S = (3L * num_sms) / tiles;
    if (S > 32) S = 32;
    if (S > nkb) S = nkb;
    if (S < 1) S = 1;
    return (int)S;
}

// Split-K product into an FP32 planar (dst.re, dst.im) or FP64 (dst.z) destination:
// dst = beta dst + alpha A B^T.  With S > 1 splits, each writes its partial product to the
// workspace (Pr, Pi: S m n floats each) and one reduction kernel sums the slices in a fixed order
// (deterministic).  Returns the number of kernels launched in *launched.
cudaError_t gemm_tc_split(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, int m,
                          int n, int K, float alpha, float beta, TcScale sc, TcDest dst, int S, float* Pr, float* Pi,
                          int* d_err, int* launched) {
    *launched = 0;
    if (m <= 0 || n <= 0 || K <= 0) return cudaSuccess;
    const bool z64 = dst.z != nullptr;
    if (S <= 1) {
        dim3 grid(ceil_div(m, BM), ceil_div(n, BN), 1);
        *launched = 1;
        if (z64)
            return launch_tc<OUT_Z64>(s, grid, tAr, tAi, tBr, tBi, nullptr, nullptr, dst.z, dst.ld, 0, m, n, K, 1,
                                      alpha, beta, d_err, sc);
        return launch_tc<OUT_C32>(s, grid, tAr, tAi, tBr, tBi, dst.re, dst.im, nullptr, dst.ld, 0, m, n, K, 1,
                                  alpha, beta, d_err, sc);
    }
    dim3 grid(ceil_div(m, BM), ceil_div(n, BN), S);
    const long zs = (long)m * n;
    cudaError_t e = launch_tc<OUT_PART>(s, grid, tAr, tAi, tBr, tBi, Pr, Pi, nullptr, m, zs, m, n, K, S, 1.f, 0.f,
                                        d_err, sc);
    if (e != cudaSuccess) return e;
    const int nb = (int)ceil_div(zs, 256L);
    if (z64)
        splitk_reduce_z64_kernel<<<nb, 256, 0, s>>>(Pr, Pi, S, m, n, alpha, beta, dst.z, dst.ld);
    else
        splitk_reduce_c32_kernel<<<nb, 256, 0, s>>>(Pr, Pi, S, m, n, alpha, beta, dst.re, dst.im, dst.ld);
    *launched = 2;
    return cudaGetLastError();
}

cudaError_t launch_pack_b(cudaStream_t s, const float* Vr, const float* Vi, long ldv, int K, int half,
                          const int* shift, int nrhs, __half* Br, __half* Bi, long ldk, int* eB) {
    if (K <= 0 || nrhs <= 0) return cudaSuccess;
    pack_b_kernel<<<nrhs, TC_PACK_THREADS, 0, s>>>(Vr, Vi, ldv, K, half, shift, Br, Bi, ldk, eB);
    return cudaGetLastError();
}

// Batched Schur-type product: for each of B entries (maps: 4 opaque 128-byte tensor maps, outputs)
// C = alpha A B^T (beta = 0), one launch with grid.z = B.  d_entries: device scratch of
// B * tc_batch_entry_bytes() bytes, filled here.
size_t tc_batch_entry_bytes() { return sizeof(TcBatchEntry); }
cudaError_t gemm_tc_batch(cudaStream_t s, int B, const void* const* maps, float* const* Cr, float* const* Ci,
                          const long* ldc, const TcScale* sc, int m, int n, int K, float alpha, void* d_entries,
                          int* d_err) {
    if (B < 1 || m <= 0 || n <= 0 || K <= 0) return cudaSuccess;
    static DeviceFlags attr;
    if (attr.pending()) {
        cudaError_t e = cudaFuncSetAttribute(cgemm_tc_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             SMEM_BYTES);
        if (e != cudaSuccess) return e;
        attr.done();
    }
    std::vector<TcBatchEntry> h(B);
    for (int b = 0; b < B; ++b) {
        for (int q = 0; q < 4; ++q)
            std::memcpy(&h[b].map[q], static_cast<const unsigned char*>(maps[b]) + 128 * q, sizeof(CUtensorMap));
        h[b].Cr = Cr[b];
        h[b].Ci = Ci[b];
        h[b].ldc = ldc[b];
        h[b].sc = sc[b];
    }
    cudaError_t e = cudaMemcpyAsync(d_entries, h.data(), sizeof(TcBatchEntry) * B, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    dim3 grid(ceil_div(m, BM), ceil_div(n, BN), B);
    cgemm_tc_batch_kernel<<<grid, 128, SMEM_BYTES, s>>>(reinterpret_cast<const TcBatchEntry*>(d_entries), m, n, K,
                                                        alpha, d_err);
    return cudaGetLastError();
}
