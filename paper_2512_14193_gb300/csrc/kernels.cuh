// Launchers shared between the library's translation units (internal).
#pragma once
#include "common.cuh"

#include <cuda_fp16.h>

// assemble.cu
cudaError_t launch_geometry(cudaStream_t s, int kind, const double p[4], int N, const double* d_user, double* d_geom);
cudaError_t launch_assemble(cudaStream_t s, const bm_ctx* c);
size_t asm_args_bytes();
cudaError_t launch_assemble_batch(cudaStream_t s, bm_ctx* const* cs, int B, void* d_args);
cudaError_t launch_zeta_band(cudaStream_t s, const bm_ctx* c);  // high-order zeta corrections (zeta_p > 0)
cudaError_t launch_normA(cudaStream_t s, const bm_ctx* c);
cudaError_t launch_plane_wave(cudaStream_t s, const bm_ctx* c, const double* d_ang, int nrhs, double2* B, long ldb);
cudaError_t launch_far_field(cudaStream_t s, const bm_ctx* c, const double2* X, long ldx, int nrhs, const double* d_ang,
                             int M, double2* U, long ldu);
cudaError_t launch_hankel_probe(cudaStream_t s, const bm_ctx* c, const double2* z, int n, double2* h0, double2* h1);
cudaError_t launch_f32_convert(cudaStream_t s, const double* x, int n, float* rn);
cudaError_t launch_pack_schur(cudaStream_t s, const bm_ctx* c);  // Schur operands (in bm_factor)
cudaError_t launch_pack_solve(cudaStream_t s, const bm_ctx* c);  // [M13; M23] rows (assembly)
cudaError_t launch_to_c32(cudaStream_t s, const double2* A, long lda, int m, int n, float* Fr, float* Fi, long ldf);

// gemm_simt.cu
// (stop: the launch does nothing when this word is not zero)
cudaError_t gemm_z64(cudaStream_t s, int m, int n, int k, double alpha, Z64 A, Z64 B, double beta, Z64 C,
                     const int* stop = nullptr);
cudaError_t gemm_z64_skinny(cudaStream_t s, int num_sms, int m, int n, int k, double alpha, Z64 A, Z64 B, double beta,
                            Z64 C);
cudaError_t gemm_c32(cudaStream_t s, int m, int n, int k, float alpha, C32 A, C32 B, float beta, C32 C);

// gemm_tc.cu (tensor maps are CUtensorMap, passed as opaque 128-byte blobs)
bm_status tc_make_map(void* tmap, const __half* base, long rows, long K, long ldk, int box_rows);
constexpr long tc_ldk(long K) { return (K + 31) / 32 * 64; }  // halves per pack row of K entries (hi and lo)
// Scales of a product's packs: entry (i, j) of A B^T is the packed product times 2^(eA[i] + eB[j] + e0)
// (eA null: zeros)
struct TcScale {
    const int* eA = nullptr;
    const int* eB = nullptr;
    int e0 = 0;
};
TcScale schur_scale(const bm_ctx* c);          // of the Schur complement's packs (and the A of the skinny product with them)
// Balance of the product [M31 M32] [M13; M23]: 2^s moved from the columns of M32 to the rows of M23, so that one
// scale per row of the one and per column of the other loses neither block (balance_kernel).
constexpr int BAL_G = 0;      // exponents of the largest entries of M13, M23, M31, M32
constexpr int BAL_SHIFT = 4;  // s
constexpr int BAL_ROWS = 8;   // exponents of the rows of M31, then of M32
constexpr size_t bal_ints(long N) { return BAL_ROWS + 2 * (size_t)N; }
constexpr int TC_E_DGE = -16;  // e0 of rows scaled by the digit planes' exponents (entries below 2^(e - 1))
// TcGate: the launch skips its first 128 x 128 tile (another launch takes it), and does nothing when the
// word *fail, if any, names a block of the factorisation up to `block` (lu_fast.cu)
struct TcGate {
    const int* fail = nullptr;
    int block = 0;
    int first_tile = 0;
};
cudaError_t gemm_tc(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, float* Cr,
                    float* Ci, long ldc, int m, int n, int K, float alpha, TcScale sc, int* d_err);
cudaError_t gemm_tc_upd(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, float* Cr,
                        float* Ci, long ldc, int m, int n, int K, TcScale sc, int ctas, int* d_err,
                        TcGate gate = TcGate{});
constexpr int TC_BM = 128;
constexpr int TC_BN = 128;
// destination of a split-K product: FP32 planar (re, im) or, when z is set, FP64 interleaved
struct TcDest {
    float* re;
    float* im;
    double2* z;
    long ld;
};
int tc_split_k(int m, int n, int K, int num_sms);
cudaError_t gemm_tc_split(cudaStream_t s, const void* tAr, const void* tAi, const void* tBr, const void* tBi, int m,
                          int n, int K, float alpha, float beta, TcScale sc, TcDest dst, int S, float* Pr, float* Pi,
                          int* d_err, int* launched);
cudaError_t launch_pack_b(cudaStream_t s, const float* Vr, const float* Vi, long ldv, int K, int half, const int* shift,
                          int nrhs, __half* Br, __half* Bi, long ldk, int* eB);
size_t tc_batch_entry_bytes();
cudaError_t gemm_tc_batch(cudaStream_t s, int B, const void* const* maps, float* const* Cr, float* const* Ci,
                          const long* ldc, const TcScale* sc, int m, int n, int K, float alpha, void* d_entries,
                          int* d_err);

// lu.cu
bm_status lu_setup(bm_ctx* c, int cluster_cap, int panel_kernel);
bm_status lu_factor_enqueue(bm_ctx* c);       // factor d_F64 / d_F32 in place (stream-ordered)
// continue a factorisation that stopped at a block (the value of its stop word) with the pivot search
bm_status lu_resume_enqueue(bm_ctx* c, int stop);
size_t lu_fast_bytes(int n);                  // work buffer of the search-free blocks (d_fd)
size_t lu_fast_z_bytes(int n);                // and of the FP64 ones
size_t swap_map_bytes();
constexpr int FLOW_BN = 8;                  // right-hand sides per item of the FP32 triangular solve
constexpr size_t FLOW_ITEM_BYTES = 64 * FLOW_BN * sizeof(float2);  // an item's 64 rows in its exchange buffer
bm_status getrs_z64(bm_ctx* c, double2* Y, long ldy, int nrhs);   // in place; Y holds P B (rows gathered by perm)
bm_status getrs_c32(bm_ctx* c, float* Yr, float* Yi, long ldy, int nrhs);
cudaError_t launch_gather_rows_z64(cudaStream_t s, const int* perm, int n, int nrhs, const double2* B, long ldb,
                                   double2* Y, long ldy);
cudaError_t launch_gather_rows_c32(cudaStream_t s, const int* perm, int n, int nrhs, const float* Br, const float* Bi,
                                   long ldb, float* Yr, float* Yi, long ldy);

// solve.cu
bm_status solve_fp64(bm_ctx* c, const double2* B, double2* X, long ld, int nrhs);
bm_status residual_fp64(bm_ctx* c, const double2* B, const double2* X, double2* R, long ld, int nrhs);
bm_status backward_error(bm_ctx* c, const double2* R, const double2* X, const double2* B, long ld, int nrhs,
                         double* d_eta);
bm_status correction_c32(bm_ctx* c, const double2* R, double2* X, long ld, int nrhs);
bm_status residual_update_c32(bm_ctx* c, double2* R, long ld, int nrhs);
bm_status residual_df(bm_ctx* c, const double2* B, const double2* X, double2* R, long ld, int nrhs);
bm_status residual_tc(bm_ctx* c, const double2* B, const double2* X, double2* R, long ld, int nrhs);

// resid_df.cu: C += alpha A X in double-float arithmetic (A as split planes, X and C FP64)
// one product C (m x n) += alpha A (m x k) X (k x n) of a double-float residual; S K splits (S > 1
// writes S m n raw partial sums to W, reduced in order afterwards)
struct DfProd {
    const float4* A;   // split planes of the operator (re_hi, re_lo, im_hi, im_lo)
    const float2* Q;   // split re + im
    long lda;
    const float4* XP;  // the iterate split the same way
    const float2* XQ;
    long ldx;
    double2* C;
    long ldc;
    double2* W;
    int m, k, S;
};
cudaError_t gemm_df(cudaStream_t s, const DfProd* prods, int nprod, int n, double alpha, int* launched);
cudaError_t launch_split_planes(cudaStream_t s, const double2* A, long lda, int m, int n, float4* P, float2* Q,
                                long ldp);
// gemm_simt.cu: C (FP64) += alpha A_hi B with A the hi parts of split planes, FP32 arithmetic
cudaError_t gemm_update_f4hi_c32(cudaStream_t s, int m, int n, int k, float alpha, F4Hi A, C32 B, Z64 C);
cudaError_t launch_copy_z64(cudaStream_t s, const double2* S, long lds, int m, int n, double2* D, long ldd);

// resid_tc.cu: r += alpha A x to FP64-level accuracy from exact bf16 digit products on the tensor
// cores (digit planes of A made once after assembly, of x per residual)
struct RtArgs {
    const void* tmA;   // host copies of the tensor maps (opaque 128-byte blobs)
    const void* tmX;
    const int* eA;     // row exponents of A (device)
    const int* fX;     // column exponents of x (device)
    double2* C;        // output, C += alpha A x
    long ldc;
    double* Wr;        // split-K workspace (S > 1): S m n doubles each
    double* Wi;
    int m, K, S;
};
long rt_ldk(long K);                 // leading dimension of a digit plane row (K rounded to 64)
int rt_digit_planes(int nd);         // planes of A (nd digits x Re, Im)
int rt_x_planes(int nd);             // planes of x
int rt_col_tile(int nd);             // right-hand sides per CTA
// K splits S[q] of the nprod products (m[q] rows, K[q] columns) of one launch with n right-hand sides
void rt_plan_splits(int nprod, const long* m, const long* K, int n, int nd, int num_sms, int* S);
bm_status rt_make_map(void* tmap, const void* base, long rows, long K, long ldk, long plane_elems, int box_rows,
                      int nd);
bm_status rt_make_map_x(void* tmaps, const void* base, long cols, long K, long ldk, int nd);  // two blobs
// Inner scale of a block's product L21 U12 of an LU: column k of L21 times 2^d, row k of U12 times 2^-d, d the
// difference of the exponents `re` of the matrix's rows that became the block's rows k and 0.  U12's rows have
// the size of those rows (the ordinary system's two block rows differ by beta), L21's columns its inverse, and a block
// where the two meet would otherwise lose the smaller under one scale per row and column.
__device__ __forceinline__ int inner_exponent(int ek, int e0) { return min(max(ek - e0, -100), 100); }
// K entries k are taken times 2^-at(k) (A) or 2^at(k) (x): from `half` on at = *shift, or the inner scale
// of a block whose rows have the exponents re[0], re[1], ..
struct RtShift {
    const int* shift = nullptr;
    int half = 0;
    const int* re = nullptr;
    __device__ __forceinline__ int at(int k) const {
        if (shift != nullptr) return k >= half ? __ldg(shift) : 0;
        return re != nullptr ? -inner_exponent(re[k], re[0]) : 0;
    }
};
// (rowmax: scratch of `rows` words to find the row exponents e with; null: e holds them)
cudaError_t launch_digits_a(cudaStream_t s, const double2* A, long lda, int rows, int K, int* e, void* D, long ldk,
                            void* rowmax, int nd, RtShift sh = RtShift{}, const int* stop = nullptr);
// |v| as the bits of a non-negative double, which order as the doubles do; infinities and NaN are the largest
__device__ __forceinline__ unsigned long long mag_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
// the bits of v 2^d from those of |v| (0 below the normal range)
__device__ __forceinline__ unsigned long long scaled_mag(unsigned long long b, int d) {
    if (d == 0 || b >= 0x7FF0000000000000ull) return b;
    const int e = (int)(b >> 52), n = e + d;
    if (e == 0 || n < 1) return 0;
    return (b & 0xFFFFFFFFFFFFFull) | (unsigned long long)min(n, 2046) << 52;
}
// Exponent of a row or column with an infinity or a NaN: its digits are zeros and its outputs NaN
constexpr int RT_NONFINITE = 1 << 20;
// e with m < 2^(e - 1) of the largest magnitude m of a row, given as its bits (`zero` for a zero row)
__device__ __forceinline__ int row_exponent(unsigned long long mx, int zero = 0) {
    if (mx >= 0x7FF0000000000000ull) return RT_NONFINITE;
    const double m = __longlong_as_double((long long)mx);
    int ex = 0;
    if (m > 0.0) frexp(m, &ex);  // m = f 2^ex, f in [1/2, 1)
    return m > 0.0 ? ex + 1 : zero;
}
cudaError_t launch_digits_x(cudaStream_t s, const double2* X, long ldx, int r0, int K, int n, int npad, int* f,
                            void* D, long ldk, long plane, int nd, RtShift sh = RtShift{}, const int* stop = nullptr);
cudaError_t gemm_rt(cudaStream_t s, const RtArgs* prods, int nprod, int n, double alpha, int* d_err, int* launched,
                    int nd, const int* stop = nullptr);

// FP64 products from nine-digit products (FP64 precision): workspace (0: the CUDA cores are the better
// place), and C += alpha A B (eA, sh: A's row exponents and the balance of the K entries, if they are there; stop:
// nothing is done when this word is not zero)
size_t dg_bytes(int m, int n, int K, int num_sms);
bm_status gemm_z64_dg(cudaStream_t s, void* work, int num_sms, int m, int n, int K, double alpha, Z64 A, Z64 B, Z64 C,
                      int* d_err, int* eA = nullptr, RtShift sh = RtShift{}, const int* stop = nullptr);

// api.cu: what a factorisation takes where the budget has room (before any capture), and gives back; the Schur
// complement of the FP64 precision into d_F64
void opt_reserve(bm_ctx* c);
void opt_release(bm_ctx* c, size_t bytes);
void ssm_yield_optional(int device);  // ssm.cu
bm_status schur_z64(bm_ctx* c, cudaStream_t s);
// api.cu: assembly in two halves (the batched contour solver assembles many handles at once)
bm_status assemble_impl(bm_ctx* c, const bm_curve* curve, int N, bm_c64 k_out, bm_c64 k_in, bm_formulation form,
                        const bm_opts* opts, bool defer_kernels);
bm_status assemble_post(bm_ctx* c, bool run_assembly_kernel, bool wait);  // wait: synchronise the stream
bm_status factor_lu_enqueue(bm_ctx* c);              // LU of the Schur complement in place (graph)
bm_status factor_continue(bm_ctx* c);                // waits; enqueues the rest of a factorisation that stopped
bm_status factor_result(bm_ctx* c, int* info);       // waits, reads info / timeout, sets the state
bm_status set_panel_cluster(bm_ctx* c, int cap);     // panel cluster cap of an assembled handle
