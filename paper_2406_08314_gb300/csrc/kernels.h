// Host-side launchers of the libmsd kernels (internal to csrc/).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

// Optional per-kernel event timing, supplied by the context.
struct TimerHook {
    void* self = nullptr;
    void (*begin_fn)(void*, const char*, cudaStream_t) = nullptr;
    void (*end_fn)(void*, cudaStream_t) = nullptr;
    void begin(const char* name, cudaStream_t st) const { if (begin_fn) begin_fn(self, name, st); }
    void end(cudaStream_t st) const { if (end_fn) end_fn(self, st); }
};

// k_wick.cu
// Reference inverse of one spin: inputs, outputs and, where ref_dg_use, the
// scratch of the tensor-core product (Sinv [nw][N][N]; cs [nw][N], the columns' scales;
// sa, ea: M rows, sb, eb: 2 N rows of dg_row_bytes(2 N) per walker; all NULL
// otherwise). GactT: the active block with the walkers contiguous, [nh np][nw].
struct RefSpinIn {
    const SpinTables* T = nullptr;
    const double2* phi = nullptr;
    double2 *Gr = nullptr, *O0 = nullptr, *Gact = nullptr, *GactT = nullptr;
    double2* Sinv = nullptr;
    double* cs = nullptr;
    void *sa = nullptr, *sb = nullptr;
    int *ea = nullptr, *eb = nullptr;
};
bool ref_dg_use(int M, int N);
size_t ref_dg_bytes(int M, int N);   // that scratch per walker (0 if unused)
int launch_refs(const RefSpinIn* in, int n_spin, int nw, int M, unsigned* err, cudaStream_t st);
// FP64 ratios r[w][s] and rT[s][w] and FP64 inverse minors by pivoted LU (trials whose
// sub-minors are too many for launch_inverse_ratios).
void launch_strings(const SpinTables& tb, int nw, const double2* Gact, double2* r, double2* rT, void* B, cudaStream_t st,
                    const TimerHook& th);
// Marks the walkers with large active blocks (big [nw]) and replaces their ratios and FP64
// inverse minors by those of the LU.
void launch_strings_large(const SpinTables& ta, const SpinTables& tb, int nw, double2* const GT[2], double2* const Gact[2],
                          int* const big[2], double2* const r[2], double2* const rT[2], void* const B[2], cudaStream_t st);
// k_minors.cu: FP64 ratios rT[s][w] of both spins by expansions over shared
// minors, those that cancel by LU (m2, t2: scratch, minor2_count entries per walker;
// tr: minor_marks entries; all NULL: every ratio by LU), FP32 inverse minors, and the CI
// weights.
size_t minor2_count(const SpinTables& t);
size_t minor_marks(const SpinTables& t);
void launch_minors(const SpinTables& ta, const SpinTables& tb, int nw, double2* const GT[2], double2* const m2[2],
                   int* const t2[2], int* const tr[2], double2* const rT[2], cudaStream_t st);
void launch_inverse_minors(const SpinTables& ta, const SpinTables& tb, int nw, double2* const Gact[2], void* const B[2],
                           cudaStream_t st);
int weights_blocks(const SpinTables& tb);
void launch_weights(const SpinTables& ta, const SpinTables& tb, int nw, double2* const rT[2], double2* const wts[2],
                    float2* const rf[2], double2* part, int nslot, bool beta, cudaStream_t st,
                    double2* const wT[2] = nullptr, int* const big[2] = nullptr);
// FP64 inverse minors and the FP64 cofactor matrix from the minors: per spin the trial's
// strings followed by the sub-minors outside the trial. V: [nh np + n2 + n_ext][nw] (G, 2
// x 2 minors, ratios), its first part given. Bv: [n_str + n_piece][nw], on entry to
// launch_cofactors the weights of the trial's strings (of a walker with a large active
// block those of its vanishing ratios only: the others go by their inverse minors).
struct ExtTables {
    int n_ext = 0, n2 = 0, n_piece = 0;
    int vbucket[MSD_KMAX + 2] = {0};
    uint4* str_hp = nullptr;     // [n_ext]
    int8_t* str_sign = nullptr;  // [n_ext]
    int* sub = nullptr;          // [n_ext][MSD_KMAX]
    int* row = nullptr;          // rows of V of the inverse minors' entries, at SpinTables::cmx_off
    // lists of the cofactor matrix: n_piece pieces, then the nh np sums of pieces
    int *cof_row = nullptr, *cof_off = nullptr;
    int2* cof_ent = nullptr;
};
// t2 [n2][nw], tr [n_ext - bucket[3]][nw]: scratch. B (may be NULL): the inverse minors of
// the strings whose ratios take the LU.
void launch_minors_ext(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw, double2* const V[2],
                       int* const t2[2], int* const tr[2], void* const B[2], cudaStream_t st);
// The other FP64 inverse minors from V and tr as launch_minors_ext left them.
void launch_inverse_ratios(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw,
                           double2* const V[2], int* const tr[2], void* const B[2], cudaStream_t st);
void launch_cofactors(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw, double2* const V[2],
                      double2* const Bv[2], double2* const Cm[2], int* const big[2], cudaStream_t st);
void launch_untranspose(int n_str, int nw, const double2* rT, double2* r, cudaStream_t st);
void launch_det_ratios(const PairTables& pt, int nw, int n_str_a, int n_str_b, const double2* ra,
                       const double2* rb, double2* out, cudaStream_t st);
void launch_sum_slots(int nw, const double2* part, int nslot, int slot0, int n, double2* out,
                      const double2* O0a, const double2* O0b, double2* ovlp, cudaStream_t st);
void launch_ref_ovlp(int nw, const double2* O0a, const double2* O0b, double2* out, cudaStream_t st);
void launch_cmat(const SpinTables& ta, const SpinTables& tb, int nw, const double2* wts_a, const double2* wts_b,
                 const void* Ba, const void* Bb, bool fp32, double2* Cm_a, double2* Cm_b, cudaStream_t st,
                 int* const big[2] = nullptr);
void launch_gt(const SpinTables& ta, const SpinTables& tb, int nw, int M, double2* const Gr[2], const double2* const Cm[2],
               const double2* R, double2* GT, long long ld, const long long off[2], bool minus_ref, cudaStream_t st);
void launch_rdm_scatter(const SpinTables& tb, int nw, int M, const double2* GT, long long ld, long long off, int spin,
                        double2* rdm, cudaStream_t st);

// k_energy.cu
void launch_gemm_zd(int Mr, int Nc, int K, const double2* A, long long lda, const double* B,
                    long long ldb, double2* C, long long ldc, cudaStream_t st);
size_t fepi_smem(const SpinTables& tb);
void launch_fepi(const SpinTables& tb, int nw, int M, int n_chol, const double2* F, long long ldf,
                 const double2* Gr, double2* v0, double2* xx, double2* Lact, double2* Xic,
                 cudaStream_t st);
// hl: the matrix of the Lambda_h part (h1, or h1 + J).
void launch_onebody(const SpinTables& ta, const SpinTables& tb, int nw, int M, const double* const h1[2],
                    const double2* const Gr[2], double2* const e1[2], double2* const Lh[2], cudaStream_t st,
                    const double* const hl[2]);
void launch_gamma_reduce(int nw, const int X[2], int n_chol, const double2* const v0[2], const double2* const xx[2],
                         const double2* const Lact[2], const double2* const Xic[2], const double2* const Lh[2],
                         double2* const Y[2], double2* scal, cudaStream_t st);
void launch_gram(int nw, int Xp, int Xq, int n_chol, const double2* P, const double2* Q, void* K,
                 bool fp32, cudaStream_t st);
int string_energy_blocks(const SpinTables& tb, int k);
size_t string_energy_smem(const SpinTables& tb, bool fp32);
int string_energy_slots(const SpinTables& tb);
void launch_string_energy(const SpinTables& ta, const SpinTables& tb, int nw, const double2* const wts[2],
                          const void* const B[2], const void* const K[2], const void* const Y[2], bool fp32,
                          double2* part, int nslot, int slot0, cudaStream_t st);
int pair_cross_slots(const PairTables& pt, bool use_runs = false);
// k_pair_y.cu: the opposite-spin term per beta string (mixed precision)
bool pair_y_ok(const SpinTables& ta, const SpinTables& tb);
int pair_y_slots(const SpinTables& tb);
void launch_pair_y(const SpinTables& ta, const SpinTables& tb, int nw, const float2* rfa, const float2* rfb,
                   const void* Ba, const void* Bb, const void* Kab, double2* part, int nslot, int slot0,
                   cudaStream_t st);
// ra, rb: the string ratios in the working precision (double2 in FP64 mode,
// their FP32 copies in mixed mode)
// use_runs: buckets with run_side != 0 take the runs form (k_pair_run.cu).
void launch_pair_cross(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int nw,
                       const void* ra, const void* rb, const void* Ba, const void* Bb,
                       const void* K, bool fp32, double2* part, int nslot, int slot0,
                       cudaStream_t st, bool use_runs = false);
// k_pair_run.cu
int pair_run_blocks(const PairTables& pt, int bidx);
size_t pair_run_smem(const SpinTables& ta, const SpinTables& tb, bool fp32);
void launch_pair_run(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int bidx, int ka, int kb,
                     int nw, const void* ra, const void* rb, const void* Ba, const void* Bb, const void* K, bool fp32,
                     double2* part, int nslot, int slot, cudaStream_t st);
void launch_final(int nw, const double2* part, int nslot, int nR, double e0, const double2* e1a,
                  const double2* e1b, const double2* scal, const double2* O0a, const double2* O0b,
                  double2* eloc, double2* ovlp, cudaStream_t st);

// tc_gemm.cu: 3xTF32 tensor-core GEMM C[m][n] = sum_k A[m][k] B[n][k] with
// A, B given as hi/lo TF32 parts, K-major with row pitch ld (elements).
struct TcOperand {
    const float* hi;
    const float* lo;
    long long ld;
};
// K is split over `splits` CTAs along grid.z; split z writes C + z * c_split_stride.
// bn: output tile width (128 or 256; 0 picks by Nc).
int tc_gemm_3xtf32(const TcOperand& A, const TcOperand& B, int Mr, int Nc, int K, float* C, long long ldc,
                   unsigned* err, cudaStream_t st, int splits = 1, long long c_split_stride = 0, int bn = 0);
// BF16 tensor-core GEMM C[m][n] = sum_k A[m][k] B[n][k] (FP32 accumulation;
// A, B row-major BF16 with K contiguous, K a multiple of 64).
// epi, ep: 0 plain; 1 and 2 the network layers' epilogues (tc_gemm.cu, EPI), with C,
// h and zin of row pitch ldc and ht [Nc][ldt].
struct NetEpi {
    const float* bias = nullptr;
    const float* zin = nullptr;
    __nv_bfloat16 *h = nullptr, *ht = nullptr;
    int ldt = 0, Bp = 0;
};
int tc_gemm_bf16(const void* A, long long lda, const void* B, long long ldb, int Mr, int Nc, int K, float* C,
                 long long ldc, unsigned* err, cudaStream_t st, int epi = 0, const NetEpi* ep = nullptr);
// part_rows: rows per (block, part) in the output (0: R; larger pads each
// part with zero rows). eye0 >= 0: columns [eye0, eye0 + 2 part_rows) hold
// two identity blocks on the real-part rows r < R (1 at column eye0 + r and
// eye0 + part_rows + r), zero on the imaginary-part rows.
void launch_split_complex_rows(int nb, int R, int Kg, int Kp, const double2* src, long long src_ld,
                               const int* cols, float* hi, float* lo, cudaStream_t st, int part_rows = 0,
                               int eye0 = -1);
void launch_split_real_rows(long long R, int Kg, int Kp, const double* src, long long src_ld, const int* cols,
                            float* hi, float* lo, cudaStream_t st);
// Slices of x[r][j] (r < R, j < n, FP64) into two column blocks of rows of
// pitch ld: hi/lo[r][k0 + j] = (h, m) and hi/lo[r][k0 + RB + j] = (q, s),
// h = tf32(x), m = tf32(x - h), q = tf32(x - h - m), s = tf32(x - h - m - q),
// so that h + m + q + s equals x to about 44 bits.
void launch_split_blocks(long long R, int n, int RB, int ld, int k0, const double* x, float* hi, float* lo,
                         cudaStream_t st);
void launch_pack_complex(int nw, int n, const float* C, long long ldc, int splits, long long split_stride,
                         const double* add, double2* out, long long ldo, cudaStream_t st);

// tc_dgemm.cu: FP64 products on the BF16 tensor cores (exact-integer split).
// An operand: the digit slices [8][rows][dg_k_padded(K)] of its rows and their
// exponents [rows]; batch entry z starts at row z * batch_rows (0: shared). A
// complex operand has two rows (real, imaginary part) per complex row.
struct DgOperand {
    const void* s = nullptr;
    const int* e = nullptr;
    int rows = 0;
    int batch_rows = 0;
};
// C[z c_batch + n c_n + m c_m] = mul sum_k A_z[m][k] B_z[n][k], m < Mr rows of
// A, n < Nc complex rows of B; acc (optional, same layout) = acc_in + C. With
// splits > 1 (batch must be 1) the contraction is divided and split z writes its
// part at z c_batch, for dg_sum_splits. gx >= 0: the rows of A and B stack gx
// alpha and gy beta entries, and the (alpha, alpha), (beta, beta) and (alpha,
// beta) blocks go to K[0], K[2], K[1] ([batch][rows][columns] each) instead of C.
// eye [Mr]: rows m with eye[m] >= 0 are written as unit vectors (1 at n = eye[m]); live
// [batch]: entries z with live[z] = 0 are written as zeros.
struct DgOut {
    int Mr = 0, Nc = 0, batch = 1, splits = 1;
    double2* C = nullptr;
    long long c_batch = 0, c_n = 0, c_m = 1;
    double2* acc = nullptr;
    const double2* acc_in = nullptr;
    double mul = 1.0;
    int gx = -1, gy = 0;
    double2* K[3] = {nullptr, nullptr, nullptr};
    const int* eye = nullptr;
    const double2* live = nullptr;
};
int dg_k_padded(int K);
size_t dg_row_bytes(int K);              // slices and exponent of one real row
int dg_splits(int Mr, int K);
// scale (optional): row r's elements 2 k and 2 k + 1 times scale[r / rows][k], a power
// of two (K / 2 of them).
void dg_slice_real(long long R, int K, const double* src, long long ld, void* S, int* ex, cudaStream_t st,
                   const double* scale = nullptr, int rows = 1);
void dg_slice_complex(long long R, int K, const double2* src, long long ld, void* S, int* ex, cudaStream_t st);
// Columns of src[z][k][c] (k < K, c < nc) as the operand rows z rows + row0 + c:
// mode 0 a left operand (Sa, length 2 K) and the matching complex right operand
// (Sb, two rows each), mode 1 the right operand alone, mode 2 the two parts as
// plain rows of length K (Sb).
void dg_slice_columns(int mode, int K, int nc, int batch, const double2* src, long long ld, long long src_batch,
                      int row0, int rows, void* Sa, int* ea, void* Sb, int* eb, cudaStream_t st);
int dg_gemm(const DgOperand& A, const DgOperand& B, const DgOut& o, int K, unsigned* err, cudaStream_t st);
void dg_sum_splits(int R, int Cc, int splits, const double2* part, double2* out, long long ldo, cudaStream_t st);

// tc_fepi.cu: the Cholesky contraction of the energy fused with its
// per-(walker, vector) epilogue (same outputs as tc_gemm_3xtf32 followed by
// launch_fepi_f32). A: split rows of dG[occ0][virt], part c of walker w at
// rows (2w + c) RB; B: split half-rotated Cholesky rows, vector g's at
// g NCf + [occ0 (N), zero (RB - N), particles (np)]; both pitch ld,
// contraction K. F0P: [n_chol][f0s], F0[j][col] = L_g[occ0_j][col] at
// g f0s + j NCP + col in the same column order, zero padded.
struct TcFepiPlan {
    int RB = 0, RW = 0, WPT = 0, NCf = 0, BN = 0, GPT = 0, BNe = 0, slot = 0, NCP = 0, f0s = 0;
    size_t smem = 0;
};
bool tc_fepi_plan(const SpinTables& tb, TcFepiPlan& p);
int tc_fepi_fused(const SpinTables& tb, const TcFepiPlan& p, int nw, int M, int n_chol, const float* a_hi,
                  const float* a_lo, const float* b_hi, const float* b_lo, int ld, int K, const double2* Gr,
                  const float* F0P, const double* c0, const double* x0, double2* v0, double2* xx,
                  float2* Lact, float2* Xic, unsigned* err, cudaStream_t st, bool traces);

// tc_ozaki.cu: the reference-determinant Cholesky sums of the mixed local
// energy in FP64 accuracy (exact-integer BF16 slices on the tensor cores).
// Constant operand of one spin: B = [V | 0 | W]^T sliced, V's N Kv rows padded
// with zero rows to a whole number of column tiles (NVp), NB = NVp + G rows.
struct OzConst {
    int N = 0, Kv = 0, G = 0, NK = 0, NVp = 0, NB = 0, NBp = 0, Kp = 0;   // V rows padded to NVp
    void* Bs = nullptr;   // [OZ_S][NBp][Kp] BF16
    int* eb = nullptr;    // [NBp] row exponents
};
// One spin's inputs to the per-walker reduction.
struct RefSpin {
    int N, M, Kv, nparts, Mpad;
    const double2* Gr;
    const int* virt;
    const double* JJ;     // [N Kv] J[v_r][o_j], J = sum_g (c0a_g + c0b_g) L_g
    const double* KK;     // [N Kv] (sum_g L_g P0 L_g)[v_r][o_j]
    const double* t1;     // [2 nw][G]
    const double2* part;  // [nparts][Mpad]
    double x0sum;         // sum_g x0_g of this spin
};
size_t oz_const_bytes(int N, int Kv, int G);
int oz_rows_padded(int nrow);
int oz_k_padded(int NK);
int oz_parts(int NB);                // partial-sum rows of a constant operand with NB rows
int oz_parts_for(int NK, int G);     // the same from N (M - N) and n_chol
int oz_slices();
// d_XT: [N Kv][G] FP64, XT[r N + l][g] = L_g[v_r][o_l]. Allocates out's arrays.
int oz_prepare_const(int N, int Kv, int G, const double* d_XT, OzConst& out, cudaStream_t st);
void oz_free_const(OzConst& c);
// One spin's walker rows: As [OZ_S][pad(2 nw)][Kp] BF16 scratch, ea [pad(2 nw)];
// written are part [oz_parts(NB)][pad(2 nw)] and t1 [2 nw][G].
struct OzSpin {
    const OzConst* K;
    const double2* Gr;
    const int* virt;
    void* As;
    int* ea;
    double2* part;
    double* t1;
};
int oz_both(const OzSpin in[2], int nw, int M, unsigned* err, cudaStream_t st);
// Also writes the walker parts t1a_g + t1b_g of V0_g as FP32 pairs v0w[w][g].
void launch_ref_reduce(int nw, int G, const RefSpin& a, const RefSpin& b, double C2sum, double2* scal,
                       float2* v0w, cudaStream_t st);

// k_debug.cu: E_I of sampled (walker, determinant) pairs.
struct DetRec {
    int w, a, b, ka, kb;   // walker, alpha and beta string, their levels
};
void launch_det_energy(int n, const DetRec* recs, int w0, int nw, const SpinTables& ta, const SpinTables& tb,
                       const void* Ba, const void* Bb, const void* Kaa, const void* Kbb, const void* Kab,
                       const void* Ya, const void* Yb, const double2* scal, const double2* e1a, const double2* e1b,
                       double e0, bool fp32, double2* out, cudaStream_t st);

// k_mixed.cu
size_t fepi_f32_smem(const SpinTables& tb);
void launch_fepi_f32(const SpinTables& tb, int nw, int M, int n_chol, const float* dF, long long ldf,
                     const double2* Gr, const float* F0T, const double* c0, const double* x0, double2* v0,
                     double2* xx, float2* Lact, float2* Xic, cudaStream_t st);
void launch_gamma_reduce_f32(int nw, const int X[2], int n_chol, const double2* const v0[2], const double2* const xx[2],
                             const float2* const Lact[2], const float2* const Xic[2], const double2* const Lh[2],
                             float2* const Y[2], double2* scal, cudaStream_t st, bool traces,
                             const float2* v0w = nullptr);
// K[w][x][y] = sum_g P[w][g][x] Q[w][g][y] (FP32) for up to three
// (P, Q, K) products of shapes Xp x Xq in one launch.
struct GramJob {
    int Xp, Xq;          // entries; P and Q rows have the pitch lam_pitch(X)
    const float2* P;
    const float2* Q;
    float2* K;
};
struct GramJobs {
    GramJob j[3];
};
void launch_gram_f32(int nw, int n_chol, const GramJobs& jobs, int nj, cudaStream_t st);
// tc_gram.cu: the same Gram matrices on the tensor cores (3xTF32, FP32
// accumulation in TMEM) for 2 X <= 256 per spin; returns 0 or -1.
// Rows first: T[w][2x + c][g] = part c of Lam[w][g][x] (FP32, Lam rows of the
// pitch lam_pitch(X)); then K_aa, K_bb, K_ab from Ta, Tb ([nw][X][X'] pairs).
// tc_gram needs n_chol a multiple of 4 and tc_gram_ok; returns 0 or -1.
bool tc_gram_ok(int Xa, int Xb);
void launch_gram_transpose(int nw, int n_chol, int X, const float2* Lam, float* T, cudaStream_t st);
int tc_gram(int nw, int n_chol, int Xa, int Xb, const float* Ta, const float* Tb, float2* Kaa, float2* Kbb,
            float2* Kab, unsigned* err, cudaStream_t st);

// k_batch.cu: per-determinant energy terms of many systems in one
// persistent launch.
struct BatchSys {
    SpinTables t[2];
    PairTables pt;
    const double2* r[2];
    const float2* rf[2];  // FP32 copies of r (mixed mode)
    const double2* wts[2];
    const void* B[2];
    const void* K[3];   // same-spin alpha, same-spin beta, opposite-spin Gram matrices
    const void* Y[2];
    double2* part;
    int nslot;
    int pad_;
};
struct BatchItem {
    int sys, w;
    int kind;           // 0: same-spin string block, 1: opposite-spin determinant block
    int spin;           // kind 0
    int ka, kb;         // level (kind 0: ka); level pair (kind 1)
    int blk, slot;      // block within the bucket, partial-sum slot
};
int launch_det_batched(const BatchSys* systems, const BatchItem* items, int n_items, unsigned* counter,
                       size_t smem, bool fp32, int grid, cudaStream_t st);

// mlp.cu
void launch_features(int nw, int M, int N, int n_core, int n_act, const int* pos0, const double2* Gr, float* feat,
                     int spin, cudaStream_t st);
void launch_features_rows(int nw, int M, int N, const double2* Gr, float* feat, long long ld, long long off,
                          cudaStream_t st);

// k_prop.cu: one phaseless propagation step (FP64).
void launch_sum_LL(int M, int G, const double* Lt, double* corr, cudaStream_t st);
void launch_prop_coef(int nw, int G, double dt, const double* x, const double2* vbias, double2* c, double2* expo,
                      cudaStream_t st);
int launch_apply_rows(int nw, int M, int N, const double2* A, long long a_stride, const double* Ar,
                      const double2* in, double2* out, double2* acc, double scale, cudaStream_t st);
void launch_prop_weight(int nw, const double2* o_old, const double2* o_new, const double2* expo, double* w,
                        double2* ratio, cudaStream_t st);
int launch_qr_mgs(int nw, int M, int N, double2* phi, unsigned* err, cudaStream_t st);

// k_pair.cu: the opposite-spin term with both levels compiled in (ka + kb <=
// 8); false for other level pairs.
bool launch_pair_cross2(int ka, int kb, bool fp32, dim3 grid, size_t smem, const SpinTables& ta, const SpinTables& tb,
                        const PairTables& pt, int lo, int n, const void* ra, const void* rb, const void* Ba,
                        const void* Bb, const void* K, double2* part, int nslot, int slot, cudaStream_t st);
// All level pairs (ka + kb <= 6, no runs) in one launch where that is worth it;
// false if the caller has to launch them one by one.
bool launch_pair_cross_all(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int nw, const void* ra,
                           const void* rb, const void* Ba, const void* Bb, const void* K, bool fp32, double2* part,
                           int nslot, int slot0, cudaStream_t st, bool use_runs);
