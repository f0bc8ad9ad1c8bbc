// Reference inverse, excitation-string minors and CI weights: the overlap
// part of the generalized-Wick evaluation (Sec. III "Implementation":
// get_dets), plus the cofactor accumulation behind the mixed Green's
// function (reduce_CI) and its rank-n_p update.
#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "minor_lu.cuh"

// ------------------------------------------------------------------------
// Reference determinant per (walker, spin): S = D0^dag phi = phi[occ0, :]
// (Sec. II A overlap of two determinants). Gauss-Jordan elimination with partial
// pivoting (by the larger of |Re|, |Im|) in FP64 gives O0 = det S and S^-1; then
//   Gr[j][r]  = (phi S^-1)[r][j] = G[occ0_j][r]   (G = G0^T, G0 = Theta D0^dag)
//               (rows r in occ0 of phi are S itself, so there Gr is exactly
//               the identity and is written, not computed)
//   Gact[h][p] = G[H_h][P_p]                       (active hole x particle block)
// One block per (walker, spin). A walker whose |det S| falls below 1e-14 times
// the product of the column norms of S is flagged singular.
//
// All N^2 entries of a step are independent (an LU followed by column solves left
// one thread per column with a serial chain: 35 us for a 5 x 5 block, and two
// thirds of the inversion's FP64 operations on one warp). The product with phi,
// (M - N) N^2 complex FMAs and most of the FP64 work at larger N, runs on the
// tensor cores from ref_dg_use on (S^-1 then goes out to Sinv), else here. Its operands
// are rounded to 56 bits of a row's largest value over the walker's columns, and G does
// not depend on the columns' scales: so column k of phi enters as phi_k 2^-e_k, |phi_k|
// < 2^e_k, and row k of S^-1 as 2^e_k of it (exact; without it columns 1e8 apart left 9
// digits of G; 0.012 ms of the copper-oxo time below).
// Measured, both spins: N = 5, 16 walkers 70 -> 21 us; iron-sulfur (N = 30, M = 160)
// 640 walkers 1.95 -> 1.00 ms, 64 walkers 0.81 -> 0.23 ms; copper-oxo (N = 16, M =
// 108) 640 walkers 0.73 -> 0.37 ms.
struct RefIn {
    const double2* phi;     // [nw][M][N]
    int N, nh, np;
    const int *occ0, *pos0, *hole_pos, *part_orb;
    double2 *Gr, *O0;
    double2 *Gact, *GactT;  // [nw][nh np], [nh np][nw] (either may be NULL)
    double2* Sinv;          // [nw][N][N], or NULL: form Gr and the active block here
    double* cs;             // [nw][N] with Sinv: the columns' scales
};
struct RefArgs { RefIn s[2]; };

__global__ void __launch_bounds__(256)
k_ref(const __grid_constant__ RefArgs args, int M, unsigned* err)
{
    extern __shared__ double2 S[];   // [N][N], overwritten by its inverse (columns permuted)
    __shared__ double2 prow[MSD_NMAX], pcol[MSD_NMAX], pinv;
    __shared__ int piv[MSD_NMAX], col[MSD_NMAX];
    __shared__ double cn[MSD_NMAX];
    __shared__ int ce[MSD_NMAX];     // with Sinv: largest magnitude (high word), then exponent of phi's columns
    __shared__ int singular;
    const RefIn& R = args.s[blockIdx.y];
    const int w = blockIdx.x, nw = gridDim.x, N = R.N;
    const int t = threadIdx.x, nt = blockDim.x;
    const double2* ph = R.phi + (size_t)w * M * N;

    for (int e = t; e < N * N; e += nt) S[e] = ph[(size_t)R.occ0[e / N] * N + e % N];
    if (t == 0) singular = 0;
    if (R.Sinv)
        for (int j = t; j < N; j += nt) ce[j] = 0;
    __syncthreads();
    if (R.Sinv) {
        for (int e = t; e < M * N; e += nt) atomicMax(&ce[e % N], mag_key(ph[e]));
        __syncthreads();
    }
    for (int j = t; j < N; j += nt) {
        if (R.Sinv) {
            ce[j] = min(1000, max(-1000, (ce[j] >> 20) - 1022));
            R.cs[(size_t)w * N + j] = ldexp(1.0, -ce[j]);
        }
        double a = 0;
        for (int i = 0; i < N; ++i) a += S[i * N + j].x * S[i * N + j].x + S[i * N + j].y * S[i * N + j].y;
        cn[j] = sqrt(a);
    }
    double2 det = cz(1, 0);   // thread 0
    for (int k = 0; k < N; ++k) {
        if (t < 32) {
            int best = -1, bi = k;
            for (int i = k + t; i < N; i += 32) {
                const int v = mag_key(S[i * N + k]);
                if (v > best) { best = v; bi = i; }
            }
            const int top = __reduce_max_sync(0xffffffffu, best);
            bi = __reduce_min_sync(0xffffffffu, best == top ? bi : 0x7fffffff);
            if (t == 0) {
                const double2 p = S[bi * N + k];
                piv[k] = bi;
                if (p.x == 0.0 && p.y == 0.0) singular = 1;
                det = cmul(det, p);
                if (bi != k) det = cz(-det.x, -det.y);
                pinv = crecip(p);
            }
        }
        __syncthreads();
        if (singular) break;
        const int p = piv[k];
        const double2 pi = pinv;
        // row p to the pivot place, scaled; row k to row p; column k set aside
        for (int j = t; j < N; j += nt) {
            const double2 a = S[p * N + j];
            prow[j] = j == k ? pi : cmul(a, pi);
            pcol[j] = j == p ? S[k * N + k] : S[j * N + k];
        }
        __syncthreads();
        for (int e = t; e < N * N; e += nt) {
            const int i = e / N, j = e - i * N;
            if (i == k) continue;
            const double2 f = pcol[i];
            const double2 a = j == k ? cz(0, 0) : i == p ? S[k * N + j] : S[e];
            S[e] = cfms(f, prow[j], a);
        }
        __syncthreads();
        for (int j = t; j < N; j += nt) S[k * N + j] = prow[j];
        // the pivot search below reads rows > k of column k + 1 only
        if (t < 32) __syncwarp();
    }
    if (t == 0) {
        double nrm = 1;
        if (!singular) {
            for (int k = 0; k < N; ++k) { nrm *= cn[k]; col[k] = k; }
            if (!(sqrt(det.x * det.x + det.y * det.y) > 1e-14 * nrm)) singular = 1;
            // the row exchanges, undone as column exchanges in reverse order
            for (int k = N - 1; k >= 0; --k) { const int c = col[k]; col[k] = col[piv[k]]; col[piv[k]] = c; }
        }
        if (singular) { det = cz(0, 0); atomicOr(err, MSD_DEV_ERR_SINGULAR); }
        R.O0[w] = det;
    }
    __syncthreads();
    const int nh = R.nh, np = R.np;
    double2* gr = R.Gr + (size_t)w * N * M;
    if (R.Sinv) {
        double2* out = R.Sinv + (size_t)w * N * N;
        for (int e = t; e < N * N; e += nt)   // row k: of S^-1, so of the walker's column k
            out[e] = singular ? cz(0, 0) : cscale(S[e - e % N + col[e % N]], ldexp(1.0, ce[e / N]));
        return;
    }
    for (int e = t; e < M * N; e += nt) {
        const int r = e / N, j = e - r * N, q = R.pos0[r];
        double2 a = cz(0, 0);
        if (!singular) {
            if (q >= 0) {
                a = cz(q == j ? 1.0 : 0.0, 0.0);
            } else {
                const double2* pr = ph + (size_t)r * N;
                const int c = col[j];
                for (int k = 0; k < N; ++k) a = cfma(pr[k], S[k * N + c], a);
            }
        }
        gr[(size_t)j * M + r] = a;
    }
    __syncthreads();
    for (int e = t; e < nh * np; e += nt) {
        const double2 a = gr[(size_t)R.hole_pos[e / np] * M + R.part_orb[e % np]];
        if (R.Gact) R.Gact[(size_t)w * nh * np + e] = a;
        if (R.GactT) R.GactT[(size_t)e * nw + w] = a;
    }
}

// The active block from the rows of G, in both orders (walkers contiguous in
// GactT), for blockIdx.y of two spins.
__global__ void __launch_bounds__(256) k_gact(const __grid_constant__ RefArgs args, int M, int nw)
{
    const RefIn& R = args.s[blockIdx.y];
    const int X = R.nh * R.np;
    const long long e = blockIdx.x * 256ll + threadIdx.x;
    if (e >= (long long)X * nw) return;
    const int x = (int)(e / nw), w = (int)(e - (long long)x * nw);
    const double2 a = R.Gr[((size_t)w * R.N + R.hole_pos[x / R.np]) * M + R.part_orb[x % R.np]];
    if (R.Gact) R.Gact[(size_t)w * X + x] = a;
    if (R.GactT) R.GactT[e] = a;
}

// The product with phi runs on the tensor cores from this many complex FMAs per
// walker on: below, its three launches take longer than the FP64 units (16e3
// complex FMAs are about 17 us of one SM's).
bool ref_dg_use(int M, int N) { return (long long)(M - N) * N * N >= 16384; }
size_t ref_dg_bytes(int M, int N)
{
    return ref_dg_use(M, N) ? sizeof(double2) * (size_t)N * N + sizeof(double) * N + dg_row_bytes(2 * N) * (M + 2 * (size_t)N)
                            : 0;
}

int launch_refs(const RefSpinIn* in, int n_spin, int nw, int M, unsigned* err, cudaStream_t st)
{
    RefArgs a;
    int Nmax = 1, X = 0;
    bool dg = false;
    for (int s = 0; s < n_spin; ++s) {
        const SpinTables& T = *in[s].T;
        a.s[s] = RefIn{in[s].phi, T.N, T.nh, T.np, T.occ0, T.pos0, T.hole_pos, T.part_orb, in[s].Gr, in[s].O0, in[s].Gact,
                       in[s].GactT, in[s].Sinv, in[s].cs};
        Nmax = Nmax > T.N ? Nmax : T.N;
        X = X > T.nh * T.np ? X : T.nh * T.np;
        dg = dg || in[s].Sinv;
    }
    const size_t smem = sizeof(double2) * Nmax * Nmax;
    if (smem > 40 * 1024) cudaFuncSetAttribute(k_ref, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // a block's step updates N^2 entries: no more warps than it has work for
    const int threads = Nmax <= 8 ? 64 : Nmax <= 16 ? 128 : 256;
    k_ref<<<dim3(nw, n_spin), threads, smem, st>>>(a, M, err);
    msd_note_launch();
    if (!dg) return 0;
    for (int s = 0; s < n_spin; ++s) {
        if (!in[s].Sinv) continue;
        const int N = in[s].T->N;
        dg_slice_real((long long)nw * M, 2 * N, (const double*)in[s].phi, 2 * N, in[s].sa, in[s].ea, st, in[s].cs, M);
        dg_slice_columns(1, N, N, nw, in[s].Sinv, N, (long long)N * N, 0, N, nullptr, nullptr, in[s].sb, in[s].eb, st);
        DgOut o;
        o.Mr = M; o.Nc = N; o.batch = nw;
        o.C = in[s].Gr; o.c_batch = (long long)N * M; o.c_n = M; o.c_m = 1;
        o.eye = in[s].T->pos0;
        o.live = in[s].O0;   // 0 for a singular walker: zero rows, as k_ref writes them
        if (dg_gemm({in[s].sa, in[s].ea, nw * M, M}, {in[s].sb, in[s].eb, 2 * N * nw, 2 * N}, o, 2 * N, err, st)) return -1;
    }
    if (X > 0 && (in[0].Gact || in[0].GactT)) {
        // spins whose product ran in k_ref have their block already; writing it
        // again is the same values
        k_gact<<<dim3((unsigned)(((long long)X * nw + 255) / 256), n_spin), 256, 0, st>>>(a, M, nw);
        msd_note_launch();
    }
    return 0;
}

// ------------------------------------------------------------------------
// Excitation strings of level K for one spin with their FP64 inverse minors
// by an LU of its own, for FP64 energies and force bias of trials whose sub-minors are
// far more than their strings (all else: k_minors.cu):
// A[i][j] = G[h_i][p_j] (a K x K minor of G); r = sign * det A, the overlap ratio
// <D_s|phi>/<D_0|phi> of the string's spin sector, and B = A^-1 for the Green's-function
// and energy terms. One thread per (walker, string); the walker's active block lives in
// shared memory.
// String s = bucket[K] + sl of walker w, its active block in shared memory (gs).
template <int K>
__device__ __forceinline__ void string_lu(const SpinTables& tb, int nw, int w, int sl, const double2* gs, double2* r,
                                          double2* rT, double2* Bout)
{
    const int ns = tb.bucket[K + 1] - tb.bucket[K], s = tb.bucket[K] + sl;
    const uint4 rec = tb.str_hp[s];
    const double2 det = minor_lu<K>(tb.str_sign[s], [&](int i, int j) { return gs[rec_h(rec, i) * tb.np + rec_p(rec, j)]; },
                                    Bout + (size_t)tb.b_off[K] + ((size_t)w * ns + sl) * b_stride(K));
    if (r) r[(size_t)w * tb.n_str + s] = det;
    rT[(size_t)s * nw + w] = det;
}

template <int K>
__global__ void __launch_bounds__(128)
k_strings(SpinTables tb, int nw, const double2* __restrict__ Gact, double2* __restrict__ r, double2* __restrict__ rT,
          double2* __restrict__ Bout)
{
    __shared__ double2 g[MSD_XMAX];
    const int w = blockIdx.y;
    const int X = tb.nh * tb.np;
    for (int e = threadIdx.x; e < X; e += blockDim.x) g[e] = Gact[(size_t)w * X + e];
    __syncthreads();
    const int sl = blockIdx.x * blockDim.x + threadIdx.x;
    if (sl < tb.bucket[K + 1] - tb.bucket[K]) string_lu<K>(tb, nw, w, sl, g, r, rT, Bout);
}

template <int K>
static void launch_strings_k(const SpinTables& tb, int nw, const double2* Gact, double2* r, double2* rT, void* B,
                             cudaStream_t st)
{
    const int ns = tb.bucket[K + 1] - tb.bucket[K];
    if (ns <= 0) return;
    dim3 grid((ns + 127) / 128, nw);
    k_strings<K><<<grid, 128, 0, st>>>(tb, nw, Gact, r, rT, (double2*)B);
    msd_note_launch();
}

// Reference string (level 0): ratio 1.
__global__ void k_ref_string(int nw, int n_str, double2* r, double2* rT)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < nw) r[(size_t)w * n_str] = rT[w] = cz(1, 0);
}

void launch_strings(const SpinTables& tb, int nw, const double2* Gact, double2* r, double2* rT, void* B, cudaStream_t st,
                    const TimerHook& th)
{
    if (tb.bucket[1] > tb.bucket[0]) {
        th.begin("k_ref_string", st);
        k_ref_string<<<(nw + 127) / 128, 128, 0, st>>>(nw, tb.n_str, r, rT); msd_note_launch();
        th.end(st);
    }
    th.begin("k_strings", st);
    launch_strings_k<1>(tb, nw, Gact, r, rT, B, st);
    launch_strings_k<2>(tb, nw, Gact, r, rT, B, st);
    launch_strings_k<3>(tb, nw, Gact, r, rT, B, st);
    launch_strings_k<4>(tb, nw, Gact, r, rT, B, st);
    launch_strings_k<5>(tb, nw, Gact, r, rT, B, st);
    launch_strings_k<6>(tb, nw, Gact, r, rT, B, st);
    th.end(st);
}

// Walkers whose active block has an entry above 1 in magnitude (the larger of |Re|, |Im|):
// big[w]. GT [nh np][nw], both spins. A block takes 32 walkers.
struct LargeArgs {
    const double2* GT[2];
    int X[2];
    int* big[2];
};
__global__ void __launch_bounds__(256) k_large(const __grid_constant__ LargeArgs a, int nw)
{
    __shared__ int red[8][32];
    const int s = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, w = blockIdx.x * 32 + lane;
    int m = 0;
    if (w < nw)
        for (int x = warp; x < a.X[s]; x += 8) m = max(m, mag_key(a.GT[s][(size_t)x * nw + w]));
    red[warp][lane] = m;
    __syncthreads();
    if (warp || w >= nw) return;
    for (int q = 1; q < 8; ++q) m = max(m, red[q][lane]);
    a.big[s][w] = m >= 0x3ff00000;
}

// Ratios and inverse minors of the walkers marked by k_large, by LU, over what the
// expansions left (k_minors.cu). A minor's LU is the exact one of a nearby block, so G - G
// B G keeps its cancellation; inverse entries as ratios of separately rounded minors do
// not, and lose the square of the block's magnitude (rank-1 part of 30: density matrix
// 4e-13 against 3e-14, of 1e4: 4e-8 against 8e-12; entries up to 1: alike). A block takes
// 128 strings of a level; the blocks of a column share the marked walkers. Levels 1 to 4
// and 5, 6 apart: 134 and 255 registers. None marked: 3 us a launch; all of 640 copper-oxo
// walkers marked: density matrix 2.2 -> 6.2 ms (6.3 with an LU for every walker).
struct StringsLargeArgs {
    SpinTables t[2];
    const double2* Gact[2];
    const int* big[2];
    double2 *r[2], *rT[2], *B[2];
    int blk[2][MSD_KMAX + 2];   // first block of each level
};
template <int LO, int HI>
__global__ void __launch_bounds__(128) k_strings_large(const __grid_constant__ StringsLargeArgs a, int nw)
{
    const int spin = blockIdx.z, t = threadIdx.x;
    const SpinTables& tb = a.t[spin];
    if ((int)blockIdx.x >= a.blk[spin][HI + 1]) return;
    __shared__ double2 g[MSD_XMAX];
    __shared__ unsigned marks[32];
    int k = LO;
    while ((int)blockIdx.x >= a.blk[spin][k + 1]) ++k;
    const int X = tb.nh * tb.np, sl = ((int)blockIdx.x - a.blk[spin][k]) * 128 + t;
    const bool on = sl < tb.bucket[k + 1] - tb.bucket[k];
    unsigned turn = 0;
    for (int w0 = 0; w0 < nw; w0 += 1024) {
        __syncthreads();
        for (int q = t >> 5; q < 32; q += 4) {
            const int w = w0 + q * 32 + (t & 31);
            const unsigned m = __ballot_sync(0xffffffffu, w < nw && a.big[spin][w]);
            if ((t & 31) == 0) marks[q] = m;
        }
        __syncthreads();
        for (int q = 0; q < 32; ++q)
            for (unsigned m = marks[q]; m; m &= m - 1) {
                if (turn++ % gridDim.y != blockIdx.y) continue;
                const int w = w0 + q * 32 + __ffs(m) - 1;
                __syncthreads();
                for (int e = t; e < X; e += 128) g[e] = a.Gact[spin][(size_t)w * X + e];
                __syncthreads();
                if (!on) continue;
                auto lu = [&](auto level) {
                    constexpr int K = decltype(level)::value;
                    if constexpr (LO <= K && K <= HI)
                        if (k == K) string_lu<K>(tb, nw, w, sl, g, a.r[spin], a.rT[spin], a.B[spin]);
                };
                lu(std::integral_constant<int, 1>{});
                lu(std::integral_constant<int, 2>{});
                lu(std::integral_constant<int, 3>{});
                lu(std::integral_constant<int, 4>{});
                lu(std::integral_constant<int, 5>{});
                lu(std::integral_constant<int, 6>{});
            }
    }
}

// r may be NULL (both).
void launch_strings_large(const SpinTables& ta, const SpinTables& tb, int nw, double2* const GT[2], double2* const Gact[2],
                          int* const big[2], double2* const r[2], double2* const rT[2], void* const B[2], cudaStream_t st)
{
    LargeArgs l;
    StringsLargeArgs a;
    const SpinTables* T[2] = {&ta, &tb};
    for (int s = 0; s < 2; ++s) {
        l.GT[s] = GT[s]; l.X[s] = T[s]->nh * T[s]->np; l.big[s] = big[s];
        a.t[s] = *T[s]; a.Gact[s] = Gact[s]; a.big[s] = big[s];
        a.r[s] = r[s]; a.rT[s] = rT[s]; a.B[s] = (double2*)B[s];
    }
    k_large<<<dim3((nw + 31) / 32, 2), 256, 0, st>>>(l, nw);
    msd_note_launch();
    auto go = [&](auto kern, int lo, int hi) {
        int nb = 0;
        for (int s = 0; s < 2; ++s) {
            for (int k = 0; k <= lo; ++k) a.blk[s][k] = 0;
            for (int k = lo; k <= hi; ++k)
                a.blk[s][k + 1] = a.blk[s][k] + (T[s]->bucket[k + 1] - T[s]->bucket[k] + 127) / 128;
            nb = nb > a.blk[s][hi + 1] ? nb : a.blk[s][hi + 1];
        }
        if (nb <= 0) return;
        // columns enough to fill the GPU when many walkers are marked
        const int cols = nb >= 512 ? 4 : nb >= 128 ? 16 : 64;
        kern<<<dim3(nb, nw < cols ? nw : cols, 2), 128, 0, st>>>(a, nw);
        msd_note_launch();
    };
    go(k_strings_large<1, 4>, 1, 4);
    go(k_strings_large<5, 6>, 5, 6);
}

// ------------------------------------------------------------------------
// Per-determinant ratios r_I = r_a(I) * r_b(I) in the caller's order.
__global__ void k_det_ratios(PairTables pt, int n_str_a, int n_str_b, const double2* __restrict__ ra,
                             const double2* __restrict__ rb, double2* __restrict__ out)
{
    const int w = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pt.n_det) return;
    out[(size_t)w * pt.n_det + pt.det_index[i]] =
        cmul(ra[(size_t)w * n_str_a + pt.a[i]], rb[(size_t)w * n_str_b + pt.b[i]]);
}

void launch_det_ratios(const PairTables& pt, int nw, int n_str_a, int n_str_b, const double2* ra,
                       const double2* rb, double2* out, cudaStream_t st)
{
    dim3 grid((pt.n_det + 255) / 256, nw);
    k_det_ratios<<<grid, 256, 0, st>>>(pt, n_str_a, n_str_b, ra, rb, out); msd_note_launch();
}

// Sum of partial slots [slot0, slot0 + n) per walker -> out[w] (and
// O_T = O0a * O0b * sum when ovlp is given). One warp per walker.
__global__ void k_sum_slots(int nw, const double2* __restrict__ part, int nslot, int slot0, int n,
                            double2* __restrict__ out, const double2* __restrict__ O0a,
                            const double2* __restrict__ O0b, double2* __restrict__ ovlp)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= nw) return;
    const double2 a = warp_sum_slots(part + (size_t)w * nslot + slot0, n, lane);
    if (lane) return;
    if (out) out[w] = a;
    if (ovlp) ovlp[w] = cmul(cmul(O0a[w], O0b[w]), a);
}

void launch_sum_slots(int nw, const double2* part, int nslot, int slot0, int n, double2* out,
                      const double2* O0a, const double2* O0b, double2* ovlp, cudaStream_t st)
{
    k_sum_slots<<<(nw + 3) / 4, 128, 0, st>>>(nw, part, nslot, slot0, n, out, O0a, O0b, ovlp); msd_note_launch();
}

// ------------------------------------------------------------------------
// Cofactor accumulation (reduce_CI): per (walker, spin)
//   Cm[p][h] = sum_s w_s r_s B_s[i][j]  at (p_i, h_j) = (p, h)
// (wts holds the products r_s w_s).
// One block per walker. The k^2 entries of one string's minor land on
// distinct (p, h), so a group of lanes takes a whole string at once and adds
// its entries into the group's own shared-memory copy of Cm with plain
// read-modify-writes: B is read in its stored order (coalesced) and nothing
// is atomic. Strings with k^2 <= 16 go two to a warp (half-warp groups),
// longer ones one to a warp. Each group takes its strings in ascending order
// and the copies are summed in a fixed order, so the result does not depend
// on scheduling. Products and the per-copy sums are in T (double in FP64
// mode, float in mixed mode); the copies are summed in double.
#define CMAT_COPIES 16
template <typename T, int GS, int EPL, int U>
__device__ __forceinline__ void cmat_level(T* __restrict__ a, int g, int ng, int l, int kk, int kst, int ns, int s0,
                                           const T* __restrict__ B, const uint8_t* __restrict__ xt,
                                           const double2* __restrict__ ww)
{
    for (int base = 0; base < ns; base += ng * U) {
        T vr[U][EPL], vi[U][EPL];
        int vx[U][EPL];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int sl = base + u * ng + g;
            double2 f = cz(0, 0);
            if (sl < ns) f = ww[s0 + sl];
            const T fr = (T)f.x, fi = (T)f.y;
#pragma unroll
            for (int q = 0; q < EPL; ++q) {
                const int e = l + q * GS;
                vx[u][q] = -1;
                vr[u][q] = 0;
                vi[u][q] = 0;
                if (sl < ns && e < kk) {
                    const size_t o = (size_t)sl * kk + e, ob = (size_t)sl * kst + e;
                    const T br = B[2 * ob], bi = B[2 * ob + 1];
                    vx[u][q] = xt[o];
                    vr[u][q] = fr * br - fi * bi;
                    vi[u][q] = fr * bi + fi * br;
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
#pragma unroll
            for (int q = 0; q < EPL; ++q)
                if (vx[u][q] >= 0) {
                    a[2 * vx[u][q]] += vr[u][q];
                    a[2 * vx[u][q] + 1] += vi[u][q];
                }
            __syncwarp();   // the group's next string may share entries with this one
        }
    }
}

template <typename T>
__device__ __forceinline__ void cmat_walker(const SpinTables& tb, int w, const double2* __restrict__ wts,
                                            const void* __restrict__ Bin, double2* __restrict__ Cm, T* accp, bool add)
{
    T (*acc)[2 * MSD_XMAX] = reinterpret_cast<T (*)[2 * MSD_XMAX]>(accp);
    const int X = tb.nh * tb.np;
    for (int e = threadIdx.x; e < CMAT_COPIES * 2 * MSD_XMAX; e += blockDim.x) accp[e] = 0;
    __syncthreads();
    const T* Bb = reinterpret_cast<const T*>(Bin);
    const double2* ww = wts + (size_t)w * tb.n_str;
    for (int k = 1; k <= MSD_KMAX; ++k) {
        const int s0 = tb.bucket[k], ns = tb.bucket[k + 1] - s0, kk = k * k;
        if (ns == 0) continue;
        const T* B = Bb + 2 * ((size_t)tb.b_off[k] + (size_t)w * ns * b_stride(k));
        const uint8_t* xt = tb.cmx + tb.cmx_off[k];
        if (kk <= 16)
            cmat_level<T, 16, 1, 3>(acc[threadIdx.x >> 4], threadIdx.x >> 4, 16, threadIdx.x & 15, kk, b_stride(k), ns, s0, B, xt,
                                    ww);
        else if (kk <= 32)
            cmat_level<T, 32, 1, 3>(acc[(threadIdx.x >> 5) * 2], threadIdx.x >> 5, 8, threadIdx.x & 31, kk, b_stride(k), ns, s0, B,
                                    xt, ww);
        else
            cmat_level<T, 32, 2, 3>(acc[(threadIdx.x >> 5) * 2], threadIdx.x >> 5, 8, threadIdx.x & 31, kk, b_stride(k), ns, s0, B,
                                    xt, ww);
    }
    __syncthreads();
    for (int x = threadIdx.x; x < X; x += blockDim.x) {
        double re = 0, im = 0;
        for (int q = 0; q < CMAT_COPIES; ++q) { re += (double)acc[q][2 * x]; im += (double)acc[q][2 * x + 1]; }
        double2* o = Cm + (size_t)w * X + x;
        *o = add ? cadd(*o, cz(re, im)) : cz(re, im);
    }
}

// Both spins in one grid (blockIdx.y = spin), so the two spins' blocks fill
// the machine together. big (may be NULL): only the walkers marked there, added to Cm.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 3)
k_cmat(SpinTables ta, SpinTables tb, const double2* __restrict__ wts_a, const double2* __restrict__ wts_b,
       const void* __restrict__ Ba, const void* __restrict__ Bb, double2* __restrict__ Cm_a,
       double2* __restrict__ Cm_b, const int* __restrict__ big_a, const int* __restrict__ big_b)
{
    __shared__ T acc[CMAT_COPIES][2 * MSD_XMAX];
    const int* big = blockIdx.y == 0 ? big_a : big_b;
    if (big && !big[blockIdx.x]) return;
    if (blockIdx.y == 0) {
        if (ta.nh * ta.np > 0) cmat_walker<T>(ta, blockIdx.x, wts_a, Ba, Cm_a, &acc[0][0], big != nullptr);
    } else {
        if (tb.nh * tb.np > 0) cmat_walker<T>(tb, blockIdx.x, wts_b, Bb, Cm_b, &acc[0][0], big != nullptr);
    }
}

void launch_cmat(const SpinTables& ta, const SpinTables& tb, int nw, const double2* wts_a, const double2* wts_b,
                 const void* Ba, const void* Bb, bool fp32, double2* Cm_a, double2* Cm_b, cudaStream_t st,
                 int* const big[2])
{
    const int *ga = big ? big[0] : nullptr, *gb = big ? big[1] : nullptr;
    if (ta.nh * ta.np <= 0 && tb.nh * tb.np <= 0) return;
    const dim3 grid(nw, 2);
    if (fp32) k_cmat<float><<<grid, 256, 0, st>>>(ta, tb, wts_a, wts_b, Ba, Bb, Cm_a, Cm_b, ga, gb);
    else k_cmat<double><<<grid, 256, 0, st>>>(ta, tb, wts_a, wts_b, Ba, Bb, Cm_a, Cm_b, ga, gb);
    msd_note_launch();
}

// ------------------------------------------------------------------------
// Rows of the mixed Green's function G_T (Eq. 7 numerator), per (walker,
// spin), restricted to the rows that can be non-zero (occ0 then P):
//   Y[p][c] = sum_h Cm[p][h] G[H_h][c]
//   G_T[occ0_l][c] = G[occ0_l][c] - sum_p G[occ0_l][P_p] Y[p][c] / R
//   G_T[P_p][c]    = Y[p][c] / R
// Written to GT[w][row][c] with row stride M, at column offset `off` of a
// row of length ld (both spins are concatenated per walker). With
// minus_ref the reference part D0 D0^T (ones at (occ0_l, occ0_l)) is
// subtracted, for the mixed path that adds its contraction in FP64.
#define GT_COLS 16   // output columns per block
struct GtArgs {
    SpinTables t[2];
    const double2 *Gr[2], *Cm[2];
    long long off[2];
};
__global__ void __launch_bounds__(256)
k_gt(const __grid_constant__ GtArgs a, int M, const double2* __restrict__ Rsum, double2* __restrict__ GT, long long ld,
     int minus_ref)
{
    __shared__ double2 cm[MSD_XMAX];
    __shared__ double2 y[MSD_XMAX * GT_COLS];   // [np][GT_COLS columns]
    const int s = blockIdx.z;
    const SpinTables& tb = a.t[s];
    const int w = blockIdx.y;
    const int c0 = blockIdx.x * GT_COLS;
    const int N = tb.N, nh = tb.nh, np = tb.np;
    const double2* gr = a.Gr[s] + (size_t)w * N * M;
    for (int e = threadIdx.x; e < nh * np; e += blockDim.x) cm[e] = a.Cm[s][(size_t)w * nh * np + e];
    __syncthreads();
    const double2 R = Rsum[w];
    const double2 iR = cdiv(cz(1, 0), R);
    for (int e = threadIdx.x; e < np * GT_COLS; e += blockDim.x) {
        const int p = e / GT_COLS, c = c0 + e % GT_COLS;
        double2 v = cz(0, 0);
        if (c < M)
            for (int h = 0; h < nh; ++h) v = cfma(cm[p * nh + h], gr[(size_t)tb.hole_pos[h] * M + c], v);
        y[e] = cmul(v, iR);
    }
    __syncthreads();
    double2* out = GT + (size_t)w * ld + a.off[s];
    for (int e = threadIdx.x; e < (N + np) * GT_COLS; e += blockDim.x) {
        const int x = e / GT_COLS, c = c0 + e % GT_COLS;
        if (c >= M) continue;
        double2 v;
        if (x < N) {
            v = gr[(size_t)x * M + c];
            for (int p = 0; p < np; ++p) v = cfms(gr[(size_t)x * M + tb.part_orb[p]], y[p * GT_COLS + e % GT_COLS], v);
            if (minus_ref && c == tb.occ0[x]) v.x -= 1.0;   // G_T - D0 D0^T
        } else {
            v = y[(x - N) * GT_COLS + e % GT_COLS];
        }
        out[(size_t)x * M + c] = v;
    }
}

// Both spins; spin s's rows go to column off[s] of a walker's row of GT.
void launch_gt(const SpinTables& ta, const SpinTables& tb, int nw, int M, double2* const Gr[2], const double2* const Cm[2],
               const double2* R, double2* GT, long long ld, const long long off[2], bool minus_ref, cudaStream_t st)
{
    GtArgs a;
    a.t[0] = ta; a.t[1] = tb;
    for (int s = 0; s < 2; ++s) { a.Gr[s] = Gr[s]; a.Cm[s] = Cm[s]; a.off[s] = off[s]; }
    k_gt<<<dim3((M + GT_COLS - 1) / GT_COLS, nw, 2), 256, 0, st>>>(a, M, R, GT, ld, minus_ref ? 1 : 0);
    msd_note_launch();
}

// The mixed one-body density matrix as full M x M matrices per walker and
// spin: rdm[w][spin][orb(x)][c] = GT[w][off + x M + c] for the rows x of G_T
// (occ0, then the particles); the caller zeroes the other rows.
__global__ void k_rdm_scatter(SpinTables tb, int M, const double2* __restrict__ GT, long long ld, long long off,
                              int spin, double2* __restrict__ rdm)
{
    const int x = blockIdx.x, w = blockIdx.y;
    const int orb = x < tb.N ? tb.occ0[x] : tb.part_orb[x - tb.N];
    const double2* src = GT + (size_t)w * ld + off + (size_t)x * M;
    double2* dst = rdm + (((size_t)w * 2 + spin) * M + orb) * M;
    for (int c = threadIdx.x; c < M; c += blockDim.x) dst[c] = src[c];
}

void launch_rdm_scatter(const SpinTables& tb, int nw, int M, const double2* GT, long long ld, long long off, int spin,
                        double2* rdm, cudaStream_t st)
{
    if (nw <= 0) return;
    k_rdm_scatter<<<dim3(tb.N + tb.np, nw), 128, 0, st>>>(tb, M, GT, ld, off, spin, rdm);
    msd_note_launch();
}

// <D_0|phi> = det(D0^dag phi_a) det(D0^dag phi_b) per walker.
__global__ void k_ref_ovlp(int nw, const double2* __restrict__ O0a, const double2* __restrict__ O0b,
                           double2* __restrict__ out)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w < nw) out[w] = cmul(O0a[w], O0b[w]);
}

void launch_ref_ovlp(int nw, const double2* O0a, const double2* O0b, double2* out, cudaStream_t st)
{
    k_ref_ovlp<<<(nw + 127) / 128, 128, 0, st>>>(nw, O0a, O0b, out); msd_note_launch();
}
