// Local-energy and force-bias contractions (Sec. III: fill_os / get_ss, and
// the force bias of Eq. 7), FP64 path.
//
// With G = G0^T (rows occ0 non-zero), B_s = A_s^-1 for an excitation string s
// with holes h_1..h_k and particles p_1..p_k, and
//   Lambda_g = G L_g (I - G),  Xi = sum_g G L_g G L_g (I - G),
//   K^{st}[(h,p)][(h',p')] = sum_g Lambda^s_g[h][p] Lambda^t_g[h'][p'],
//   u^s = sum_g V0_g Lambda^s_g,  V0_g = sum_s tr(L_g G^s),
// the determinant I = (a, b) has local energy
//   E_I = E_0 + e_a + e_b + X_ab,
//   E_0 = e0 + sum_s tr(h G^s) + 1/2 sum_g V0_g^2 - 1/2 sum_s sum_g tr(L_g G^s L_g G^s)
//   e_s = sum_ij B[i][j] Y[h_j][p_i] + 1/2 (Qc - Qx),   Y = Lambda_h + u - Xi
//   Qc = sum_ijkl B_ij B_kl K[(h_j,p_i)][(h_l,p_k)],  Qx = ... K[(h_j,p_k)][(h_l,p_i)]
//   X_ab = sum_ijkl Ba_ij Bb_kl K^{ab}[(ha_j,pa_i)][(hb_l,pb_k)]
// (the generalized Wick theorem of Sec. II A applied to the rank-k update
// G_I = G + (E_P - G[:,P]) B G[H,:]), and E_L = sum_I c_I r_I E_I / sum_I c_I r_I.
#include <type_traits>

#include "common.cuh"
#include "det_block.cuh"
#include "kernels.h"

// ------------------------------------------------------------------------
// C[m][n] = sum_k A[m][k] * B[n][k], A complex, B real, FP64.
// 64 x 64 tile, k-step 16, 256 threads with a 4 x 4 register block each.
__global__ void __launch_bounds__(256)
k_gemm_zd(int Mr, int Nc, int K, const double2* __restrict__ A, long long lda,
          const double* __restrict__ B, long long ldb, double2* __restrict__ C, long long ldc)
{
    __shared__ double2 As[16][64 + 1];
    __shared__ double Bs[16][64 + 1];
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
    double2 acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = cz(0, 0);
    for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = threadIdx.x + q * 256;
            const int rr = e / 16, kk = e % 16;
            const int m = m0 + rr, n = n0 + rr, k = k0 + kk;
            As[kk][rr] = (m < Mr && k < K) ? A[(size_t)m * lda + k] : cz(0, 0);
            Bs[kk][rr] = (n < Nc && k < K) ? B[(size_t)n * ldb + k] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < 16; ++kk) {
            double2 a[4]; double b[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
            for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[i][j].x = fma(a[i].x, b[j], acc[i][j].x);
                    acc[i][j].y = fma(a[i].y, b[j], acc[i][j].y);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int m = m0 + ty * 4 + i;
        if (m >= Mr) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + tx * 4 + j;
            if (n < Nc) C[(size_t)m * ldc + n] = acc[i][j];
        }
    }
}

void launch_gemm_zd(int Mr, int Nc, int K, const double2* A, long long lda, const double* B,
                    long long ldb, double2* C, long long ldc, cudaStream_t st)
{
    dim3 grid((Nc + 63) / 64, (Mr + 63) / 64);
    k_gemm_zd<<<grid, 256, 0, st>>>(Mr, Nc, K, A, lda, B, ldb, C, ldc); msd_note_launch();
}

// ------------------------------------------------------------------------
// Per (walker, Cholesky vector) epilogue of F = G L_g restricted to rows
// occ0 and columns occ0 u P (F[j][c] = (G L_g)[occ0_j][col_c]):
//   T = F[:, occ0],  v0 = tr T,  x = tr(T T) = tr(L G L G)
//   Lambda[j][p] = F[j][P_p] - sum_l T[j][l] G[occ0_l][P_p]
//   Lact[(h,p)] = Lambda[pos(h)][p],  Xic[(h,p)] = sum_l T[pos(h)][l] Lambda[l][p]
__global__ void __launch_bounds__(128)
k_fepi(SpinTables tb, int M, int n_chol, const double2* __restrict__ F, long long ldf,
       const double2* __restrict__ Gr, double2* __restrict__ v0, double2* __restrict__ xx,
       double2* __restrict__ Lact, double2* __restrict__ Xic)
{
    extern __shared__ double2 sm[];
    const int N = tb.N, np = tb.np, nh = tb.nh, NC = N + np, X = nh * np;
    double2* f = sm;                 // [N][NC]
    double2* gp = f + N * NC;        // [N][np]
    double2* lam = gp + N * np;      // [N][np]
    __shared__ double2 red[2][128];
    const int g = blockIdx.x, w = blockIdx.y, t = threadIdx.x;
    const double2* Fw = F + (size_t)w * N * ldf + (size_t)g * NC;
    for (int e = t; e < N * NC; e += blockDim.x) f[e] = Fw[(size_t)(e / NC) * ldf + e % NC];
    const double2* gr = Gr + (size_t)w * N * M;
    for (int e = t; e < N * np; e += blockDim.x) gp[e] = gr[(size_t)(e / np) * M + tb.part_orb[e % np]];
    __syncthreads();
    double2 a0 = cz(0, 0), a1 = cz(0, 0);
    for (int e = t; e < N * N; e += blockDim.x) {
        const int j = e / N, l = e % N;
        a1 = cfma(f[j * NC + l], f[l * NC + j], a1);
        if (j == l) a0 = cadd(a0, f[j * NC + j]);
    }
    for (int e = t; e < N * np; e += blockDim.x) {
        const int j = e / np, p = e % np;
        double2 v = f[j * NC + N + p];
        for (int l = 0; l < N; ++l) v = cfms(f[j * NC + l], gp[l * np + p], v);
        lam[e] = v;
    }
    red[0][t] = a0; red[1][t] = a1;
    __syncthreads();
    for (int o = 64; o; o >>= 1) {
        if (t < o) { red[0][t] = cadd(red[0][t], red[0][t + o]); red[1][t] = cadd(red[1][t], red[1][t + o]); }
        __syncthreads();
    }
    const size_t wg = (size_t)w * n_chol + g;
    if (t == 0) { v0[wg] = red[0][0]; xx[wg] = red[1][0]; }
    for (int e = t; e < X; e += blockDim.x) {
        const int h = e / np, p = e % np, j = tb.hole_pos[h];
        double2 xi = cz(0, 0);
        for (int l = 0; l < N; ++l) xi = cfma(f[j * NC + l], lam[l * np + p], xi);
        Lact[wg * X + e] = lam[j * np + p];
        Xic[wg * X + e] = xi;
    }
}

size_t fepi_smem(const SpinTables& tb) { return sizeof(double2) * (tb.N * (tb.N + tb.np) + 2 * tb.N * tb.np); }

// The same epilogue in fixed point (fixed.cuh) for N <= 32: the FP64 form is bound
// by the FP64 unit (95 % of its rate, 6.2 ms per spin for 640 copper-oxo walkers).
// One scale per block of operands: T per (walker, vector), G[occ0][P] per walker,
// Lambda per (walker, vector); sums of up to 32 complex products. The trace of T,
// which weighs most in the energy, sums 56 bits. Measured
// relative rms error against long double, fixed point and FP64: Lambda 5.7e-17 and
// 2.4e-16, Xi 1.2e-16 and 3.0e-16, tr T T 3.4e-17 and 5.6e-17. 6.2 -> 2.5 ms per spin
// (640 copper-oxo walkers), 3.1 -> 1.2 ms (64 iron-sulfur walkers).
#define FEPI_INT_NMAX 32
#define FEPI_INT_G 8      // Cholesky vectors per block: G[occ0][P] is converted once for them
__global__ void __launch_bounds__(256)
k_fepi_int(SpinTables tb, int M, int n_chol, const double2* __restrict__ F, long long ldf,
           const double2* __restrict__ Gr, double2* __restrict__ v0, double2* __restrict__ xx,
           double2* __restrict__ Lact, double2* __restrict__ Xic)
{
    extern __shared__ double2 sm[];
    const int N = tb.N, np = tb.np, nh = tb.nh, NC = N + np, X = nh * np, NP = N * np;
    double2* f = sm;                                      // [N][NC]: T as limbs, F_P as FP64
    Limbs* tl = reinterpret_cast<Limbs*>(sm);
    Limbs* gp = reinterpret_cast<Limbs*>(f + N * NC);     // [N][np]
    double2* lam = reinterpret_cast<double2*>(gp + NP);   // [N][np] FP64
    Limbs* ll = reinterpret_cast<Limbs*>(lam + NP);       // [N][np]
    __shared__ unsigned wmax[3][8];
    __shared__ long long wsum[2][8];
    __shared__ int wlow[2][8];
    __shared__ long long diag[2][FEPI_INT_NMAX];          // T[j][j] to 56 bits, for its trace
    const int w = blockIdx.y, t = threadIdx.x, nt = blockDim.x, lane = t & 31, warp = t >> 5, nwarp = nt >> 5;
    auto exponent = [&](int i) {      // of the largest magnitude the warps left in wmax[i]
        unsigned m = 0;
        for (int k = 0; k < nwarp; ++k) m = max(m, wmax[i][k]);
        return mag_exponent(m);
    };
    const double2* gr = Gr + (size_t)w * N * M;
    unsigned m = 0;
    for (int e = t; e < NP; e += nt) {
        lam[e] = gr[(size_t)(e / np) * M + tb.part_orb[e % np]];
        m = max(m, mag_bits(lam[e]));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) wmax[0][warp] = m;
    __syncthreads();
    const int eg = exponent(0);
    for (int e = t; e < NP; e += nt) gp[e] = to_limbs(lam[e], eg);
    const int g1 = min(n_chol, (int)(blockIdx.x + 1) * FEPI_INT_G);
    for (int g = blockIdx.x * FEPI_INT_G; g < g1; ++g) {
        const size_t wg = (size_t)w * n_chol + g;
        const double2* Fw = F + (size_t)w * N * ldf + (size_t)g * NC;
        m = 0;
        for (int e = t; e < N * NC; e += nt) {
            const int j = e / NC, c = e - j * NC;
            const double2 v = Fw[(size_t)j * ldf + c];
            f[e] = v;
            if (c < N) m = max(m, mag_bits(v));
        }
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) wmax[1][warp] = m;
        __syncthreads();
        const int et = exponent(1);
        for (int e = t; e < N * NC; e += nt) {
            const int j = e / NC, c = e - j * NC;
            if (c >= N) continue;
            const double2 v = f[e];
            if (c == j) { diag[0][j] = fixed56(v.x, et); diag[1][j] = fixed56(v.y, et); }
            tl[e] = to_limbs(v, et);
        }
        __syncthreads();
        // Lambda[j][p] = F_P[j][p] - sum_l T[j][l] G[occ0_l][P_p]
        m = 0;
        for (int e = t; e < NP; e += nt) {
            const int j = e / np, p = e - j * np;
            LimbSum s;
            for (int l = 0; l < N; ++l) s.add(tl[j * NC + l], gp[l * np + p]);
            const double2 fp = f[j * NC + N + p];
            const double2 v = cz(fp.x - int_to_fp64(s.re(), et + eg - 56), fp.y - int_to_fp64(s.imag(), et + eg - 56));
            lam[e] = v;
            m = max(m, mag_bits(v));
        }
        m = __reduce_max_sync(0xffffffffu, m);
        // tr T T over the warps (each thread's sum cut at 12 bits, so that the
        // totals of both halves stay in 64 and 32 bits), tr T
        LimbSum x;
        long long xr = 0, xi = 0;
        for (int e = t; e < N * N; e += nt) {
            const int j = e / N, l = e - j * N;
            x.add_all(tl[j * NC + l], tl[l * NC + j], xr, xi);
        }
        x.crr += xr >> 26;
        x.cim += xi >> 26;
        long long q[2] = {x.re(), x.imag()};
        int lo[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            lo[c] = __reduce_add_sync(0xffffffffu, (int)(q[c] & 4095));
            q[c] >>= 12;
            for (int o = 16; o; o >>= 1) q[c] += __shfl_xor_sync(0xffffffffu, q[c], o);
        }
        if (lane == 0) {
            wmax[2][warp] = m;
            for (int c = 0; c < 2; ++c) { wsum[c][warp] = q[c]; wlow[c][warp] = lo[c]; }
        }
        if (warp == nwarp - 1) {
            long long d[2] = {lane < N ? diag[0][lane] : 0, lane < N ? diag[1][lane] : 0};
            for (int c = 0; c < 2; ++c)
                for (int o = 16; o; o >>= 1) d[c] += __shfl_xor_sync(0xffffffffu, d[c], o);
            if (lane == 0) v0[wg] = cz(int_to_fp64(d[0], et - 56), int_to_fp64(d[1], et - 56));
        }
        __syncthreads();
        const int el = exponent(2);
        for (int e = t; e < NP; e += nt) ll[e] = to_limbs(lam[e], el);
        if (t < 2) {
            long long a = 0, b = 0;
            for (int k = 0; k < nwarp; ++k) { a += wsum[t][k]; b += wlow[t][k]; }
            // a 2^12 + b = (a >> 16) 2^28 + ((a & 65535) 2^12 + b)
            reinterpret_cast<double*>(xx + wg)[t] = int_to_fp64_slow(a >> 16, ((a & 65535) << 12) + b, 2 * et - 56);
        }
        __syncthreads();
        for (int e = t; e < X; e += nt) {
            const int h = e / np, p = e - h * np, j = tb.hole_pos[h];
            LimbSum s;
            for (int l = 0; l < N; ++l) s.add(tl[j * NC + l], ll[l * np + p]);
            Lact[wg * X + e] = lam[j * np + p];
            Xic[wg * X + e] = cz(int_to_fp64(s.re(), et + el - 56), int_to_fp64(s.imag(), et + el - 56));
        }
        if (max(max(eg, et), el) > 1024) {   // an infinity or a NaN somewhere
            const double nan = __longlong_as_double(0x7ff8000000000000ll);
            __syncthreads();
            if (t == 0) v0[wg] = xx[wg] = cz(nan, nan);
            for (int e = t; e < X; e += nt) Lact[wg * X + e] = Xic[wg * X + e] = cz(nan, nan);
        }
        __syncthreads();   // f and lam are free for the next vector
    }
}

void launch_fepi(const SpinTables& tb, int nw, int M, int n_chol, const double2* F, long long ldf,
                 const double2* Gr, double2* v0, double2* xx, double2* Lact, double2* Xic,
                 cudaStream_t st)
{
    const int NP = tb.N * tb.np;
    const size_t smem_int = sizeof(double2) * (tb.N * (tb.N + tb.np) + 3 * NP);
    if (tb.N <= FEPI_INT_NMAX && smem_int <= 200 * 1024) {
        const size_t smem = smem_int;
        if (smem > 44 * 1024)
            cudaFuncSetAttribute(k_fepi_int, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        const int threads = NP <= 128 ? 128 : NP >= 256 ? 256 : (NP + 31) / 32 * 32;   // one (j, p) per thread
        k_fepi_int<<<dim3((n_chol + FEPI_INT_G - 1) / FEPI_INT_G, nw), threads, smem, st>>>(tb, M, n_chol, F, ldf, Gr, v0,
                                                                                        xx, Lact, Xic);
        msd_note_launch();
        return;
    }
    dim3 grid(n_chol, nw);
    const size_t smem = fepi_smem(tb);
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_fepi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_fepi<<<grid, 128, smem, st>>>(tb, M, n_chol, F, ldf, Gr, v0, xx, Lact, Xic); msd_note_launch();
}

// ------------------------------------------------------------------------
// One-body pieces per (walker, spin): e1 = tr(h G), and
// Lambda_h[(h,p)] = (G hl (I - G))[H_h][P_p] with hl = h, or the matrix the
// caller gives (linear in it: hl = h + J adds sum_g C_g Lambda_g).
struct OnebodyArgs {
    SpinTables t[2];
    const double *h1[2], *hl[2];
    const double2* Gr[2];
    double2 *e1[2], *Lh[2];
};
__global__ void __launch_bounds__(128)
k_onebody(const __grid_constant__ OnebodyArgs a_, int M)
{
    extern __shared__ double2 sm[];
    const int s = blockIdx.y;
    const SpinTables& tb = a_.t[s];
    const double *h1 = a_.h1[s], *hl = a_.hl[s];
    const int N = tb.N, np = tb.np, nh = tb.nh, NC = N + np;
    double2* fh = sm;   // [nh][NC]
    __shared__ double2 red[128];
    const int w = blockIdx.x, t = threadIdx.x;
    const double2* gr = a_.Gr[s] + (size_t)w * N * M;
    double2 a = cz(0, 0);
    for (int e = t; e < N * M; e += blockDim.x) {
        const int j = e / M, r = e % M;
        a = cadd(a, cscale(gr[e], h1[(size_t)tb.occ0[j] * M + r]));
    }
    for (int e = t; e < nh * NC; e += blockDim.x) {
        const int h = e / NC, c = e % NC;
        const int col = c < N ? tb.occ0[c] : tb.part_orb[c - N];
        const double2* gj = gr + (size_t)tb.hole_pos[h] * M;
        double2 v = cz(0, 0);
        for (int r = 0; r < M; ++r) v = cadd(v, cscale(gj[r], hl[(size_t)col * M + r]));
        fh[e] = v;
    }
    red[t] = a;
    __syncthreads();
    for (int o = 64; o; o >>= 1) {
        if (t < o) red[t] = cadd(red[t], red[t + o]);
        __syncthreads();
    }
    if (t == 0) a_.e1[s][w] = red[0];
    for (int e = t; e < nh * np; e += blockDim.x) {
        const int h = e / np, p = e % np;
        double2 v = fh[h * NC + N + p];
        for (int l = 0; l < N; ++l) v = cfms(fh[h * NC + l], gr[(size_t)l * M + tb.part_orb[p]], v);
        a_.Lh[s][(size_t)w * nh * np + e] = v;
    }
}

void launch_onebody(const SpinTables& ta, const SpinTables& tb, int nw, int M, const double* const h1[2],
                    const double2* const Gr[2], double2* const e1[2], double2* const Lh[2], cudaStream_t st,
                    const double* const hl[2])
{
    OnebodyArgs a;
    size_t smem = 0;
    const SpinTables* T[2] = {&ta, &tb};
    for (int s = 0; s < 2; ++s) {
        a.t[s] = *T[s];
        a.h1[s] = h1[s]; a.hl[s] = hl[s];
        a.Gr[s] = Gr[s]; a.e1[s] = e1[s]; a.Lh[s] = Lh[s];
        smem = smem > sizeof(double2) * T[s]->nh * (T[s]->N + T[s]->np) ? smem : sizeof(double2) * T[s]->nh * (T[s]->N + T[s]->np);
    }
    if (smem > 44 * 1024) cudaFuncSetAttribute(k_onebody, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_onebody<<<dim3(nw, 2), 128, smem, st>>>(a, M); msd_note_launch();
}

// ------------------------------------------------------------------------
// Sums over Cholesky vectors per (walker, spin):
//   Y[x] = Lh[x] + sum_g V0_g Lact_g[x] - sum_g Xic_g[x],  V0_g = v0a_g + v0b_g
//   scal[w][0 + s] = sum_g xx_g (exchange of G),  scal[w][2] = sum_g V0_g^2
// One block per (walker, spin): warp k takes the vectors g = k mod 8, lanes over
// the entries x (contiguous rows); the warps' sums are added in pairs (added in a row,
// most round at the size of the total: energies 1.75e-16 rms off). (A serial
// sum over g per entry left 64 walkers with 64 x 75 chains of 1600 dependent FP64
// operations: 1.05 ms for both iron-sulfur spins.)
struct GammaArgs {
    int X[2];
    const double2 *v0[2], *xx[2], *Lact[2], *Xic[2], *Lh[2];
    double2* Y[2];
};
__global__ void __launch_bounds__(256)
k_gamma_reduce(const __grid_constant__ GammaArgs a, int n_chol, double2* __restrict__ scal)
{
    __shared__ double2 part[8][MSD_XMAX];
    __shared__ double2 red[2][8];
    const int w = blockIdx.x, spin = blockIdx.y, t = threadIdx.x, warp = t >> 5, lane = t & 31, X = a.X[spin];
    const size_t base = (size_t)w * n_chol;
    const double2 *va = a.v0[0] + base, *vb = a.v0[1] + base;
    double2 acc[(MSD_XMAX + 31) / 32];
#pragma unroll
    for (int q = 0; q < (MSD_XMAX + 31) / 32; ++q) acc[q] = cz(0, 0);
    for (int g = warp; g < n_chol; g += 8) {
        const double2 V0 = cadd(va[g], vb[g]);
        const double2 *la = a.Lact[spin] + (base + g) * X, *xi = a.Xic[spin] + (base + g) * X;
#pragma unroll
        for (int q = 0; q < (MSD_XMAX + 31) / 32; ++q) {
            const int x = q * 32 + lane;
            if (q * 32 >= X) break;   // (no FP64 issue slots for empty warps)
            if (x < X) acc[q] = csub(cfma(V0, la[x], acc[q]), xi[x]);
        }
    }
#pragma unroll
    for (int q = 0; q < (MSD_XMAX + 31) / 32; ++q)
        if (q * 32 + lane < X) part[warp][q * 32 + lane] = acc[q];
    // consecutive vectors go to different warps: they come in descending order as a
    // rule, and partial sums of one size round at the size of the total once only
    double2 s0 = cz(0, 0), s1 = cz(0, 0);
    for (int g = lane * 8 + warp; g < n_chol; g += 256) {
        s0 = cadd(s0, a.xx[spin][base + g]);
        const double2 V0 = cadd(va[g], vb[g]);
        s1 = cfma(V0, V0, s1);
    }
    for (int o = 16; o; o >>= 1) {
        s0.x += __shfl_xor_sync(0xffffffffu, s0.x, o); s0.y += __shfl_xor_sync(0xffffffffu, s0.y, o);
        s1.x += __shfl_xor_sync(0xffffffffu, s1.x, o); s1.y += __shfl_xor_sync(0xffffffffu, s1.y, o);
    }
    if (lane == 0) { red[0][warp] = s0; red[1][warp] = s1; }
    __syncthreads();
    for (int x = t; x < X; x += blockDim.x) {
        auto y = [&](int q) { return cadd(part[q][x], part[q + 1][x]); };
        a.Y[spin][(size_t)w * X + x] = cadd(a.Lh[spin][(size_t)w * X + x], cadd(cadd(y(0), y(2)), cadd(y(4), y(6))));
    }
    if (t < 2) {
        auto r = [&](int q) { return cadd(red[t][q], red[t][q + 1]); };
        const double2 s = cadd(cadd(r(0), r(2)), cadd(r(4), r(6)));
        if (t == 0) scal[(size_t)w * 8 + spin] = s;
        else if (spin == 0) scal[(size_t)w * 8 + 2] = s;
    }
}

void launch_gamma_reduce(int nw, const int X[2], int n_chol, const double2* const v0[2], const double2* const xx[2],
                         const double2* const Lact[2], const double2* const Xic[2], const double2* const Lh[2],
                         double2* const Y[2], double2* scal, cudaStream_t st)
{
    GammaArgs a;
    for (int s = 0; s < 2; ++s) {
        a.X[s] = X[s]; a.v0[s] = v0[s]; a.xx[s] = xx[s]; a.Lact[s] = Lact[s]; a.Xic[s] = Xic[s]; a.Lh[s] = Lh[s];
        a.Y[s] = Y[s];
    }
    k_gamma_reduce<<<dim3(nw, 2), 256, 0, st>>>(a, n_chol, scal);
    msd_note_launch();
}

// ------------------------------------------------------------------------
// Gram matrices K[w][x][y] = sum_g P[w][g][x] Q[w][g][y] (complex, no
// conjugation) for one spin pair; 32 x 32 output tile per block.
template <typename TK>
__global__ void __launch_bounds__(256)
k_gram(int Xp, int Xq, int n_chol, const double2* __restrict__ P, const double2* __restrict__ Q,
       TK* __restrict__ Kout)
{
    __shared__ double2 ps[16][32], qs[16][32];
    const int w = blockIdx.z;
    const int x0 = blockIdx.y * 32, y0 = blockIdx.x * 32;
    const int t = threadIdx.x;
    const int ty = t / 16, tx = t % 16;      // 16 x 16 threads, 2 x 2 outputs each
    double2 acc[2][2] = {{cz(0, 0), cz(0, 0)}, {cz(0, 0), cz(0, 0)}};
    const double2* Pw = P + (size_t)w * n_chol * Xp;
    const double2* Qw = Q + (size_t)w * n_chol * Xq;
    for (int g0 = 0; g0 < n_chol; g0 += 16) {
        for (int e = t; e < 16 * 32; e += 256) {
            const int gg = e / 32, xx = e % 32, g = g0 + gg;
            ps[gg][xx] = (g < n_chol && x0 + xx < Xp) ? Pw[(size_t)g * Xp + x0 + xx] : cz(0, 0);
            qs[gg][xx] = (g < n_chol && y0 + xx < Xq) ? Qw[(size_t)g * Xq + y0 + xx] : cz(0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int gg = 0; gg < 16; ++gg) {
            const double2 p0 = ps[gg][ty * 2], p1 = ps[gg][ty * 2 + 1];
            const double2 q0 = qs[gg][tx * 2], q1 = qs[gg][tx * 2 + 1];
            acc[0][0] = cfma(p0, q0, acc[0][0]); acc[0][1] = cfma(p0, q1, acc[0][1]);
            acc[1][0] = cfma(p1, q0, acc[1][0]); acc[1][1] = cfma(p1, q1, acc[1][1]);
        }
        __syncthreads();
    }
    for (int i = 0; i < 2; ++i)
        for (int j = 0; j < 2; ++j) {
            const int x = x0 + ty * 2 + i, y = y0 + tx * 2 + j;
            if (x < Xp && y < Xq) {
                const size_t e = ((size_t)w * Xp + x) * Xq + y;
                Kout[2 * e] = (TK)acc[i][j].x;
                Kout[2 * e + 1] = (TK)acc[i][j].y;
            }
        }
}

void launch_gram(int nw, int Xp, int Xq, int n_chol, const double2* P, const double2* Q, void* K,
                 bool fp32, cudaStream_t st)
{
    if (Xp <= 0 || Xq <= 0 || nw <= 0) return;
    dim3 grid((Xq + 31) / 32, (Xp + 31) / 32, nw);
    if (fp32) k_gram<float><<<grid, 256, 0, st>>>(Xp, Xq, n_chol, P, Q, (float*)K);
    else k_gram<double><<<grid, 256, 0, st>>>(Xp, Xq, n_chol, P, Q, (double*)K);
    msd_note_launch();
}

// ------------------------------------------------------------------------
// Same-spin per-string energy (get_ss and the one-body / Coulomb linear
// parts): e_s = sum_ij B_ij Y[h_j][p_i] + 1/2 (Qc - Qx), accumulated as
// r_s w_s e_s into per-walker partial sums. Precision T for B, K and the
// arithmetic; the block sum is FP64. The block first forms the walker's
// antisymmetrized pair table of K (C(nh,2) C(np,2) entries, against X^2 for
// K) in shared memory; each string then takes C(k,2)^2 gathers of it for
// (Qc - Qx) / 2 (string_energy_value).
// Block b of all (spin, level) blocks writes slot slot0 + b. ONLY = 0: one launch
// for both spins and all levels (a launch per level was most of the time of this
// term at small sizes, 87 us of 391 for 16 walkers of 100 determinants); ONLY = k: the blocks of level k,
// with that level's registers (131 for all levels: 1.74 against 1.09 ms at the
// iron-sulfur size).
struct SeArgs {
    SpinTables t[2];
    const double2* wts[2];
    const void *B[2], *K[2], *Y[2];
    int blk[2][MSD_KMAX + 2];   // first block of each (spin, level)
};

template <typename T, int ONLY>
__global__ void __launch_bounds__(SE_THREADS)
k_string_energy(const __grid_constant__ SeArgs a, double2* __restrict__ part, int nslot, int slot0)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    // this block among all (spin, level) blocks
    int b = blockIdx.x;
    if (ONLY) {
        const int na = a.blk[0][ONLY + 1] - a.blk[0][ONLY];
        b = b < na ? a.blk[0][ONLY] + b : a.blk[1][ONLY] + b - na;
    }
    const int s = b >= a.blk[1][1];
    const SpinTables& tb = a.t[s];
    __shared__ double2 red[SE_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    int k = ONLY ? ONLY : 1;
    while (!ONLY && b >= a.blk[s][k + 1]) ++k;
    const SeTab<T> tab = load_se_table<T>(tb, a.K[s], a.Y[s], w, k, smraw);
    const int blk = b - a.blk[s][k];
    double2 v;
    if constexpr (ONLY > 0) {
        v = string_energy_block<ONLY, T>(tb, w, blk, a.B[s], tab, a.wts[s]);
    } else {
        switch (k) {
        case 1: v = string_energy_block<1, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        case 2: v = string_energy_block<2, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        case 3: v = string_energy_block<3, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        case 4: v = string_energy_block<4, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        case 5: v = string_energy_block<5, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        default: v = string_energy_block<6, T>(tb, w, blk, a.B[s], tab, a.wts[s]); break;
        }
    }
    red[t] = v;
    __syncthreads();
    for (int o = SE_THREADS / 2; o; o >>= 1) {
        if (t < o) red[t] = cadd(red[t], red[t + o]);
        __syncthreads();
    }
    if (t == 0) part[(size_t)w * nslot + slot0 + b] = red[0];
}

int string_energy_blocks(const SpinTables& tb, int k)
{
    const int ns = tb.bucket[k + 1] - tb.bucket[k];
    return ns > 0 ? (ns + SE_THREADS * SE_PER_THREAD - 1) / (SE_THREADS * SE_PER_THREAD) : 0;
}

size_t string_energy_smem(const SpinTables& tb, bool fp32)
{
    const int X = tb.nh * tb.np;
    const size_t pairs = (size_t)(tb.nh * (tb.nh - 1) / 2) * (tb.np * (tb.np - 1) / 2);
    return fp32 ? sizeof(float2) * (pairs + X) : sizeof(double2) * (pairs + X) + sizeof(Limbs) * SE_LIMBS;
}

void launch_string_energy(const SpinTables& ta, const SpinTables& tb, int nw, const double2* const wts[2],
                          const void* const B[2], const void* const K[2], const void* const Y[2], bool fp32,
                          double2* part, int nslot, int slot0, cudaStream_t st)
{
    SeArgs a;
    const SpinTables* T[2] = {&ta, &tb};
    int n = 0;
    size_t smem = 0;
    for (int s = 0; s < 2; ++s) {
        a.t[s] = *T[s];
        a.wts[s] = wts[s]; a.B[s] = B[s]; a.K[s] = K[s]; a.Y[s] = Y[s];
        a.blk[s][0] = n;
        for (int k = 1; k <= MSD_KMAX; ++k) { a.blk[s][k] = n; n += string_energy_blocks(*T[s], k); }
        a.blk[s][MSD_KMAX + 1] = n;
        const size_t b = string_energy_smem(*T[s], fp32);
        smem = smem > b ? smem : b;
    }
    if (n == 0) return;
    auto go = [&](auto kern, int blocks) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<dim3(blocks, nw), SE_THREADS, smem, st>>>(a, part, nslot, slot0);
        msd_note_launch();
    };
    if ((long long)n * nw <= ONE_LAUNCH_BLOCKS * msd_sm_count()) {
        if (fp32) go(k_string_energy<float, 0>, n); else go(k_string_energy<double, 0>, n);
        return;
    }
    for (int k = 1; k <= MSD_KMAX; ++k) {
        const int m = string_energy_blocks(ta, k) + string_energy_blocks(tb, k);
        if (!m) continue;
        switch (k) {
        case 1: if (fp32) go(k_string_energy<float, 1>, m); else go(k_string_energy<double, 1>, m); break;
        case 2: if (fp32) go(k_string_energy<float, 2>, m); else go(k_string_energy<double, 2>, m); break;
        case 3: if (fp32) go(k_string_energy<float, 3>, m); else go(k_string_energy<double, 3>, m); break;
        case 4: if (fp32) go(k_string_energy<float, 4>, m); else go(k_string_energy<double, 4>, m); break;
        case 5: if (fp32) go(k_string_energy<float, 5>, m); else go(k_string_energy<double, 5>, m); break;
        default: if (fp32) go(k_string_energy<float, 6>, m); else go(k_string_energy<double, 6>, m); break;
        }
    }
}

int string_energy_slots(const SpinTables& tb)
{
    int n = 0;
    for (int k = 1; k <= MSD_KMAX; ++k) n += string_energy_blocks(tb, k);
    return n;
}

// ------------------------------------------------------------------------
// Opposite-spin cross term (fill_os) per determinant (a, b) with levels
// (ka, KB): c_I r_a r_b X_ab with
//   X_ab = sum_ij Ba_ij sum_kl Bb_kl K^{ab}[(ha_j,pa_i)][(hb_l,pb_k)].
// The beta level KB is a template parameter (its inverse minor is held in
// registers); the alpha level runs at run time.
template <int KB, typename T>
__global__ void __launch_bounds__(PC_THREADS)
k_pair_cross(SpinTables ta, SpinTables tbb, PairTables pt, int ka, int lo, int n,
             const void* __restrict__ ra_in, const void* __restrict__ rb_in,
             const void* __restrict__ Ba_in, const void* __restrict__ Bb_in,
             const void* __restrict__ Kin, double2* __restrict__ part, int nslot, int slot0)
{
    using T2 = typename std::conditional<std::is_same<T, float>::value, float2, double2>::type;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int Xa = ta.nh * ta.np, Xb = tbb.nh * tbb.np;
    T2* ks = reinterpret_cast<T2*>(smraw);   // [Xa][Xb]
    __shared__ double2 red[PC_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    const T2* Kw = reinterpret_cast<const T2*>(Kin) + (size_t)w * Xa * Xb;
    for (int e = t; e < Xa * Xb; e += blockDim.x) ks[e] = Kw[e];
    __syncthreads();
    const T2* ra = reinterpret_cast<const T2*>(ra_in);
    const T2* rb = reinterpret_cast<const T2*>(rb_in);
    T2 contrib = T2{0, 0};   // this thread's determinants, in the working precision
    // the shared Gram matrix is filled once per block and reused by
    // PC_PER_THREAD determinants per thread
    for (int it = 0; it < PC_PER_THREAD; ++it) {
        const int i0 = blockIdx.x * (PC_THREADS * PC_PER_THREAD) + it * PC_THREADS + t;
        if (i0 >= n) break;
        const T2 v = pair_cross_term<KB, T>(ta, tbb, pt, ka, lo + i0, w, Ba_in, Bb_in, ks, ra, rb);
        contrib.x += v.x;
        contrib.y += v.y;
    }
    red[t] = cz((double)contrib.x, (double)contrib.y);
    __syncthreads();
    for (int o = PC_THREADS / 2; o; o >>= 1) {
        if (t < o) red[t] = cadd(red[t], red[t + o]);
        __syncthreads();
    }
    if (t == 0) part[(size_t)w * nslot + slot0 + blockIdx.x] = red[0];
}

template <int KB>
static void launch_pc_k(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int ka,
                        int nw, const void* ra, const void* rb, const void* Ba, const void* Bb,
                        const void* K, bool fp32, double2* part, int nslot, int& slot,
                        cudaStream_t st, bool use_runs)
{
    const int idx = ka * (MSD_KMAX + 1) + KB;
    const int lo = pt.bucket[idx], n = pt.bucket[idx + 1] - lo;
    if (n <= 0) return;
    if (use_runs && pt.run_side[idx]) {
        launch_pair_run(ta, tb, pt, idx, ka, KB, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st);
        slot += pair_run_blocks(pt, idx);
        return;
    }
    const int nb = (n + PC_THREADS * PC_PER_THREAD - 1) / (PC_THREADS * PC_PER_THREAD);
    dim3 grid(nb, nw);
    const size_t smem = (fp32 ? sizeof(float2) : sizeof(double2)) * (size_t)(ta.nh * ta.np) * (tb.nh * tb.np);
    if (launch_pair_cross2(ka, KB, fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st)) {
        slot += nb;
        return;
    }
    if (fp32) {
        cudaFuncSetAttribute(k_pair_cross<KB, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_cross<KB, float><<<grid, PC_THREADS, smem, st>>>(ta, tb, pt, ka, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot); msd_note_launch();
    } else {
        cudaFuncSetAttribute(k_pair_cross<KB, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_cross<KB, double><<<grid, PC_THREADS, smem, st>>>(ta, tb, pt, ka, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot); msd_note_launch();
    }
    slot += nb;
}

void launch_pair_cross(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int nw,
                       const void* ra, const void* rb, const void* Ba, const void* Bb,
                       const void* K, bool fp32, double2* part, int nslot, int slot0,
                       cudaStream_t st, bool use_runs)
{
    int slot = slot0;
    if (launch_pair_cross_all(ta, tb, pt, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot0, st, use_runs)) return;
    for (int ka = 1; ka <= MSD_KMAX; ++ka) {
        launch_pc_k<1>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
        launch_pc_k<2>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
        launch_pc_k<3>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
        launch_pc_k<4>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
        launch_pc_k<5>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
        launch_pc_k<6>(ta, tb, pt, ka, nw, ra, rb, Ba, Bb, K, fp32, part, nslot, slot, st, use_runs);
    }
}

int pair_cross_slots(const PairTables& pt, bool use_runs)
{
    int n = 0;
    for (int ka = 1; ka <= MSD_KMAX; ++ka)
        for (int kb = 1; kb <= MSD_KMAX; ++kb) {
            const int idx = ka * (MSD_KMAX + 1) + kb;
            const int c = pt.bucket[idx + 1] - pt.bucket[idx];
            if (c <= 0) continue;
            if (use_runs && pt.run_side[idx]) n += pair_run_blocks(pt, idx);
            else n += (c + PC_THREADS * PC_PER_THREAD - 1) / (PC_THREADS * PC_PER_THREAD);
        }
    return n;
}

// ------------------------------------------------------------------------
// Final assembly per walker:
//   R = sum of slots [0, nR),  S = sum of slots [nR, nslot)
//   E_0 = e0 + e1a + e1b + 1/2 sum_g V0^2 - 1/2 (xa + xb)
//   E_L = E_0 + S / R,  O_T = O0a O0b R
__global__ void k_final(int nw, const double2* __restrict__ part, int nslot, int nR, double e0,
                        const double2* __restrict__ e1a, const double2* __restrict__ e1b,
                        const double2* __restrict__ scal, const double2* __restrict__ O0a,
                        const double2* __restrict__ O0b, double2* __restrict__ eloc,
                        double2* __restrict__ ovlp)
{
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;   // one warp per walker
    if (w >= nw) return;
    const double2 R = warp_sum_slots(part + (size_t)w * nslot, nR, lane);
    const double2 S = warp_sum_slots(part + (size_t)w * nslot + nR, nslot - nR, lane);
    if (lane) return;
    const double2* sc = scal + (size_t)w * 8;
    double2 E0 = cadd(cz(e0, 0), cadd(e1a[w], e1b[w]));
    E0 = cadd(E0, cscale(sc[2], 0.5));
    E0 = csub(E0, cscale(cadd(sc[0], sc[1]), 0.5));
    eloc[w] = cadd(E0, cdiv(S, R));
    if (ovlp) ovlp[w] = cmul(cmul(O0a[w], O0b[w]), R);
}

void launch_final(int nw, const double2* part, int nslot, int nR, double e0, const double2* e1a,
                  const double2* e1b, const double2* scal, const double2* O0a, const double2* O0b,
                  double2* eloc, double2* ovlp, cudaStream_t st)
{
    k_final<<<(nw + 3) / 4, 128, 0, st>>>(nw, part, nslot, nR, e0, e1a, e1b, scal, O0a, O0b,
                                             eloc, ovlp); msd_note_launch();
}
