// Excitation-string minors and CI weights with the walkers along the lanes
// (get_dets of Sec. III), and the FP32 inverse minors of the mixed path.
//
// Ratios. r_s = sign * det A_s, A_s[i][j] = G[h_i][p_j], of every string and
// walker in FP64. A k x k LU costs about 4 k^3 / 3 FP64 FMAs and k reciprocals;
// here a minor is a Laplace expansion over smaller minors that its neighbours
// share: all 2 x 2 minors of the active block once per walker (8 FMAs each),
// then level 3 along its last row (3 complex products), level 4 over pairs of
// 2 x 2 minors (6) or along its last row over the level-3 ratios (4), levels 5
// and 6 along the last row over the level below (5, 6) where the trial holds all
// the k strings that takes, else over the 2 x 2 minors (35, 105). GB300 issues
// two FP64 FMAs per clock and SM, so the operation count is the time.
//
// Cancellation. An expansion is off by a few ulps of its largest product, a pivoted LU
// by those times the minor's own conditioning. The two are alike for blocks whose
// products do not cancel (random ones, levels 3 to 6: 1.1e-16 to 2.2e-16 relative,
// median, the LU 1.4e-16 to 3.1e-16; graded rows and columns: the expansions half the
// LU's), but the active block of a walker that overlaps the reference little is a large
// part of low rank plus one of order one, and there the expansions lose g^(k-1) where
// the LU loses g. So every minor carries log2 of its largest product, the maximum over
// all permutations (max-plus arithmetic on the operands' high words, 16 fractional
// bits: no FP64 operation), and a minor 2^3 below that is evaluated once more by an LU
// of its own (k_minor_lu). Random blocks: 0.1 to 0.4 % of the minors, error then at or
// below the LU's; with blocks of rank 1 or 2 times 3 to 1e4 added the error stays
// within 1.2 of it (limits of 2^4: 1.5, 2^6: 3).
//
// Layout. Arrays of a string (or an active entry) hold its walkers contiguously,
// rT[s][nw]: a warp's lanes are walkers of the same string, so index lists are
// read once per warp, every gather of another string's ratios is a contiguous
// row, and lanes do not diverge over lists of different length (one string per
// lane left half of the FP64 issue slots of the weights kernel idle). The
// weights leave through a shared-memory tile in the [walker][string] order that
// the per-determinant kernels read.
//
// Iron-sulfur trial, 640 walkers (12.5e3 strings per spin): ratios and FP32
// inverse minors 3.60 (one pivoted LU per string) -> 1.48 ms (1.33 without the
// check of the cancellation and its LUs), weights 1.32 -> 0.89
// ms; 1e6 determinants, 10 walkers: weights 0.93 -> 0.28 ms.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "minor_lu.cuh"

namespace {

struct MinorSpin {
    int nh, np, n_str;
    int bucket[MSD_KMAX + 2];
    int vbucket[MSD_KMAX + 2];   // strings outside the trial, by level: [vbucket[k], vbucket[k + 1])
    const uint4* str_hp;
    const int8_t* str_sign;
    const int* sub;          // [n_str][MSD_KMAX] (string << 1 | negative), -1 first if one is missing
    const double2* GT;       // [nh np][nw]
    double2* m2;             // [C(nh,2) C(np,2)][nw]
    double2* rT;             // [n_str][nw]
    int* t2;                 // as m2: log2 of the larger product (log_mag)
    int* tr;                 // from string bucket[3] on, as rT: log2 of the largest product; odd: evaluate by LU
    double2* B;              // inverse minors of the trial's strings to write with the LU, or NULL
    long long b_off[MSD_KMAX + 2];
};
// Both spins of a launch (indexed by the block, in constant memory).
struct MinorArgs { MinorSpin s[2]; };

// log2 max(|Re v|, |Im v|) to 0.09, 16 fractional bits; far below any sum of six for 0.
__device__ __forceinline__ int log_mag(double2 v)
{
    const int k = mag_key(v) >> 4;
    return k ? k - (1023 << 16) : -(2400 << 16);
}
#define MINOR_BITS 3   // a minor this far below its largest product takes the LU

__device__ __forceinline__ void pair_of(int e, int n, int& a, int& b)
{
    a = 0;
    while (e >= n - 1 - a) { e -= n - 1 - a; ++a; }
    b = a + 1 + e;
}

// m2[(h,h')(p,p')] = G[h][p] G[h'][p'] - G[h][p'] G[h'][p]
__global__ void __launch_bounds__(256) k_minor2(const __grid_constant__ MinorArgs a, int nw)
{
    const MinorSpin& S = a.s[blockIdx.y];
    const int npp = S.np * (S.np - 1) / 2, n2 = S.nh * (S.nh - 1) / 2 * npp;
    const long long e = blockIdx.x * 256ll + threadIdx.x;
    if (e >= (long long)n2 * nw) return;
    const int pr = (int)(e / nw), w = (int)(e - (long long)pr * nw);
    int h, h2, p, p2;
    pair_of(pr / npp, S.nh, h, h2);
    pair_of(pr % npp, S.np, p, p2);
    const double2* g = S.GT + w;
    auto G = [&](int a, int b) { return g[(size_t)(a * S.np + b) * nw]; };
    const double2 g0 = G(h, p), g1 = G(h, p2), g2 = G(h2, p), g3 = G(h2, p2);
    S.m2[e] = cfms(g1, g2, cmul(g0, g3));
    S.t2[e] = max(log_mag(g0) + log_mag(g3), log_mag(g1) + log_mag(g2));
}

// Minors of the strings of levels k0 to k1, the trial's and, for k0 = k1, those
// outside it; subs: through the ratios of the level below where the string has them.
__global__ void __launch_bounds__(256, 4)
k_minors(const __grid_constant__ MinorArgs a, int k0, int k1, bool subs, int nw)
{
    const MinorSpin& S = a.s[blockIdx.y];
    const int s0 = S.bucket[k0], n = S.bucket[k1 + 1] - s0, nv = k0 == k1 ? S.vbucket[k0 + 1] - S.vbucket[k0] : 0;
    const long long e = blockIdx.x * 256ll + threadIdx.x;
    if (e >= (long long)(n + nv) * nw) return;
    const int i = (int)(e / nw), w = (int)(e % nw), s = i < n ? s0 + i : S.vbucket[k0] + i - n;
    int k = k0;
    while (k < k1 && s >= S.bucket[k + 1]) ++k;
    double2* out = S.rT + (size_t)s * nw + w;
    if (k == 0) { *out = cz(1, 0); return; }
    const int np = S.np, nh = S.nh, npp = np * (np - 1) / 2;
    const uint4 rec = S.str_hp[s];
    const double2* g = S.GT + w;
    const double2* m2 = S.m2 + w;
    const int* t2 = S.t2 + w;
    int* tr = S.tr + w;
    const double sg = S.str_sign[s];
    auto G = [&](int i, int j) { return g[(size_t)(rec_h(rec, i) * np + rec_p(rec, j)) * nw]; };
    // 2 x 2 minor of rows a < b, columns c < d of the string's block, and its row
    auto R2 = [&](int a, int b, int c, int d) {
        const int hp = pair_index(rec_h(rec, a), rec_h(rec, b), nh), pp = pair_index(rec_p(rec, c), rec_p(rec, d), np);
        return (size_t)(hp * npp + pp) * nw;
    };
    auto M2 = [&](int a, int b, int c, int d) { return m2[R2(a, b, c, d)]; };
    if (k == 1) { *out = cscale(G(0, 0), sg); return; }
    if (k == 2) { *out = cscale(M2(0, 1, 0, 1), sg); return; }
    // 4 x 4 minor of rows a < b < c < d, columns q0 < q1 < q2 < q3, log2 of its largest
    // product to l
    auto M4 = [&](int a, int b, int c, int d, int q0, int q1, int q2, int q3, int& l) {
        const size_t r01 = R2(a, b, q0, q1), r02 = R2(a, b, q0, q2), r03 = R2(a, b, q0, q3), r12 = R2(a, b, q1, q2),
                     r13 = R2(a, b, q1, q3), r23 = R2(a, b, q2, q3);
        const size_t s01 = R2(c, d, q0, q1), s02 = R2(c, d, q0, q2), s03 = R2(c, d, q0, q3), s12 = R2(c, d, q1, q2),
                     s13 = R2(c, d, q1, q3), s23 = R2(c, d, q2, q3);
        double2 v = cmul(m2[r01], m2[s23]);
        v = cfms(m2[r02], m2[s13], v);
        v = cfma(m2[r03], m2[s12], v);
        v = cfma(m2[r12], m2[s03], v);
        v = cfms(m2[r13], m2[s02], v);
        v = cfma(m2[r23], m2[s01], v);
        l = max(max(max(t2[r01] + t2[s23], t2[r02] + t2[s13]), max(t2[r03] + t2[s12], t2[r12] + t2[s03])),
                max(t2[r13] + t2[s02], t2[r23] + t2[s01]));
        return v;
    };
    const int* sub = S.sub + (size_t)s * MSD_KMAX;
    double2 v = cz(0, 0);
    int top = -(1 << 30);   // log2 of the largest product
    if (k == 3) {
        const size_t r0 = R2(0, 1, 1, 2), r1 = R2(0, 1, 0, 2), r2 = R2(0, 1, 0, 1);
        const double2 g0 = G(2, 0), g1 = G(2, 1), g2 = G(2, 2);
        v = cmul(g0, m2[r0]);
        v = cfms(g1, m2[r1], v);
        v = cscale(cfma(g2, m2[r2], v), sg);
        top = max(max(log_mag(g0) + t2[r0], log_mag(g1) + t2[r1]), log_mag(g2) + t2[r2]);
    } else if (subs && sub[0] >= 0) {
        for (int j = 0; j < k; ++j) {
            const int q = sub[j];
            double2 gj = G(k - 1, j);
            top = max(top, log_mag(gj) + tr[(size_t)((q >> 1) - S.bucket[3]) * nw]);
            if (q & 1) gj = cz(-gj.x, -gj.y);
            v = cfma(gj, S.rT[(size_t)(q >> 1) * nw + w], v);
        }
    } else if (k == 4) {
        v = cscale(M4(0, 1, 2, 3, 0, 1, 2, 3, top), sg);
    } else if (k == 5) {
        for (int j = 0; j < 5; ++j) {
            const int a = j > 0 ? 0 : 1, b = j > 1 ? 1 : 2, c = j > 2 ? 2 : 3, d = j > 3 ? 3 : 4;
            int l;
            const double2 m = M4(0, 1, 2, 3, a, b, c, d, l), gj = G(4, j);
            v = (j & 1) ? cfms(gj, m, v) : cfma(gj, m, v);
            top = max(top, log_mag(gj) + l);
        }
        v = cscale(v, sg);
    } else {
        // rows 4, 5 over all column pairs; sign (-1)^(4 + 5 + c + d)
        for (int c = 0; c < 5; ++c)
            for (int d = c + 1; d < 6; ++d) {
                auto q = [&](int j) { j += j >= c; return j + (j >= d); };   // the other columns
                int l;
                const double2 x = M4(0, 1, 2, 3, q(0), q(1), q(2), q(3), l), y = M2(4, 5, c, d);
                v = ((c + d) & 1) ? cfma(y, x, v) : cfms(y, x, v);
                top = max(top, l + t2[R2(4, 5, c, d)]);
            }
        v = cscale(v, sg);
    }
    *out = v;
    const bool lu = top - ((mag_key(v) >> 4) - (1023 << 16)) > (MINOR_BITS << 16);
    tr[(size_t)(s - S.bucket[3]) * nw] = (top & ~1) | (lu ? 1 : 0);
}

// The minors that k_minors marked, by LU: a block looks through LU_PAIRS (string, walker)
// pairs from string s0 on and then its threads take those marked (few: one in a warp
// would occupy all of it). With B their inverse minors too: entries as ratios of separately
// rounded minors are accurate one by one, but the string's energy cancels between them where
// the minor is close to low rank (rank one but for 1e-4, entries below 1: median error
// of the energy 1.7e-13 against 1.3e-13). No marks (tr NULL): all of them. 0.106 of the 0.78 ms that the
// ratios of 640 iron-sulfur walkers take; 12 us for 16 small ones, the latency of one LU.
#define LU_PAIRS 4096
#define LU_THREADS 128
template <bool INVERSE>
__global__ void __launch_bounds__(LU_THREADS) k_minor_lu(const __grid_constant__ MinorArgs a, int level0, int nw)
{
    const MinorSpin& S = a.s[blockIdx.y];
    __shared__ unsigned short list[LU_PAIRS];
    __shared__ int count;
    const int s0 = S.bucket[level0], t = threadIdx.x;
    const int n_all = S.vbucket[MSD_KMAX + 1] > S.n_str ? S.vbucket[MSD_KMAX + 1] : S.n_str;
    const long long pairs = (long long)(n_all - s0) * nw, e0 = blockIdx.x * (long long)LU_PAIRS;
    if (e0 >= pairs) return;
    const int n = (int)(pairs - e0 < LU_PAIRS ? pairs - e0 : LU_PAIRS);
    if (t == 0) count = S.tr ? 0 : n;
    __syncthreads();
    if (S.tr) {
        for (int i = t * 4; i < n; i += LU_THREADS * 4) {
            int m[4] = {0, 0, 0, 0};
            if (i + 4 <= n) {
                const int4 v = *reinterpret_cast<const int4*>(S.tr + e0 + i);
                m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w;
            } else {
                for (int q = 0; i + q < n; ++q) m[q] = S.tr[e0 + i + q];
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (m[q] & 1) list[atomicAdd(&count, 1)] = (unsigned short)(i + q);
        }
        __syncthreads();
    }
    const int total = count;
    for (int i = t; i < total; i += LU_THREADS) {
        const long long e = e0 + (S.tr ? list[i] : i);
        const int s = s0 + (int)(e / nw), w = (int)(e % nw);
        int k = 0;
        if (s < S.n_str) while (s >= S.bucket[k + 1]) ++k;
        else while (s >= S.vbucket[k + 1]) ++k;
        const uint4 rec = S.str_hp[s];
        const double2* g = S.GT + w;
        const double sg = S.str_sign[s];
        auto G = [&](int i, int j) { return g[(size_t)(rec_h(rec, i) * S.np + rec_p(rec, j)) * nw]; };
        double2* B = nullptr;
        if (INVERSE && s < S.n_str)
            B = S.B + S.b_off[k] + ((size_t)w * (S.bucket[k + 1] - S.bucket[k]) + s - S.bucket[k]) * b_stride(k);
        double2 r = cz(1, 0);
        switch (k) {
        case 0: break;
        case 1: r = minor_lu<1>(sg, G, INVERSE ? B : nullptr); break;
        case 2: r = minor_lu<2>(sg, G, INVERSE ? B : nullptr); break;
        case 3: r = minor_lu<3>(sg, G, INVERSE ? B : nullptr); break;
        case 4: r = minor_lu<4>(sg, G, INVERSE ? B : nullptr); break;
        case 5: r = minor_lu<5>(sg, G, INVERSE ? B : nullptr); break;
        default: r = minor_lu<6>(sg, G, INVERSE ? B : nullptr); break;
        }
        S.rT[(size_t)s * nw + w] = r;
    }
}

// ----------------------------------------------------------------- weights
struct WeightSpin {
    int n_str;
    const int* off;
    const int* other;
    const double* c;
    const double2* self;     // rT of this spin, [n_str][nw]
    const double2* opp;      // rT of the other spin
    double2* wts;            // [nw][n_str] r_s w_s (may be NULL)
    float2* rf;              // [nw][n_str] r_s in FP32 (may be NULL)
    double2* part;           // [nw][nslot] partial sums over 32 strings (may be NULL)
    double2* wT;             // [n_str][nw] the sums themselves (may be NULL)
    int* big;                // [nw] with wT: walkers (1) whose sums go to wT for vanishing ratios only, 2 if it has any
};
struct WeightArgs { WeightSpin s[2]; };

// w_s = sum over determinants I containing string s of c_I r_other(I); stored
// is r_s w_s (what every consumer needs). One block per tile of 32 strings and
// up to 32 walkers; a thread's sum runs in list order.
#define WT_S 32
__global__ void __launch_bounds__(256) k_weights(const __grid_constant__ WeightArgs a, int nw, int wt, int nslot)
{
    const WeightSpin& S = a.s[blockIdx.z];
    const int s0 = blockIdx.x * WT_S, w0 = blockIdx.y * wt;
    if (s0 >= S.n_str) return;
    __shared__ double2 tw[WT_S][33];
    __shared__ float2 tr[WT_S][33];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < WT_S * wt; e += 256) {
        const int sl = e / wt, wl = e - sl * wt, s = s0 + sl, w = w0 + wl;
        double2 rw = cz(0, 0), r = cz(0, 0);
        if (s < S.n_str && w < nw) {
            const double2* ro = S.opp + w;
            double2 acc = cz(0, 0);
            int i = S.off[s];
            const int i1 = S.off[s + 1];
            for (; i + 8 <= i1; i += 8) {
                int o[8];
                double c[8];
                double2 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) { o[q] = S.other[i + q]; c[q] = S.c[i + q]; }
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = ro[(size_t)o[q] * nw];
#pragma unroll
                for (int q = 0; q < 8; ++q) acc = cz(fma(v[q].x, c[q], acc.x), fma(v[q].y, c[q], acc.y));
            }
            for (; i < i1; ++i) {
                const double2 v = ro[(size_t)S.other[i] * nw];
                const double c = S.c[i];
                acc = cz(fma(v.x, c, acc.x), fma(v.y, c, acc.y));
            }
            r = S.self[(size_t)s * nw + w];
            if (S.wT) {
                const bool zero = r.x == 0 && r.y == 0;
                if (zero && S.big[w]) S.big[w] = 2;
                S.wT[(size_t)s * nw + w] = S.big[w] && !zero ? cz(0, 0) : acc;
            }
            rw = cmul(r, acc);
        }
        tw[sl][wl] = rw;
        if (S.rf) tr[sl][wl] = make_float2((float)r.x, (float)r.y);
    }
    __syncthreads();
    const int s = s0 + lane;
    for (int wl = warp; wl < wt && w0 + wl < nw; wl += 8) {
        const size_t w = w0 + wl;
        double2 v = tw[lane][wl];
        if (s < S.n_str) {
            if (S.wts) S.wts[w * S.n_str + s] = v;
            if (S.rf) S.rf[w * S.n_str + s] = tr[lane][wl];
        }
        if (S.part) {
            for (int o = 16; o; o >>= 1) {
                v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
                v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
            }
            if (lane == 0) S.part[w * nslot + blockIdx.x] = v;
        }
    }
}

// r[w][s] = rT[s][w]
__global__ void __launch_bounds__(256) k_untranspose(int n_str, int nw, const double2* __restrict__ rT, double2* __restrict__ r)
{
    __shared__ double2 tile[32][33];
    const int s0 = blockIdx.x * 32, w0 = blockIdx.y * 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < 32; i += 8)
        if (s0 + i < n_str && w0 + lane < nw) tile[i][lane] = rT[(size_t)(s0 + i) * nw + w0 + lane];
    __syncthreads();
    for (int i = warp; i < 32; i += 8)
        if (w0 + i < nw && s0 + lane < n_str) r[(size_t)(w0 + i) * n_str + s0 + lane] = tile[lane][i];
}

// ------------------------------------------------------ FP32 inverse minors
struct InvSpin {
    int nh, np;
    int bucket[MSD_KMAX + 2];
    const uint4* str_hp;
    const double2* Gact;     // [nw][nh np]
    float2* B;
    long long b_off[MSD_KMAX + 2];
    int blk[MSD_KMAX + 2];   // first block of each level
};
struct InvArgs { InvSpin s[2]; };

// B = A^-1 of one string in FP32: elimination with partial pivoting by the
// larger of |Re|, |Im| (compared to 20 mantissa bits), column solves, then the
// K^2 entries (and the pad) as 16-byte stores.
template <int K>
__device__ __forceinline__ void inverse_minor(const uint4 rec, int np, const float2* __restrict__ gf, float2* __restrict__ B)
{
    float2 lu[K][K], di[K];
    int perm[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        perm[i] = i;
#pragma unroll
        for (int j = 0; j < K; ++j) lu[i][j] = gf[rec_h(rec, i) * np + rec_p(rec, j)];
    }
    auto key = [](float2 v) { return max(__float_as_int(v.x) & 0x7fffffff, __float_as_int(v.y) & 0x7fffffff) >> 3; };
#pragma unroll
    for (int k = 0; k < K; ++k) {
        int p = k, best = key(lu[k][k]);
#pragma unroll
        for (int i = k + 1; i < K; ++i) {
            const int v = key(lu[i][k]);
            if (v > best) { best = v; p = i; }
        }
#pragma unroll
        for (int i = k + 1; i < K; ++i)
            if (i == p) {
#pragma unroll
                for (int j = 0; j < K; ++j) { const float2 t = lu[k][j]; lu[k][j] = lu[i][j]; lu[i][j] = t; }
                const int t = perm[k]; perm[k] = perm[i]; perm[i] = t;
            }
        const float m2 = fmaf(lu[k][k].x, lu[k][k].x, lu[k][k].y * lu[k][k].y);
        const float im2 = !(m2 > 0.f) ? 0.f : 1.f / m2;
        di[k] = make_float2(lu[k][k].x * im2, -lu[k][k].y * im2);
#pragma unroll
        for (int i = k + 1; i < K; ++i) {
            const float2 f = fmul(lu[i][k], di[k]);
            lu[i][k] = f;
#pragma unroll
            for (int j = k + 1; j < K; ++j) {
                lu[i][j].x -= f.x * lu[k][j].x - f.y * lu[k][j].y;
                lu[i][j].y -= f.x * lu[k][j].y + f.y * lu[k][j].x;
            }
        }
    }
    float2 inv[K * K + (K & 1)];
    if (K & 1) inv[K * K] = make_float2(0.f, 0.f);   // the pad entry
#pragma unroll
    for (int c = 0; c < K; ++c) {
        float2 x[K];
#pragma unroll
        for (int i = 0; i < K; ++i) x[i] = make_float2(perm[i] == c ? 1.f : 0.f, 0.f);
#pragma unroll
        for (int i = 0; i < K; ++i)
#pragma unroll
            for (int k = 0; k < i; ++k) {
                x[i].x -= lu[i][k].x * x[k].x - lu[i][k].y * x[k].y;
                x[i].y -= lu[i][k].x * x[k].y + lu[i][k].y * x[k].x;
            }
#pragma unroll
        for (int i = K - 1; i >= 0; --i) {
#pragma unroll
            for (int k = i + 1; k < K; ++k) {
                x[i].x -= lu[i][k].x * x[k].x - lu[i][k].y * x[k].y;
                x[i].y -= lu[i][k].x * x[k].y + lu[i][k].y * x[k].x;
            }
            const float2 t = x[i];
            x[i] = make_float2(t.x * di[i].x - t.y * di[i].y, t.x * di[i].y + t.y * di[i].x);
        }
#pragma unroll
        for (int i = 0; i < K; ++i) inv[i * K + c] = x[i];
    }
#pragma unroll
    for (int e = 0; e < b_stride(K); e += 2)
        *reinterpret_cast<float4*>(B + e) = make_float4(inv[e].x, inv[e].y, inv[e + 1].x, inv[e + 1].y);
}

__global__ void __launch_bounds__(128) k_inverse_minors(const __grid_constant__ InvArgs a)
{
    const InvSpin& S = a.s[blockIdx.z];
    __shared__ float2 gf[MSD_XMAX];
    const int w = blockIdx.y, X = S.nh * S.np;
    if ((int)blockIdx.x >= S.blk[MSD_KMAX + 1]) return;
    for (int e = threadIdx.x; e < X; e += 128) {
        const double2 v = S.Gact[(size_t)w * X + e];
        gf[e] = make_float2((float)v.x, (float)v.y);
    }
    __syncthreads();
    int k = 1;
    while ((int)blockIdx.x >= S.blk[k + 1]) ++k;
    const int ns = S.bucket[k + 1] - S.bucket[k], sl = ((int)blockIdx.x - S.blk[k]) * 128 + threadIdx.x;
    if (sl >= ns) return;
    const uint4 rec = S.str_hp[S.bucket[k] + sl];
    float2* B = S.B + S.b_off[k] + ((size_t)w * ns + sl) * b_stride(k);
    switch (k) {
    case 1: inverse_minor<1>(rec, S.np, gf, B); break;
    case 2: inverse_minor<2>(rec, S.np, gf, B); break;
    case 3: inverse_minor<3>(rec, S.np, gf, B); break;
    case 4: inverse_minor<4>(rec, S.np, gf, B); break;
    case 5: inverse_minor<5>(rec, S.np, gf, B); break;
    default: inverse_minor<6>(rec, S.np, gf, B); break;
    }
}

// ------------------------------------------------------ FP64 inverse minors
// B = A^-1 of every string as its cofactors over its determinant. The cofactors are
// the (k - 1)-minors that the ratios' expansions leave (and the sub-minors that the
// trial does not hold, appended to its strings): 4 FP64 FMAs per entry and one
// reciprocal per string, against 8 k^3 / 3 and k reciprocals of an LU with its column
// solves, which the FP64 unit bounds. The relative error of an entry is that of two
// minors. Bound by memory now: k^2 gathered rows of the walkers in, k^2
// entries out per string and walker. A warp takes 32 (string, walker) pairs, walkers
// fastest, and writes their entries through shared memory, up to 16 (256 bytes) of a
// pair at a time. 640 copper-oxo walkers, ratios and inverses 3.06 -> 1.44 ms.
// Walkers with large active blocks are done again by LU (k_strings_large in k_wick.cu).
struct InvRatioSpin {
    int bucket[MSD_KMAX + 2];
    const int* row;
    long long row_off[MSD_KMAX + 2];
    const double2* V;        // [row][nw]
    const double2* r;        // [string][nw], within V
    double2* B;
    long long b_off[MSD_KMAX + 2];
    const int* tr;           // from level 3 on: marked ones have theirs (k_minor_lu)
    int blk[MSD_KMAX + 2];   // first block of each level
};
struct InvRatioArgs { InvRatioSpin s[2]; };

#define IR_E 16   // entries per pass
template <int K>
__device__ __forceinline__ void inverse_ratios(const InvRatioSpin& S, int nw, double2 (*tile)[IR_E + 1])
{
    constexpr int KK = K * K, KST = b_stride(K);
    const int ns = S.bucket[K + 1] - S.bucket[K], lane = threadIdx.x & 31;
    const long long items = (long long)ns * nw;
    const long long e0 = ((long long)blockIdx.x - S.blk[K]) * 128 + (threadIdx.x & ~31), e = e0 + lane;
    if (e0 >= items) return;
    const bool on = e < items;
    // 32-bit division where the count allows it
    const int sl = !on ? 0 : items < 0x7fffffff ? (int)((unsigned)e / (unsigned)nw) : (int)(e / nw);
    const int w = on ? (int)(e - (long long)sl * nw) : 0;
    const double2 r = S.r[(size_t)(S.bucket[K] + sl) * nw + w];
    // 1 / r at a scale where |r|^2 neither underflows nor overflows; 0 for r = 0
    const double m = fmax(fabs(r.x), fabs(r.y));
    const int ex = min(1000, max(-1000, ((__double2hiint(m) >> 20) & 2047) - 1023));
    const double sc = __hiloint2double((1023 - ex) << 20, 0);
    const double2 q = cscale(r, sc);
    const double d = r.x == 0 && r.y == 0 ? 0.0 : 1.0 / fma(q.x, q.x, q.y * q.y);
    const double2 inv = cz(q.x * d * sc, -q.y * d * sc);
    const int* row = S.row + S.row_off[K] + (size_t)sl * KK;
    const double2* V = S.V + w;
    const long long base = ((long long)w * ns + sl) * KST;
    double2* B = S.B + S.b_off[K];
    const bool mine = on && !(K >= 3 && (S.tr[(size_t)(S.bucket[K] - S.bucket[3] + sl) * nw + w] & 1));
    const unsigned write = __ballot_sync(0xffffffffu, mine);
#pragma unroll 1
    for (int p = 0; p < KST; p += IR_E) {
        const int n = KST < IR_E ? KST : min(IR_E, KST - p);
#pragma unroll 4
        for (int i = 0; i < n; ++i) {
            double2 v = cz(0, 0);
            if (p + i < KK) {
                const int c = row[p + i];
                if (K == 1) v = inv;
                else v = cmul(V[(size_t)(c >> 1) * nw], inv);
                if (c & 1) v = cz(-v.x, -v.y);
            }
            tile[lane][i] = v;
        }
        __syncwarp();
        for (int i = 0; i < n; ++i) {
            const int f = i * 32 + lane, it = f / n;   // pair, entry
            const long long b = __shfl_sync(0xffffffffu, base, it);
            if (write >> it & 1) B[b + p + f - it * n] = tile[it][f - it * n];
        }
        __syncwarp();
    }
}

__global__ void __launch_bounds__(128) k_inverse_ratios(const __grid_constant__ InvRatioArgs a, int nw)
{
    const InvRatioSpin& S = a.s[blockIdx.y];
    __shared__ double2 tile[4][32][IR_E + 1];
    if ((int)blockIdx.x >= S.blk[MSD_KMAX + 1]) return;
    int k = 1;
    while ((int)blockIdx.x >= S.blk[k + 1]) ++k;
    double2 (*t)[IR_E + 1] = tile[threadIdx.x >> 5];
    switch (k) {
    case 1: inverse_ratios<1>(S, nw, t); break;
    case 2: inverse_ratios<2>(S, nw, t); break;
    case 3: inverse_ratios<3>(S, nw, t); break;
    case 4: inverse_ratios<4>(S, nw, t); break;
    case 5: inverse_ratios<5>(S, nw, t); break;
    default: inverse_ratios<6>(S, nw, t); break;
    }
}

MinorSpin minor_spin(const SpinTables& t, const double2* GT, double2* m2, double2* rT, int* t2, int* tr)
{
    MinorSpin s;
    s.nh = t.nh; s.np = t.np; s.n_str = t.n_str;
    for (int k = 0; k < MSD_KMAX + 2; ++k) { s.bucket[k] = t.bucket[k]; s.vbucket[k] = 0; }
    s.str_hp = t.str_hp; s.str_sign = t.str_sign; s.sub = t.sub;
    s.GT = GT; s.m2 = m2; s.rT = rT; s.t2 = t2; s.tr = tr;
    s.B = nullptr;
    for (int k = 0; k < MSD_KMAX + 2; ++k) s.b_off[k] = t.b_off[k];
    return s;
}

// The marked minors of both spins from level 3 on (all of every level without marks).
void launch_lu(const MinorArgs& a, int nw, cudaStream_t st)
{
    const int level0 = a.s[0].tr ? 3 : 0;
    long long n = 0;
    for (const MinorSpin& s : a.s) n = std::max(n, (long long)std::max(s.n_str, s.vbucket[MSD_KMAX + 1]) - s.bucket[level0]);
    if (n <= 0) return;
    const dim3 grid((unsigned)((n * nw + LU_PAIRS - 1) / LU_PAIRS), 2);
    if (a.s[0].B) k_minor_lu<true><<<grid, LU_THREADS, 0, st>>>(a, level0, nw);
    else k_minor_lu<false><<<grid, LU_THREADS, 0, st>>>(a, level0, nw);
    msd_note_launch();
}

// ------------------------------------------------------------- cofactors
// Cofactor matrix of the FP64 force bias and density matrix,
//   Cm[p][h] = sum_s w_s r_s B_s[i][j] at (p_i, h_j) = (p, h),
// from the cofactors r_s B_s themselves, which are rows of V: no inverse minor, and right
// where a ratio vanishes and its cofactors do not. An entry's list holds (row of V, string,
// sign); the lists are cut in pieces of 64 (few entries with long lists), then the
// pieces are added. 4 FP64 FMAs and two 16-byte rows of a warp's 32 walkers per entry.
// Walkers with a large active block (k_large in k_wick.cu) take theirs from the LU's
// inverse minors, the vanishing ratios excepted. 640 copper-oxo walkers 0.76 ms. (Reverse
// differentiation of the expansions takes half the operations, 0.65 ms; but it sums the
// cofactors' own expansions again, with their cancellation.)
struct CofSpin {
    int t0, t1;              // targets of this launch
    const int* row;          // [target] row of Bv, or entry of G (the sums)
    const int* off;          // [target + 1]
    const int2* ent;         // (a << 1 | negative, b): +-V[a] Bv[b]; a = -1: +-Bv[b]
    const double2* V;
    double2* Bv;
    double2* Cm;             // the sums: [nw][np][nh], entry x = h np + p to p nh + h
    const int* big;          // [nw] 1: nothing to sum for the walker
    int nh, np;
};
struct CofArgs { CofSpin s[2]; };

__global__ void __launch_bounds__(256) k_cofactors(const __grid_constant__ CofArgs args, int nw)
{
    const CofSpin& S = args.s[blockIdx.y];
    const long long e = blockIdx.x * 256ll + threadIdx.x;
    if (e >= (long long)(S.t1 - S.t0) * nw) return;
    const int t = S.t0 + (int)(e / nw), w = (int)(e % nw);
    double2 acc = cz(0, 0);
    const int i1 = S.big[w] == 1 ? 0 : S.off[t + 1];
    for (int i = S.off[t]; i < i1; i += 4) {
        double2 a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (i + q < i1) {
                const int2 c = S.ent[i + q];
                a[q] = c.x >= 0 ? S.V[(size_t)(c.x >> 1) * nw + w] : cz(1, 0);
                b[q] = S.Bv[(size_t)c.y * nw + w];
                if (c.x & 1) b[q] = cz(-b[q].x, -b[q].y);
            } else {
                a[q] = b[q] = cz(0, 0);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (i + q < i1) acc = cfma(a[q], b[q], acc);
    }
    const int r = S.row[t];
    if (S.Cm) {
        const int h = r / S.np, p = r - h * S.np;
        S.Cm[(size_t)w * S.nh * S.np + p * S.nh + h] = acc;
    } else {
        S.Bv[(size_t)r * nw + w] = acc;
    }
}

}  // namespace

// Ratios of the trial's strings and of the sub-minors outside it.
void launch_minors_ext(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw, double2* const V[2],
                       int* const t2[2], int* const tr[2], void* const B[2], cudaStream_t st)
{
    MinorArgs a;
    const SpinTables* T[2] = {&ta, &tb};
    for (int s = 0; s < 2; ++s) {
        double2* m2 = V[s] + (size_t)T[s]->nh * T[s]->np * nw;
        a.s[s] = minor_spin(*T[s], V[s], m2, m2 + (size_t)g[s].n2 * nw, t2[s], tr[s]);
        a.s[s].B = B ? (double2*)B[s] : nullptr;
        a.s[s].str_hp = g[s].str_hp; a.s[s].str_sign = g[s].str_sign; a.s[s].sub = g[s].sub;
        for (int k = 0; k < MSD_KMAX + 2; ++k) a.s[s].vbucket[k] = g[s].vbucket[k];
    }
    auto blocks = [&](long long n) { return dim3((unsigned)((n * nw + 255) / 256), 2); };
    k_minor2<<<blocks(std::max(1, std::max(g[0].n2, g[1].n2))), 256, 0, st>>>(a, nw);
    msd_note_launch();
    auto count = [&](int s, int k) {
        return T[s]->bucket[k + 1] - T[s]->bucket[k] + g[s].vbucket[k + 1] - g[s].vbucket[k];
    };
    k_minors<<<blocks(std::max(ta.bucket[3], tb.bucket[3])), 256, 0, st>>>(a, 0, 2, false, nw);
    msd_note_launch();
    for (int k = 3; k <= MSD_KMAX; ++k) {
        const int n = std::max(count(0, k), count(1, k));
        if (n <= 0) continue;
        k_minors<<<blocks(n), 256, 0, st>>>(a, k, k, true, nw);
        msd_note_launch();
    }
    launch_lu(a, nw, st);
}

void launch_cofactors(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw, double2* const V[2],
                      double2* const Bv[2], double2* const Cm[2], int* const big[2], cudaStream_t st)
{
    const SpinTables* T[2] = {&ta, &tb};
    for (int sums = 0; sums < 2; ++sums) {
        CofArgs a;
        int n = 0;
        for (int s = 0; s < 2; ++s) {
            const int t0 = sums ? g[s].n_piece : 0, t1 = g[s].n_piece + (sums ? T[s]->nh * T[s]->np : 0);
            a.s[s] = CofSpin{t0, t1, g[s].cof_row, g[s].cof_off, g[s].cof_ent, V[s], Bv[s], sums ? Cm[s] : nullptr, big[s],
                             T[s]->nh, T[s]->np};
            n = std::max(n, t1 - t0);
        }
        if (n <= 0) continue;
        k_cofactors<<<dim3((unsigned)(((long long)n * nw + 255) / 256), 2), 256, 0, st>>>(a, nw);
        msd_note_launch();
    }
}

size_t minor2_count(const SpinTables& t)
{
    return std::max<size_t>(1, (size_t)(t.nh * (t.nh - 1) / 2) * (t.np * (t.np - 1) / 2));
}

size_t minor_marks(const SpinTables& t) { return std::max(1, t.n_str - t.bucket[3]); }

void launch_minors(const SpinTables& ta, const SpinTables& tb, int nw, double2* const GT[2], double2* const m2[2],
                   int* const t2[2], int* const tr[2], double2* const rT[2], cudaStream_t st)
{
    const MinorArgs a = {{minor_spin(ta, GT[0], m2[0], rT[0], t2[0], tr[0]), minor_spin(tb, GT[1], m2[1], rT[1], t2[1], tr[1])}};
    if (!m2[0]) { launch_lu(a, nw, st); return; }
    auto blocks = [&](long long n) { return dim3((unsigned)((n * nw + 255) / 256), 2); };
    k_minor2<<<blocks(std::max(minor2_count(ta), minor2_count(tb))), 256, 0, st>>>(a, nw);
    msd_note_launch();
    // Level 4 over the level-3 ratios takes 4 complex products instead of 6, but a
    // launch of its own: only where there are many (the launch costs about what
    // 1000 strings' two products do for a few hundred walkers).
    auto count = [&](int k0, int k1) {
        return std::max(ta.bucket[k1 + 1] - ta.bucket[k0], tb.bucket[k1 + 1] - tb.bucket[k0]);
    };
    const bool four = count(4, 4) >= 1000;
    k_minors<<<blocks(count(0, four ? 3 : 4)), 256, 0, st>>>(a, 0, four ? 3 : 4, false, nw);
    msd_note_launch();
    for (int k = four ? 4 : 5; k <= MSD_KMAX; ++k) {
        if (count(k, k) <= 0) continue;
        k_minors<<<blocks(count(k, k)), 256, 0, st>>>(a, k, k, true, nw);
        msd_note_launch();
    }
    launch_lu(a, nw, st);
}

void launch_inverse_minors(const SpinTables& ta, const SpinTables& tb, int nw, double2* const Gact[2], void* const B[2],
                           cudaStream_t st)
{
    InvArgs args;
    InvSpin* s = args.s;
    const SpinTables* t[2] = {&ta, &tb};
    int nb = 0;
    for (int i = 0; i < 2; ++i) {
        s[i].nh = t[i]->nh; s[i].np = t[i]->np;
        s[i].str_hp = t[i]->str_hp;
        s[i].Gact = Gact[i]; s[i].B = (float2*)B[i];
        s[i].blk[0] = s[i].blk[1] = 0;
        for (int k = 0; k < MSD_KMAX + 2; ++k) { s[i].bucket[k] = t[i]->bucket[k]; s[i].b_off[k] = t[i]->b_off[k]; }
        for (int k = 1; k <= MSD_KMAX; ++k)
            s[i].blk[k + 1] = s[i].blk[k] + (s[i].bucket[k + 1] - s[i].bucket[k] + 127) / 128;
        nb = std::max(nb, s[i].blk[MSD_KMAX + 1]);
    }
    if (nb <= 0) return;
    k_inverse_minors<<<dim3(nb, nw, 2), 128, 0, st>>>(args);
    msd_note_launch();
}

void launch_inverse_ratios(const ExtTables g[2], const SpinTables& ta, const SpinTables& tb, int nw,
                           double2* const V[2], int* const tr[2], void* const B[2], cudaStream_t st)
{
    InvRatioArgs args;
    const SpinTables* t[2] = {&ta, &tb};
    int nb = 0;
    for (int i = 0; i < 2; ++i) {
        InvRatioSpin& s = args.s[i];
        s.row = g[i].row; s.V = V[i]; s.B = (double2*)B[i]; s.tr = tr[i];
        s.r = V[i] + ((size_t)t[i]->nh * t[i]->np + g[i].n2) * nw;
        s.blk[0] = s.blk[1] = 0;
        for (int k = 0; k < MSD_KMAX + 2; ++k) {
            s.bucket[k] = t[i]->bucket[k]; s.b_off[k] = t[i]->b_off[k]; s.row_off[k] = t[i]->cmx_off[k];
        }
        for (int k = 1; k <= MSD_KMAX; ++k)
            s.blk[k + 1] = s.blk[k] + (int)(((long long)(s.bucket[k + 1] - s.bucket[k]) * nw + 127) / 128);
        nb = std::max(nb, s.blk[MSD_KMAX + 1]);
    }
    if (nb <= 0) return;
    k_inverse_ratios<<<dim3(nb, 2), 128, 0, st>>>(args, nw);
    msd_note_launch();
}

int weights_blocks(const SpinTables& tb) { return (tb.n_str + WT_S - 1) / WT_S; }

// wts, rf: per spin, NULL where not wanted; beta = false: the alpha sums alone.
void launch_weights(const SpinTables& ta, const SpinTables& tb, int nw, double2* const rT[2], double2* const wts[2],
                    float2* const rf[2], double2* part, int nslot, bool beta, cudaStream_t st, double2* const wT[2],
                    int* const big[2])
{
    const WeightArgs a = {{{ta.n_str, ta.csr_off, ta.csr_other, ta.csr_c, rT[0], rT[1], wts[0], rf[0], part,
                           wT ? wT[0] : nullptr, wT ? big[0] : nullptr},
                          {tb.n_str, tb.csr_off, tb.csr_other, tb.csr_c, rT[1], rT[0], wts[1], rf[1], nullptr,
                           wT ? wT[1] : nullptr, wT ? big[1] : nullptr}}};
    const int tiles = (nw + 31) / 32, wt = (nw + tiles - 1) / tiles;   // walkers per tile, evenly
    const int nb = beta ? std::max(weights_blocks(ta), weights_blocks(tb)) : weights_blocks(ta);
    k_weights<<<dim3(nb, tiles, beta ? 2 : 1), 256, 0, st>>>(a, nw, wt, nslot);
    msd_note_launch();
}

void launch_untranspose(int n_str, int nw, const double2* rT, double2* r, cudaStream_t st)
{
    k_untranspose<<<dim3((n_str + 31) / 32, (nw + 31) / 32), 256, 0, st>>>(n_str, nw, rT, r);
    msd_note_launch();
}
