// The per-determinant energy terms as a block of the per-system kernels (k_energy.cu,
// k_pair.cu) and of the persistent batched kernel (k_batch.cu) evaluates them: the
// walker's tables in shared memory and one string's or determinant's term, in FP32
// (mixed mode) or, in FP64 mode, with the long sums in the two-limb fixed point of
// fixed.cuh.
#pragma once

#include <type_traits>

#include "det_terms.cuh"
#include "fixed.cuh"

// The walker's K^{ab} in shared memory: FP32 entries, or in FP64 mode limbs of
// fixed.cuh (the same 16 bytes) with their exponent.
template <typename T>
struct PairK { const cplx_t<T>* k; };
template <>
struct PairK<double> { const Limbs* k; int e; };

template <typename T>
__device__ __forceinline__ PairK<T> load_pair_k(const void* Kin, int w, int XX, unsigned char* sm)
{
    const cplx_t<T>* Kw = reinterpret_cast<const cplx_t<T>*>(Kin) + (size_t)w * XX;
    cplx_t<T>* ks = reinterpret_cast<cplx_t<T>*>(sm);
    if constexpr (std::is_same<T, float>::value) {
        for (int e = threadIdx.x; e < XX; e += blockDim.x) ks[e] = Kw[e];
        __syncthreads();
        return {ks};
    } else {
        __shared__ unsigned wm[32];
        unsigned m = 0;
        for (int e = threadIdx.x; e < XX; e += blockDim.x) {
            const double2 v = Kw[e];
            ks[e] = v;
            m = max(m, mag_bits(v));
        }
        const int ex = mag_exponent(block_mag(m, wm));
        Limbs* l = reinterpret_cast<Limbs*>(sm);
        for (int e = threadIdx.x; e < XX; e += blockDim.x) l[e] = to_limbs(ks[e], ex);   // its own entries
        __syncthreads();
        return {l, ex};
    }
}

// FP64 mode: c_I r_a r_b X_ab with the sum over the entries of the longer string's
// minor in fixed point (scales: K, and the string's largest entry) and the sum over
// the shorter one's in FP64. The FP64 unit bounds the plain double sum, 4 k_a^2
// k_b^2 FMAs: (3, 3) determinants 360 FP64 operations, here 52 and 972 mad.wide.
// A thread per determinant, for the batched kernel (its items share a block shape);
// the per-system kernels use pair_lanes.
template <int KA, int KB>
__device__ __forceinline__ double2 pair_term_fixed(const SpinTables& ta, const SpinTables& tbb, const PairTables& pt,
                                                   int I, int w, const void* __restrict__ Ba_in,
                                                   const void* __restrict__ Bb_in, const PairK<double>& kk,
                                                   const double2* __restrict__ ra, const double2* __restrict__ rb)
{
    constexpr bool INB = KB >= KA;
    constexpr int KI = INB ? KB : KA, KO = INB ? KA : KB;
    const int Xb = tbb.nh * tbb.np, a = pt.a[I], b = pt.b[I];
    const int nsa = ta.bucket[KA + 1] - ta.bucket[KA], nsb = tbb.bucket[KB + 1] - tbb.bucket[KB];
    const double2* Ba = reinterpret_cast<const double2*>(Ba_in) + (size_t)ta.b_off[KA] +
                        ((size_t)w * nsa + a - ta.bucket[KA]) * b_stride(KA);
    const double2* Bb = reinterpret_cast<const double2*>(Bb_in) + (size_t)tbb.b_off[KB] +
                        ((size_t)w * nsb + b - tbb.bucket[KB]) * b_stride(KB);
    const double2 *Bi = INB ? Bb : Ba, *Bo = INB ? Ba : Bb;
    const uint4 ri = INB ? tbb.str_hp[b] : ta.str_hp[a], ro = INB ? ta.str_hp[a] : tbb.str_hp[b];
    const int npi = INB ? tbb.np : ta.np, npo = INB ? ta.np : tbb.np, si = INB ? 1 : Xb, so = INB ? Xb : 1;
    const double2 rav = ra[(size_t)w * ta.n_str + a], rbv = rb[(size_t)w * tbb.n_str + b];
    Limbs bi[KI * KI];
    int xi[KI * KI], eb;
    {
        double2 v[KI * KI];
        unsigned m = 0;
#pragma unroll
        for (int e = 0; e < KI * KI; ++e) { v[e] = Bi[e]; m = max(m, mag_bits(v[e])); }
        eb = mag_exponent(m);
#pragma unroll
        for (int e = 0; e < KI * KI; ++e) {
            bi[e] = to_limbs(v[e], eb);
            xi[e] = (rec_h(ri, e % KI) * npi + rec_p(ri, e / KI)) * si;
        }
    }
    double xr = 0, xim = 0;
#pragma unroll 1
    for (int e = 0; e < KO * KO; ++e) {
        const double2 bo = Bo[e];
        const Limbs* krow = kk.k + (rec_h(ro, e % KO) * npo + rec_p(ro, e / KO)) * so;
        LimbSum s;
#pragma unroll
        for (int q = 0; q < KI * KI; ++q) s.add(bi[q], krow[xi[q]]);
        const double2 z = limb_value(s, kk.e + eb);
        xr += bo.x * z.x - bo.y * z.y;
        xim += bo.x * z.y + bo.y * z.x;
    }
    if (max(kk.e, eb) >= FIXED_EXP_INF) xr = xim = __longlong_as_double(0x7ff8000000000000ll);
    return pair_weight_times<double>(pt, I, rav, rbv, xr, xim);
}

template <int KA, int KB, typename T>
__device__ __forceinline__ cplx_t<T> pair_term(const SpinTables& ta, const SpinTables& tbb, const PairTables& pt, int I,
                                               int w, const void* Ba, const void* Bb, const PairK<T>& kk,
                                               const cplx_t<T>* ra, const cplx_t<T>* rb)
{
    if constexpr (std::is_same<T, float>::value)
        return pair_cross_term2<KA, KB, T>(ta, tbb, pt, I, w, Ba, Bb, kk.k, ra, rb);
    else
        return pair_term_fixed<KA, KB>(ta, tbb, pt, I, w, Ba, Bb, kk, ra, rb);
}

// FP64 mode: this block's determinants (PC_THREADS PC_PER_THREAD of the n from lo) in
// the sums of pair_term_fixed, with a group of lanes to a determinant, each taking
// k_o (k_o = 2: one) of the k_o^2 entries of the shorter string's minor. The longer
// one's limbs are made once, by the group's lanes, in shared memory (bs, pair_limbs
// entries); where the shorter has one entry they are used as they are made. A thread
// per determinant holds them and their table offsets in registers (226 at (2, 4), 164
// at (3, 3)): 8 warps per SM, each instruction waiting for the last. 640 copper-oxo
// walkers 3.31 -> 2.05 ms, 64 iron-sulfur ones 3.37 -> 2.24.
__host__ __device__ __forceinline__ constexpr int pair_group(int ka, int kb)
{
    const int ko = ka < kb ? ka : kb;
    return ko == 2 ? 4 : ko;
}
__host__ __device__ __forceinline__ constexpr int pair_limbs(int ka, int kb, int threads)
{
    const int ki = ka < kb ? kb : ka, g = pair_group(ka, kb);
    return g == 1 ? 0 : threads / 32 * (32 / g) * ((ki * ki) | 1);
}

template <int KA, int KB>
__device__ __forceinline__ double2 pair_lanes(const SpinTables& ta, const SpinTables& tbb, const PairTables& pt, int lo,
                                              int n, int blk, int w, const double2* Ba_in, const double2* Bb_in,
                                              const PairK<double>& kk, const double2* ra, const double2* rb, Limbs* bs)
{
    constexpr bool INB = KB >= KA;
    constexpr int KI = INB ? KB : KA, KO = INB ? KA : KB, G = pair_group(KA, KB), DPW = 32 / G, NE = KO * KO / G;
    constexpr int NI = KI * KI, EPL = (NI + G - 1) / G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane / G, j = lane - g * G;
    const int Xb = tbb.nh * tbb.np;
    const int nsa = ta.bucket[KA + 1] - ta.bucket[KA], nsb = tbb.bucket[KB + 1] - tbb.bucket[KB];
    const int npi = INB ? tbb.np : ta.np, npo = INB ? ta.np : tbb.np, si = INB ? 1 : Xb, so = INB ? Xb : 1;
    bs += (warp * DPW + (g < DPW ? g : 0)) * (NI | 1);
    const int i0 = blk * (PC_THREADS * PC_PER_THREAD), i1 = min(n, i0 + PC_THREADS * PC_PER_THREAD);
    double2 sum = cz(0, 0);
    for (int base = i0 + warp * DPW; base < i1; base += (int)(blockDim.x >> 5) * DPW) {
        const bool on = g < DPW && base + g < i1;
        const int I = lo + (on ? base + g : base), a = pt.a[I], b = pt.b[I];
        const double2* Ba = Ba_in + (size_t)ta.b_off[KA] + ((size_t)w * nsa + a - ta.bucket[KA]) * b_stride(KA);
        const double2* Bb = Bb_in + (size_t)tbb.b_off[KB] + ((size_t)w * nsb + b - tbb.bucket[KB]) * b_stride(KB);
        const double2 *Bi = INB ? Bb : Ba, *Bo = INB ? Ba : Bb;
        const uint4 ri = INB ? tbb.str_hp[b] : ta.str_hp[a], ro = INB ? ta.str_hp[a] : tbb.str_hp[b];
        const double2 rav = ra[(size_t)w * ta.n_str + a], rbv = rb[(size_t)w * tbb.n_str + b];
        double2 v[G == 1 ? KI : EPL];   // one lane: a row at a time
        unsigned m = 0;
        if constexpr (G == 1) {
#pragma unroll 1
            for (int i = 0; i < KI; ++i)
#pragma unroll
                for (int l = 0; l < KI; ++l) m = max(m, mag_bits(Bi[i * KI + l]));
        } else {
#pragma unroll
            for (int q = 0; q < EPL; ++q) {
                v[q] = j + q * G < NI ? Bi[j + q * G] : cz(0, 0);
                m = max(m, mag_bits(v[q]));
            }
#pragma unroll
            for (int d = 1; d < G; ++d)   // the group's largest: lanes j + 1 on, in a circle
                m = max(m, __shfl_sync(0xffffffffu, m, (g * G + (j + d) % G) & 31));
        }
        const int eb = mag_exponent(m);
        int hx[KI];
#pragma unroll
        for (int l = 0; l < KI; ++l) hx[l] = rec_h(ri, l) * npi * si;
        double2 x = cz(0, 0);
        if constexpr (G > 1) {
            __syncwarp();   // the previous determinants' limbs consumed
            if (g < DPW)
#pragma unroll
                for (int q = 0; q < EPL; ++q)
                    if (j + q * G < NI) bs[j + q * G] = to_limbs(v[q], eb);
            __syncwarp();
        }
#pragma unroll 1
        for (int o = 0; o < NE; ++o) {
            const int e = j * NE + o;
            const Limbs* krow = kk.k + (rec_h(ro, e % KO) * npo + rec_p(ro, e / KO)) * so;
            LimbSum s;
#pragma unroll 1
            for (int i = 0; i < KI; ++i) {
                const Limbs* kp = krow + rec_p(ri, i) * si;
                if constexpr (G == 1) {
#pragma unroll
                    for (int l = 0; l < KI; ++l) v[l] = Bi[i * KI + l];
                }
#pragma unroll
                for (int l = 0; l < KI; ++l) {
                    if constexpr (G == 1) s.add(to_limbs(v[l], eb), kp[hx[l]]);
                    else s.add(bs[i * KI + l], kp[hx[l]]);
                }
            }
            const double2 z = limb_value(s, kk.e + eb), bo = Bo[e];
            x = cfma(bo, z, x);
        }
        if (on) {
            if (max(kk.e, eb) >= FIXED_EXP_INF) x.x = x.y = __longlong_as_double(0x7ff8000000000000ll);
            // fused explicitly: the same rounding in every kernel that holds this
            sum = cfma(cfma(rav, rbv, cz(0, 0)), cscale(x, pt.c[I]), sum);
        }
    }
    return sum;
}

// One block's part of the opposite-spin term of levels (KA, KB), this thread's share:
// in FP64 mode by groups of lanes (LANES, bs with room for their limbs), else a thread
// per determinant.
template <int KA, int KB, typename T, bool LANES>
__device__ __forceinline__ double2 pair_block(const SpinTables& ta, const SpinTables& tbb, const PairTables& pt, int lo,
                                              int n, int blk, int w, const void* Ba, const void* Bb, const PairK<T>& kk,
                                              const void* ra_in, const void* rb_in, Limbs* bs)
{
    using T2 = cplx_t<T>;
    const T2 *ra = reinterpret_cast<const T2*>(ra_in), *rb = reinterpret_cast<const T2*>(rb_in);
    if constexpr (std::is_same<T, double>::value && LANES) {
        return pair_lanes<KA, KB>(ta, tbb, pt, lo, n, blk, w, reinterpret_cast<const double2*>(Ba),
                                  reinterpret_cast<const double2*>(Bb), kk, ra, rb, bs);
    } else {
        T2 sum = T2{0, 0};   // in the working precision
        for (int it = 0; it < PC_PER_THREAD; ++it) {
            const int i = blk * (PC_THREADS * PC_PER_THREAD) + it * PC_THREADS + threadIdx.x;
            if (i >= n) break;
            const T2 v = pair_term<KA, KB, T>(ta, tbb, pt, lo + i, w, Ba, Bb, kk, ra, rb);
            sum.x += v.x;
            sum.y += v.y;
        }
        return cz((double)sum.x, (double)sum.y);
    }
}

// FP64 mode, levels 1 and 2 (string_energy_lanes: 3 to 6): e_s of string_energy_value
// with the sum over Y in fixed point (scales: Y per walker, exponent ey, and the string's
// largest entry) and, level 2, its one pair of entries in FP64.
template <int KL>
__device__ __forceinline__ double2 string_energy_fixed(const SpinTables& tb, int w, int sl, int ns, const void* Bin,
                                                       const Limbs* as, int ea, const Limbs* ys, int ey)
{
    static_assert(KL <= 2, "one pair of holes and particles at most");
    const int np = tb.np, nh = tb.nh, npp = np * (np - 1) / 2;
    const uint4 rec = tb.str_hp[tb.bucket[KL] + sl];
    const double2* B = reinterpret_cast<const double2*>(Bin) + (size_t)tb.b_off[KL] + ((size_t)w * ns + sl) * b_stride(KL);
    double2 b[KL * KL];
    unsigned m = 0;
#pragma unroll
    for (int e = 0; e < KL * KL; ++e) { b[e] = B[e]; m = max(m, mag_bits(b[e])); }
    const int eb = mag_exponent(m);
    LimbSum lin;
#pragma unroll
    for (int i = 0; i < KL; ++i)
#pragma unroll
        for (int j = 0; j < KL; ++j) lin.add(to_limbs(b[i * KL + j], eb), ys[rec_h(rec, j) * np + rec_p(rec, i)]);
    double2 v = limb_value(lin, eb + ey);
    if constexpr (KL == 2) {
        const int x = pair_index(rec_h(rec, 0), rec_h(rec, 1), nh) * npp + pair_index(rec_p(rec, 0), rec_p(rec, 1), np);
        v = cfma(cfms(b[1], b[2], cfma(b[0], b[3], cz(0, 0))), limbs_fp64(as[x], ea), v);   // fused explicitly, as pair_lanes
    }
    if (max(max(ea, ey), eb) >= FIXED_EXP_INF) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
    return v;
}

// The pair table and Y of a block in shared memory, in FP64 mode as limbs with their
// exponents and with room for the strings' minors (string_energy_lanes).
template <typename T>
struct SeTab {
    const cplx_t<T>*as, *ys;
    int ea, ey;
    Limbs* bs;
};
#define SE_LANES_MIN 3   // levels that string_energy_lanes takes
static_assert(MSD_KMAX <= 8, "a group of 8 lanes holds a string's columns");
__host__ __device__ __forceinline__ constexpr int se_group(int k) { return k <= 4 ? 4 : 8; }
__host__ __device__ __forceinline__ constexpr int se_pitch(int k) { return (k * k) | 1; }
// limbs of a block's strings, the most of any level (se_group 4: level 4, 8: level 6)
#define SE_LIMBS (SE_THREADS / 8 * se_pitch(MSD_KMAX) > SE_THREADS / 4 * se_pitch(4) \
                      ? SE_THREADS / 8 * se_pitch(MSD_KMAX) : SE_THREADS / 4 * se_pitch(4))

// FP64 mode, levels 3 to 6: this block's strings (SE_THREADS SE_PER_THREAD from blk),
// e_s of string_energy_value with its long sums in fixed point (the FP64 unit bounds the
// plain form: level 4, 496 FP64 operations per string; here 48 and 1056 mad.wide):
//   e_s = sum_ij b_ij Y[h_j][p_i] + sum_{i < k-1} sum_j b_ij z_ij,
//   z_ij = sum_{m > i} sum_{l != j} (+ for l > j, - for l < j) b_ml A[h_j,h_l;p_i,p_m].
// Scales: A, Y per walker (exponents ea, ey), b the string's largest entry. A group of 4
// or 8 lanes takes a string, lane j the columns j: b_ij Y[h_j][p_i] and b_ij z_ij for all
// i. The string's limbs are made once, by the group's lanes, in shared memory. A thread
// per string holds them in registers (254 at level 4: 8 warps per SM, every instruction
// waiting for the last) and leaves the SM idle where strings are few (one level-6 string
// in 640 walkers: 0.66 ms). 640 copper-oxo walkers, levels 3 to 6: 2.94 -> 1.42 ms
// (1.31 without the rule below).
//
// The b_ml of z_ij carry 54 bits of the string's largest entry b_ab, and the term is of
// the size of the largest product b_ij b_ml, i != m, j != l: of
//   b_ab max_{m != a, l != b} b_ml   or   max_{m != a} b_mb max_{l != b} b_al,
// far below b_ab^2 where a column or row of b is large by itself (a hole or particle that
// the walker mixes with a small amplitude x: 1 / x). A string whose b_ab^2 is above 2^3
// times that takes z_ij in FP64. Error relative to the term, random minors: FP64 5e-16 to
// 2e-15 (levels 3 to 6), here 2e-16 to 7e-16, of which 0.1 % and less take FP64; at x =
// 1e-8 without the rule 1e-9.
#define SE_SPREAD 3   // bits
template <int KL>
__device__ __forceinline__ double2 string_energy_lanes(const SpinTables& tb, int w, int blk, int ns, const void* Bin,
                                                       const SeTab<double>& tab, const double2* wts)
{
    constexpr int KK = KL * KL, G = se_group(KL), SPW = 32 / G, PITCH = se_pitch(KL), EPL = (KK + G - 1) / G;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane / G, j = lane % G;
    const int np = tb.np, nh = tb.nh, npp = np * (np - 1) / 2;
    const Limbs *as = reinterpret_cast<const Limbs*>(tab.as), *ys = reinterpret_cast<const Limbs*>(tab.ys);
    Limbs* bs = tab.bs + (warp * SPW + g) * PITCH;
    double2 sum = cz(0, 0);
    for (int it = 0; it < SE_PER_THREAD * G; ++it) {
        const int s0 = blk * (SE_THREADS * SE_PER_THREAD) + (it * (SE_THREADS / 32) + warp) * SPW, sl = s0 + g;
        if (s0 >= ns) break;   // the warp's
        const bool on = sl < ns;
        const int sc = on ? sl : ns - 1;
        const double2* B = reinterpret_cast<const double2*>(Bin) + (size_t)tb.b_off[KL] + ((size_t)w * ns + sc) * b_stride(KL);
        const uint4 rec = tb.str_hp[tb.bucket[KL] + sc];
        double2 bv[EPL];
        unsigned mag = 0;
#pragma unroll
        for (int q = 0; q < EPL; ++q) {
            bv[q] = j + q * G < KK ? B[j + q * G] : cz(0, 0);
            mag = max(mag, mag_bits(bv[q]));
        }
#pragma unroll
        for (int o = 1; o < G; o <<= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
        const int eb = mag_exponent(mag);
        // the keys' high bits are log2 to 0.09: a bit is 2^16
        int at = KK, rest = 0, col = 0, row = 0;
#pragma unroll
        for (int q = 0; q < EPL; ++q)
            if (j + q * G < KK && mag_bits(bv[q]) == mag) at = min(at, j + q * G);
#pragma unroll
        for (int o = 1; o < G; o <<= 1) at = min(at, __shfl_xor_sync(0xffffffffu, at, o));
#pragma unroll
        for (int q = 0; q < EPL; ++q) {
            const int e = j + q * G, key = (int)(mag_bits(bv[q]) >> 4);
            if (e >= KK) continue;
            const bool r = e / KL == at / KL, c = e % KL == at % KL;
            if (!r && !c) rest = max(rest, key);
            if (!r && c) col = max(col, key);
            if (r && !c) row = max(row, key);
        }
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
            rest = max(rest, __shfl_xor_sync(0xffffffffu, rest, o));
            col = max(col, __shfl_xor_sync(0xffffffffu, col, o));
            row = max(row, __shfl_xor_sync(0xffffffffu, row, o));
        }
        const int top = (int)(mag >> 4);
        const bool wide = 2 * top - max(top + rest, col + row) > (SE_SPREAD << 16);
        __syncwarp();   // the previous strings' limbs consumed
#pragma unroll
        for (int q = 0; q < EPL; ++q)
            if (j + q * G < KK) bs[j + q * G] = to_limbs(bv[q], eb);
        __syncwarp();
        if (on && j < KL) {
            int hp[KL - 1], lc[KL - 1];   // pair rows of (h_j, h_l) and columns l, j + 1 on, in a circle
            const int hj = rec_h(rec, j);
#pragma unroll
            for (int d = 1; d < KL; ++d) {
                const int l = j + d < KL ? j + d : j + d - KL, hl = rec_h(rec, l);
                lc[d - 1] = l;
                hp[d - 1] = (l > j ? pair_index(hj, hl, nh) : pair_index(hl, hj, nh)) * npp;
            }
            LimbSum lin;
#pragma unroll
            for (int i = 0; i < KL; ++i) lin.add(bs[i * KL + j], ys[hj * np + rec_p(rec, i)]);
            double2 v = limb_value(lin, eb + tab.ey);
            if (wide) {
#pragma unroll 1
                for (int i = 0; i + 1 < KL; ++i) {
                    double2 z = cz(0, 0);
#pragma unroll 1
                    for (int m = i + 1; m < KL; ++m) {
                        const int pim = pair_index(rec_p(rec, i), rec_p(rec, m), np);
#pragma unroll
                        for (int d = 0; d < KL - 1; ++d) {
                            const double2 x = B[m * KL + lc[d]], y = limbs_fp64(as[hp[d] + pim], tab.ea);
                            z = lc[d] > j ? cfma(x, y, z) : cfms(x, y, z);
                        }
                    }
                    v = cfma(B[i * KL + j], z, v);
                }
            }
#pragma unroll 1
            for (int i = 0; i + 1 < KL && !wide; ++i) {
                LimbSum z;
                const int pi = rec_p(rec, i);
#pragma unroll 1
                for (int m = i + 1; m < KL; ++m) {
                    const int pim = pair_index(pi, rec_p(rec, m), np);
#pragma unroll
                    for (int d = 0; d < KL - 1; ++d) {
                        const Limbs x = bs[m * KL + lc[d]], y = as[hp[d] + pim];
                        if (lc[d] > j) z.add(x, y);
                        else z.sub(x, y);
                    }
                }
                v = cfma(B[i * KL + j], limb_value(z, eb + tab.ea), v);
            }
            if (max(max(tab.ea, tab.ey), eb) >= FIXED_EXP_INF) v.x = v.y = __longlong_as_double(0x7ff8000000000000ll);
            sum = cfma(wts[(size_t)w * tb.n_str + tb.bucket[KL] + sl], v, sum);   // wts holds r_s w_s
        }
    }
    return sum;
}

// The same-spin term of one block's strings of one level, this thread's part.
template <int KL, typename T>
__device__ __forceinline__ double2 string_energy_block(const SpinTables& tb, int w, int blk, const void* B,
                                                       const SeTab<T>& tab, const double2* wts)
{
    const int ns = tb.bucket[KL + 1] - tb.bucket[KL];
    double2 sum = cz(0, 0);
    if constexpr (std::is_same<T, double>::value && KL >= SE_LANES_MIN) {
        sum = string_energy_lanes<KL>(tb, w, blk, ns, B, tab, wts);
    } else {
        for (int it = 0; it < SE_PER_THREAD; ++it) {
            const int sl = blk * (SE_THREADS * SE_PER_THREAD) + it * SE_THREADS + threadIdx.x;
            if (sl >= ns) break;
            if constexpr (std::is_same<T, double>::value)
                sum = cfma(wts[(size_t)w * tb.n_str + tb.bucket[KL] + sl],
                           string_energy_fixed<KL>(tb, w, sl, ns, B, reinterpret_cast<const Limbs*>(tab.as), tab.ea,
                                                   reinterpret_cast<const Limbs*>(tab.ys), tab.ey), sum);
            else
                sum = cadd(sum, string_energy_term<KL, T, true>(tb, w, sl, ns, B, tab.as, tab.ys, wts));
        }
    }
    return sum;
}

// The walker's antisymmetrized pair table A[(h,h')][(p,p')] = K[(h,p)][(h',p')] -
// K[(h,p')][(h',p)], h < h', p < p' (not used by level 1), and Y, in shared memory
// for the strings of level k. The block must reach this together.
template <typename T>
__device__ __forceinline__ SeTab<T> load_se_table(const SpinTables& tb, const void* Kin, const void* Yin, int w, int k,
                                                  unsigned char* sm)
{
    using T2 = cplx_t<T>;
    const int X = tb.nh * tb.np, np = tb.np, nh = tb.nh, t = threadIdx.x;
    const int nhp = nh * (nh - 1) / 2, npp = np * (np - 1) / 2, na = k > 1 ? nhp * npp : 0;
    T2* as = reinterpret_cast<T2*>(sm);
    T2* ys = as + nhp * npp;
    const T2* Kw = reinterpret_cast<const T2*>(Kin) + (size_t)w * X * X;
    for (int e = t; e < na; e += blockDim.x) {
        int i = e / npp, c = e - i * npp, h = 0, p = 0;
        while (i >= nh - 1 - h) { i -= nh - 1 - h; ++h; }
        while (c >= np - 1 - p) { c -= np - 1 - p; ++p; }
        const int h2 = h + 1 + i, p2 = p + 1 + c;
        const T2 kc = Kw[(size_t)(h * np + p) * X + h2 * np + p2];
        const T2 kx = Kw[(size_t)(h * np + p2) * X + h2 * np + p];
        as[e] = T2{kc.x - kx.x, kc.y - kx.y};
    }
    const T2* Yw = reinterpret_cast<const T2*>(Yin) + (size_t)w * X;
    for (int e = t; e < X; e += blockDim.x) ys[e] = Yw[e];
    SeTab<T> tab = {as, ys, 0, 0, reinterpret_cast<Limbs*>(ys + X)};
    if constexpr (std::is_same<T, double>::value) {
        // each thread its own entries
        __shared__ unsigned wm[2][SE_THREADS / 32];
        unsigned ma = 0, my = 0;
        for (int e = t; e < na; e += blockDim.x) ma = max(ma, mag_bits(as[e]));
        for (int e = t; e < X; e += blockDim.x) my = max(my, mag_bits(ys[e]));
        tab.ea = mag_exponent(block_mag(ma, wm[0]));
        tab.ey = mag_exponent(block_mag(my, wm[1]));
        Limbs *la = reinterpret_cast<Limbs*>(as), *ly = reinterpret_cast<Limbs*>(ys);
        for (int e = t; e < na; e += blockDim.x) la[e] = to_limbs(as[e], tab.ea);
        for (int e = t; e < X; e += blockDim.x) ly[e] = to_limbs(ys[e], tab.ey);
    }
    __syncthreads();
    return tab;
}

