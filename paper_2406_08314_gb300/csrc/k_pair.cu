// Opposite-spin cross term (fill_os) per determinant with both excitation
// levels (ka, kb) known at compile time, for ka + kb <= 8: the indices and
// both inverse minors sit in registers and the ka^2 kb^2 gathers from the
// shared Gram matrix K^{ab} are fully unrolled, so a determinant's global
// loads are all issued before its first gather. Same value, partial-sum
// slots and block shape as k_pair_cross in k_energy.cu, which serves the
// other level pairs.
#include <type_traits>

#include "common.cuh"
#include "det_block.cuh"
#include "kernels.h"

template <int KA, int KB, typename T>
__global__ void __launch_bounds__(PC_THREADS, std::is_same<T, double>::value ? 2 : 1)
k_pair_cross2(SpinTables ta, SpinTables tbb, PairTables pt, int lo, int n, const void* __restrict__ ra_in,
              const void* __restrict__ rb_in, const void* __restrict__ Ba_in, const void* __restrict__ Bb_in,
              const void* __restrict__ Kin, double2* __restrict__ part, int nslot, int slot0)
{
    using T2 = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int Xa = ta.nh * ta.np, Xb = tbb.nh * tbb.np;
    __shared__ double2 red[PC_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    const PairK<T> ks = load_pair_k<T>(Kin, w, Xa * Xb, smraw);   // [Xa][Xb]
    const T2* ra = reinterpret_cast<const T2*>(ra_in);
    const T2* rb = reinterpret_cast<const T2*>(rb_in);
    T2 contrib = T2{0, 0};   // this thread's determinants, in the working precision
    for (int it = 0; it < PC_PER_THREAD; ++it) {
        const int i0 = blockIdx.x * (PC_THREADS * PC_PER_THREAD) + it * PC_THREADS + t;
        if (i0 >= n) break;
        const T2 v = pair_term<KA, KB, T>(ta, tbb, pt, lo + i0, w, Ba_in, Bb_in, ks, ra, rb);
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

template <int KA, int KB>
static bool go(bool fp32, dim3 grid, size_t smem, const SpinTables& ta, const SpinTables& tb, const PairTables& pt,
               int lo, int n, const void* ra, const void* rb, const void* Ba, const void* Bb, const void* K,
               double2* part, int nslot, int slot, cudaStream_t st)
{
    if (fp32) {
        cudaFuncSetAttribute(k_pair_cross2<KA, KB, float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_cross2<KA, KB, float><<<grid, PC_THREADS, smem, st>>>(ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part,
                                                                     nslot, slot);
    } else {
        cudaFuncSetAttribute(k_pair_cross2<KA, KB, double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_cross2<KA, KB, double><<<grid, PC_THREADS, smem, st>>>(ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part,
                                                                      nslot, slot);
    }
    msd_note_launch();
    return true;
}

bool launch_pair_cross2(int ka, int kb, bool fp32, dim3 grid, size_t smem, const SpinTables& ta, const SpinTables& tb,
                        const PairTables& pt, int lo, int n, const void* ra, const void* rb, const void* Ba,
                        const void* Bb, const void* K, double2* part, int nslot, int slot, cudaStream_t st)
{
    switch (ka * 8 + kb) {
        case 9: return go<1, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 10: return go<1, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 11: return go<1, 3>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 12: return go<1, 4>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 13: return go<1, 5>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 14: return go<1, 6>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 17: return go<2, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 18: return go<2, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 19: return go<2, 3>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 20: return go<2, 4>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 21: return go<2, 5>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 22: return go<2, 6>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 25: return go<3, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 26: return go<3, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 27: return go<3, 3>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 28: return go<3, 4>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 29: return go<3, 5>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 33: return go<4, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 34: return go<4, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 35: return go<4, 3>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 36: return go<4, 4>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 41: return go<5, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 42: return go<5, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 43: return go<5, 3>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 49: return go<6, 1>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        case 50: return go<6, 2>(fp32, grid, smem, ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot, st);
        default: return false;
    }
}

// All level pairs in one launch, for calls whose blocks are few: a launch per
// pair was most of this term's time there (7 us each, up to 15 of them). Block b
// writes slot slot0 + b, the slots and values of the separate launches, which
// stay where the blocks fill the GPU: one kernel for every pair takes the
// registers of the largest.
struct PairAll {
    SpinTables t[2];
    PairTables pt;
    const void *r[2], *B[2], *K;
    int blk[MSD_KMAX * MSD_KMAX + 1];   // first block of pair (ka - 1) KMAX + kb - 1
};

template <int KA, int KB, typename T>
__device__ __forceinline__ cplx_t<T> pair_block(const PairAll& a, int w, int blk, const PairK<T>& ks)
{
    using T2 = cplx_t<T>;
    const int idx = KA * (MSD_KMAX + 1) + KB, lo = a.pt.bucket[idx], n = a.pt.bucket[idx + 1] - lo;
    T2 contrib = T2{0, 0};
    for (int it = 0; it < PC_PER_THREAD; ++it) {
        const int i0 = blk * (PC_THREADS * PC_PER_THREAD) + it * PC_THREADS + threadIdx.x;
        if (i0 >= n) break;
        const T2 v = pair_term<KA, KB, T>(a.t[0], a.t[1], a.pt, lo + i0, w, a.B[0], a.B[1], ks,
                                          reinterpret_cast<const T2*>(a.r[0]), reinterpret_cast<const T2*>(a.r[1]));
        contrib.x += v.x;
        contrib.y += v.y;
    }
    return contrib;
}

template <typename T>
__global__ void __launch_bounds__(PC_THREADS)
k_pair_all(const __grid_constant__ PairAll a, double2* __restrict__ part, int nslot, int slot0)
{
    using T2 = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int XX = a.t[0].nh * a.t[0].np * a.t[1].nh * a.t[1].np;
    __shared__ double2 red[PC_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    const PairK<T> ks = load_pair_k<T>(a.K, w, XX, smraw);   // [Xa][Xb]
    int q = 0;
    while ((int)blockIdx.x >= a.blk[q + 1]) ++q;
    const int blk = (int)blockIdx.x - a.blk[q];
    T2 v = T2{0, 0};
    switch ((q / MSD_KMAX + 1) * 8 + q % MSD_KMAX + 1) {
#define PAIR_CASE(A, B) case A * 8 + B: v = pair_block<A, B, T>(a, w, blk, ks); break;
    PAIR_CASE(1, 1) PAIR_CASE(1, 2) PAIR_CASE(1, 3) PAIR_CASE(1, 4) PAIR_CASE(1, 5)
    PAIR_CASE(2, 1) PAIR_CASE(2, 2) PAIR_CASE(2, 3) PAIR_CASE(2, 4)
    PAIR_CASE(3, 1) PAIR_CASE(3, 2) PAIR_CASE(3, 3)
    PAIR_CASE(4, 1) PAIR_CASE(4, 2)
    PAIR_CASE(5, 1)
#undef PAIR_CASE
    }
    red[t] = cz((double)v.x, (double)v.y);
    __syncthreads();
    for (int o = PC_THREADS / 2; o; o >>= 1) {
        if (t < o) red[t] = cadd(red[t], red[t + o]);
        __syncthreads();
    }
    if (t == 0) part[(size_t)w * nslot + slot0 + blockIdx.x] = red[0];
}

bool launch_pair_cross_all(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int nw, const void* ra,
                           const void* rb, const void* Ba, const void* Bb, const void* K, bool fp32, double2* part,
                           int nslot, int slot0, cudaStream_t st, bool use_runs)
{
    PairAll a;
    int n = 0, used = 0;
    for (int ka = 1; ka <= MSD_KMAX; ++ka)
        for (int kb = 1; kb <= MSD_KMAX; ++kb) {
            const int idx = ka * (MSD_KMAX + 1) + kb, c = pt.bucket[idx + 1] - pt.bucket[idx];
            a.blk[(ka - 1) * MSD_KMAX + kb - 1] = n;
            if (c <= 0) continue;
            if (ka + kb > 6 || (use_runs && pt.run_side[idx])) return false;
            n += (c + PC_THREADS * PC_PER_THREAD - 1) / (PC_THREADS * PC_PER_THREAD);
            ++used;
        }
    a.blk[MSD_KMAX * MSD_KMAX] = n;
    if (used < 2 || (long long)n * nw > ONE_LAUNCH_BLOCKS * msd_sm_count()) return false;
    a.t[0] = ta; a.t[1] = tb; a.pt = pt;
    a.r[0] = ra; a.r[1] = rb; a.B[0] = Ba; a.B[1] = Bb; a.K = K;
    const size_t smem = (fp32 ? sizeof(float2) : sizeof(double2)) * (size_t)(ta.nh * ta.np) * (tb.nh * tb.np);
    if (fp32) {
        cudaFuncSetAttribute(k_pair_all<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_all<float><<<dim3(n, nw), PC_THREADS, smem, st>>>(a, part, nslot, slot0);
    } else {
        cudaFuncSetAttribute(k_pair_all<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_all<double><<<dim3(n, nw), PC_THREADS, smem, st>>>(a, part, nslot, slot0);
    }
    msd_note_launch();
    return true;
}
