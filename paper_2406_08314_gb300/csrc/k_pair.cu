// Opposite-spin cross term (fill_os) per determinant with both excitation
// levels (ka, kb) known at compile time, for ka + kb <= 8. Mixed mode: a thread
// per determinant, the indices and both inverse minors in registers, the ka^2 kb^2
// gathers from the shared Gram matrix K^{ab} fully unrolled, so a determinant's
// global loads are all issued before its first gather. FP64 mode: groups of lanes
// (pair_lanes). Same partial-sum slots as k_pair_cross in k_energy.cu, which
// serves the other level pairs.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "det_block.cuh"
#include "kernels.h"

// The block's total, on thread 0: in FP64 mode the lanes of a warp, then the warps in
// order (red: 32), else a tree (red: PC_THREADS).
template <typename T>
__device__ __forceinline__ double2 block_total(double2 v, double2* red)
{
    const int t = threadIdx.x;
    if constexpr (std::is_same<T, double>::value) {
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            v.x += __shfl_down_sync(0xffffffffu, v.x, o);
            v.y += __shfl_down_sync(0xffffffffu, v.y, o);
        }
        if ((t & 31) == 0) red[t >> 5] = v;
        __syncthreads();
        for (int q = 1; t == 0 && q < (int)(blockDim.x >> 5); ++q) v = cadd(v, red[q]);
        return v;
    } else {
        red[t] = v;
        __syncthreads();
        for (int o = PC_THREADS / 2; o; o >>= 1) {
            if (t < o) red[t] = cadd(red[t], red[t + o]);
            __syncthreads();
        }
        return red[0];
    }
}

// Mixed mode: PC_THREADS threads, one per determinant; FP64 mode: groups of lanes,
// any number of warps.
template <int KA, int KB, typename T>
__global__ void __launch_bounds__(std::is_same<T, double>::value ? 1024 : PC_THREADS)
k_pair_cross2(SpinTables ta, SpinTables tbb, PairTables pt, int lo, int n, const void* __restrict__ ra,
              const void* __restrict__ rb, const void* __restrict__ Ba, const void* __restrict__ Bb,
              const void* __restrict__ Kin, double2* __restrict__ part, int nslot, int slot0)
{
    constexpr bool LANES = std::is_same<T, double>::value;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int XX = ta.nh * ta.np * tbb.nh * tbb.np;
    __shared__ double2 red[LANES ? 32 : PC_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    const PairK<T> ks = load_pair_k<T>(Kin, w, XX, smraw);   // [Xa][Xb]
    double2 v = pair_block<KA, KB, T, LANES>(ta, tbb, pt, lo, n, blockIdx.x, w, Ba, Bb, ks, ra, rb,
                                             reinterpret_cast<Limbs*>(smraw) + XX);
    v = block_total<T>(v, red);
    if (t == 0) part[(size_t)w * nslot + slot0 + blockIdx.x] = v;
}

// Shared memory of a block in the lanes form, beside its static part.
static size_t lanes_smem(size_t k_bytes, int limbs) { return k_bytes + sizeof(Limbs) * limbs; }
static bool lanes_fit(size_t dyn, int blocks) { return (dyn + 5 * 1024) * blocks <= 227 * 1024; }
#define PL_THREADS 512   // two blocks per SM

template <int KA, int KB>
static bool go(bool fp32, dim3 grid, size_t smem, const SpinTables& ta, const SpinTables& tb, const PairTables& pt,
               int lo, int n, const void* ra, const void* rb, const void* Ba, const void* Bb, const void* K,
               double2* part, int nslot, int slot, cudaStream_t st)
{
    auto run = [&](auto kern, int threads, size_t sm) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        kern<<<grid, threads, sm, st>>>(ta, tb, pt, lo, n, ra, rb, Ba, Bb, K, part, nslot, slot);
        msd_note_launch();
    };
    if (fp32) {
        run(k_pair_cross2<KA, KB, float>, PC_THREADS, smem);
        return true;
    }
    // 32 warps per SM where they fit: two blocks of 512 threads, one loading its Gram
    // matrix while the other computes, else one of 1024 (75 x 75 active pairs); fewer
    // only beside the largest Gram matrices (112 x 112: 196 KB)
    auto bytes = [&](int threads) { return lanes_smem(smem, pair_limbs(KA, KB, threads)); };
    int threads = lanes_fit(bytes(PL_THREADS), 2) ? PL_THREADS : 1024;
    while (threads > 64 && !lanes_fit(bytes(threads), 1)) threads /= 2;
    run(k_pair_cross2<KA, KB, double>, threads, bytes(threads));
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
// writes slot slot0 + b, the slots and values of the separate launches, which stay
// where the blocks fill the GPU: one kernel for every pair takes the registers of the
// largest. (FP64: where those take PL_THREADS too, so that a walker's value does not
// depend on how many there are.)
struct PairAll {
    SpinTables t[2];
    PairTables pt;
    const void *r[2], *B[2], *K;
    int blk[MSD_KMAX * MSD_KMAX + 1];   // first block of pair (ka - 1) KMAX + kb - 1
};

template <typename T>
__global__ void __launch_bounds__(std::is_same<T, double>::value ? PL_THREADS : PC_THREADS)
k_pair_all(const __grid_constant__ PairAll a, double2* __restrict__ part, int nslot, int slot0)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const int XX = a.t[0].nh * a.t[0].np * a.t[1].nh * a.t[1].np;
    __shared__ double2 red[std::is_same<T, double>::value ? 32 : PC_THREADS];
    const int w = blockIdx.y, t = threadIdx.x;
    const PairK<T> ks = load_pair_k<T>(a.K, w, XX, smraw);   // [Xa][Xb]
    int q = 0;
    while ((int)blockIdx.x >= a.blk[q + 1]) ++q;
    const int blk = (int)blockIdx.x - a.blk[q];
    double2 v = cz(0, 0);
    Limbs* bs = reinterpret_cast<Limbs*>(smraw) + XX;
    switch ((q / MSD_KMAX + 1) * 8 + q % MSD_KMAX + 1) {
#define PAIR_CASE(KA, KB)                                                                                      \
    case KA * 8 + KB: {                                                                                        \
        const int i = KA * (MSD_KMAX + 1) + KB, lo = a.pt.bucket[i];                                           \
        v = pair_block<KA, KB, T, true>(a.t[0], a.t[1], a.pt, lo, a.pt.bucket[i + 1] - lo, blk, w, a.B[0],     \
                                        a.B[1], ks, a.r[0], a.r[1], bs);                                       \
        break;                                                                                                 \
    }
    PAIR_CASE(1, 1) PAIR_CASE(1, 2) PAIR_CASE(1, 3) PAIR_CASE(1, 4) PAIR_CASE(1, 5)
    PAIR_CASE(2, 1) PAIR_CASE(2, 2) PAIR_CASE(2, 3) PAIR_CASE(2, 4)
    PAIR_CASE(3, 1) PAIR_CASE(3, 2) PAIR_CASE(3, 3)
    PAIR_CASE(4, 1) PAIR_CASE(4, 2)
    PAIR_CASE(5, 1)
#undef PAIR_CASE
    }
    v = block_total<T>(v, red);
    if (t == 0) part[(size_t)w * nslot + slot0 + blockIdx.x] = v;
}

bool launch_pair_cross_all(const SpinTables& ta, const SpinTables& tb, const PairTables& pt, int nw, const void* ra,
                           const void* rb, const void* Ba, const void* Bb, const void* K, bool fp32, double2* part,
                           int nslot, int slot0, cudaStream_t st, bool use_runs)
{
    PairAll a;
    int n = 0, used = 0, limbs = 0;
    for (int ka = 1; ka <= MSD_KMAX; ++ka)
        for (int kb = 1; kb <= MSD_KMAX; ++kb) {
            const int idx = ka * (MSD_KMAX + 1) + kb, c = pt.bucket[idx + 1] - pt.bucket[idx];
            a.blk[(ka - 1) * MSD_KMAX + kb - 1] = n;
            if (c <= 0) continue;
            if (ka + kb > 6 || (use_runs && pt.run_side[idx])) return false;
            n += (c + PC_THREADS * PC_PER_THREAD - 1) / (PC_THREADS * PC_PER_THREAD);
            limbs = std::max(limbs, pair_limbs(ka, kb, PL_THREADS));
            ++used;
        }
    a.blk[MSD_KMAX * MSD_KMAX] = n;
    if (used < 2 || (long long)n * nw > ONE_LAUNCH_BLOCKS * msd_sm_count()) return false;
    a.t[0] = ta; a.t[1] = tb; a.pt = pt;
    a.r[0] = ra; a.r[1] = rb; a.B[0] = Ba; a.B[1] = Bb; a.K = K;
    const size_t smem = (fp32 ? sizeof(float2) : sizeof(double2)) * (size_t)(ta.nh * ta.np) * (tb.nh * tb.np) +
                        (fp32 ? 0 : sizeof(Limbs) * limbs);
    if (!fp32 && !lanes_fit(smem, 2)) return false;   // the separate launches take another block size
    if (fp32) {
        cudaFuncSetAttribute(k_pair_all<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_all<float><<<dim3(n, nw), PC_THREADS, smem, st>>>(a, part, nslot, slot0);
    } else {
        cudaFuncSetAttribute(k_pair_all<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_pair_all<double><<<dim3(n, nw), PL_THREADS, smem, st>>>(a, part, nslot, slot0);
    }
    msd_note_launch();
    return true;
}
