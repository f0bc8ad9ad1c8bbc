// Persistent batched kernel for the per-determinant energy terms of many
// independent systems (uneven orbital counts, determinant counts and
// excitation levels) in one launch. Work items are (system, walker, kind,
// spin or opposite-spin level pair, block of strings or determinants); a
// resident grid of CTAs takes items from a global counter (atomicAdd, no
// waiting), so small and large systems share the machine. Each item covers the
// strings or determinants of one block of k_string_energy / k_pair_cross and
// writes the same partial-sum slot. In mixed mode it computes what that block
// computes. In FP64 mode the opposite-spin term has other forms here (a thread per
// determinant in fixed point up to ka + kb = 6, the general FP64 form above; the
// per-system kernels give a determinant a group of lanes up to 8) and sums in
// another order: batched and per-system energies agree to rounding.
#include "common.cuh"
#include "det_block.cuh"
#include "kernels.h"

// The opposite-spin term of one block whose levels add up to more than 6, in the
// general form.
template <int KB, typename T>
__device__ double2 batch_pc_any(const BatchSys& S, const BatchItem& it, const cplx_t<T>* ks)
{
    using T2 = cplx_t<T>;
    const int idx = it.ka * (MSD_KMAX + 1) + KB, lo = S.pt.bucket[idx], n = S.pt.bucket[idx + 1] - lo;
    constexpr bool F = std::is_same<T, float>::value;
    const T2* ra = F ? reinterpret_cast<const T2*>(S.rf[0]) : reinterpret_cast<const T2*>(S.r[0]);
    const T2* rb = F ? reinterpret_cast<const T2*>(S.rf[1]) : reinterpret_cast<const T2*>(S.r[1]);
    T2 acc = T2{0, 0};
    for (int q = 0; q < PC_PER_THREAD; ++q) {
        const int i0 = it.blk * (PC_THREADS * PC_PER_THREAD) + q * PC_THREADS + threadIdx.x;
        if (i0 >= n) break;
        const T2 v = pair_cross_term<KB, T>(S.t[0], S.t[1], S.pt, it.ka, lo + i0, it.w, S.B[0], S.B[1], ks, ra, rb);
        acc.x += v.x;
        acc.y += v.y;
    }
    return cz((double)acc.x, (double)acc.y);
}

template <typename T>
// (the fixed-point sums of the FP64 mode take the registers of a whole SM)
__global__ void __launch_bounds__(256, sizeof(T) == 8 ? 1 : 2)
k_det_batched(const BatchSys* __restrict__ systems, const BatchItem* __restrict__ items, int n_items,
              unsigned* __restrict__ counter)
{
    static_assert(SE_THREADS == 256 && PC_THREADS == 256, "one block shape for both item kinds");
    using T2 = cplx_t<T>;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ BatchItem it;
    __shared__ int cur;
    __shared__ double2 red[256];
    __shared__ __align__(16) unsigned char sys_raw[sizeof(BatchSys)];
    const BatchSys& S = *reinterpret_cast<const BatchSys*>(sys_raw);
    const int t = threadIdx.x;
    int loaded = -1;
    while (true) {
        if (t == 0) {
            cur = (int)atomicAdd(counter, 1u);
            if (cur < n_items) it = items[cur];
        }
        __syncthreads();
        if (cur >= n_items) break;
        if (it.sys != loaded) {   // uniform: every thread sees the same item
            const int* src = reinterpret_cast<const int*>(systems + it.sys);
            int* dst = reinterpret_cast<int*>(sys_raw);
            for (int e = t; e < (int)(sizeof(BatchSys) / sizeof(int)); e += blockDim.x) dst[e] = src[e];
            loaded = it.sys;
            __syncthreads();
        }
        double2 v = cz(0, 0);
        if (it.kind == 0) {
            const SeTab<T> tab = load_se_table<T>(S.t[it.spin], S.K[it.spin], S.Y[it.spin], it.w, it.ka, smraw);
            const int s = it.spin;
            switch (it.ka) {
#define BATCH_SE(K) string_energy_block<K, T>(S.t[s], it.w, it.blk, S.B[s], tab, S.wts[s])
            case 1: v = BATCH_SE(1); break;
            case 2: v = BATCH_SE(2); break;
            case 3: v = BATCH_SE(3); break;
            case 4: v = BATCH_SE(4); break;
            case 5: v = BATCH_SE(5); break;
            default: v = BATCH_SE(6); break;
#undef BATCH_SE
            }
        } else {
            const int XX = S.t[0].nh * S.t[0].np * S.t[1].nh * S.t[1].np;
            if (it.ka + it.kb <= 6) {
                const PairK<T> ks = load_pair_k<T>(S.K[2], it.w, XX, smraw);
                // the ratios in the working precision, as in the per-system kernels
                constexpr bool F = std::is_same<T, float>::value;
                const void *ra = F ? (const void*)S.rf[0] : S.r[0], *rb = F ? (const void*)S.rf[1] : S.r[1];
                const int i = it.ka * (MSD_KMAX + 1) + it.kb, lo = S.pt.bucket[i], n = S.pt.bucket[i + 1] - lo;
                switch (it.ka * 8 + it.kb) {
#define PAIR_CASE(KA, KB)                                                                                         \
    case KA * 8 + KB:                                                                                             \
        v = pair_block<KA, KB, T, false>(S.t[0], S.t[1], S.pt, lo, n, it.blk, it.w, S.B[0], S.B[1], ks, ra, rb, nullptr); \
        break;
                PAIR_CASE(1, 1) PAIR_CASE(1, 2) PAIR_CASE(1, 3) PAIR_CASE(1, 4) PAIR_CASE(1, 5)
                PAIR_CASE(2, 1) PAIR_CASE(2, 2) PAIR_CASE(2, 3) PAIR_CASE(2, 4)
                PAIR_CASE(3, 1) PAIR_CASE(3, 2) PAIR_CASE(3, 3)
                PAIR_CASE(4, 1) PAIR_CASE(4, 2)
                PAIR_CASE(5, 1)
#undef PAIR_CASE
                }
            } else {
                const T2* K = reinterpret_cast<const T2*>(S.K[2]) + (size_t)it.w * XX;
                T2* ks = reinterpret_cast<T2*>(smraw);
                for (int e = t; e < XX; e += blockDim.x) ks[e] = K[e];
                __syncthreads();
                switch (it.kb) {
                case 1: v = batch_pc_any<1, T>(S, it, ks); break;
                case 2: v = batch_pc_any<2, T>(S, it, ks); break;
                case 3: v = batch_pc_any<3, T>(S, it, ks); break;
                case 4: v = batch_pc_any<4, T>(S, it, ks); break;
                case 5: v = batch_pc_any<5, T>(S, it, ks); break;
                default: v = batch_pc_any<6, T>(S, it, ks); break;
                }
            }
        }
        red[t] = v;
        __syncthreads();
        for (int o = 128; o; o >>= 1) {
            if (t < o) red[t] = cadd(red[t], red[t + o]);
            __syncthreads();
        }
        if (t == 0) S.part[(size_t)it.w * S.nslot + it.slot] = red[0];
        __syncthreads();
    }
}

int launch_det_batched(const BatchSys* systems, const BatchItem* items, int n_items, unsigned* counter,
                       size_t smem, bool fp32, int grid, cudaStream_t st)
{
    if (n_items <= 0) return 0;
    if (cudaMemsetAsync(counter, 0, sizeof(unsigned), st) != cudaSuccess) return -1;
    if (fp32) {
        cudaFuncSetAttribute(k_det_batched<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_det_batched<float><<<grid, 256, smem, st>>>(systems, items, n_items, counter);
    } else {
        cudaFuncSetAttribute(k_det_batched<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        k_det_batched<double><<<grid, 256, smem, st>>>(systems, items, n_items, counter);
    }
    msd_note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}
