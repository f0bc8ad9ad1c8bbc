// FP64 products on the BF16 tensor cores, to FP64 accuracy, for the dense
// contractions of the FP64 path: C[n][m] = sum_k A[m][k] B[n][k] with real A
// rows and complex B rows (stored as two real rows 2n, 2n + 1).
//
// GB300 issues two FP64 FMAs per clock and SM (1.1 TFLOP/s measured) against
// 1.9 PFLOP/s in BF16, so an FP64 product is evaluated here by an exact-integer
// split (Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012)): every row
// is scaled by a power of two to |x| < 1 and rounded to 56 fractional bits, cut
// into DG_S = 8 balanced digits of 7 bits (|a_1| <= 128, |a_i| <= 64, exact in
// BF16). The digit products with i + j = c share one FP32 accumulator in TMEM;
// c = 2..9 are kept (36 products per 16-element K step). Over a chunk of 384
// contraction steps every accumulator stays an integer below 2^24
// (2 * 128 * 64 + 6 * 64 * 64 = 40960 per step at c = 9), so the tensor cores
// add exactly; after a chunk the epilogue takes the eight accumulators into two
// 64-bit integers, and rounds once to FP64 at the end.
//
// Error: the operands' rounding (2^-57 of the row maximum) and the dropped
// products c >= 10 (below 2^-63 K^1/2 of the two row maxima): small against the
// rounding of an FP64 FMA chain (about 2^-53 (K / 8)^1/2 of the result) where the
// row maxima meet, less accurate than it where a row's largest entries meet only
// small ones, by their ratio. Rows whose entries differ by scales of their own are
// for the caller to scale: the reference product does (k_ref).
//
// Tile 128 x 64: eight accumulators of 64 columns are the whole TMEM (512
// columns). An MMA of N = 64 reads 6 KB of shared memory for 32 tensor clocks,
// so the tensor pipe runs at about two thirds of its peak; a wider tile has no
// room for its accumulators.
//
// Structure (persistent, one CTA per SM, 10 warps):
//   warp 0    TMA producer: k-blocks of 32 BF16 (64-byte swizzle) of all
//             slices of A and B into a two-stage ring (96 KB a stage);
//   warp 1    TMEM owner; one elected lane issues the MMAs;
//   warps 2-9 epilogue: lane quarter (warp % 4), column half; each drains the
//             accumulators in the order c = 2..9 and releases every one as soon
//             as it is read, so the next tile's products start while this
//             tile's results are converted and stored.
// Every wait is bounded; on expiry the kernel records MSD_DEV_ERR_TIMEOUT,
// every role leaves its loop, issued copies and products are drained and TMEM
// is freed.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "common.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

using namespace tcx;

namespace {

constexpr int DG_S = 8;                  // digits per operand
constexpr int DG_BETA = 7;               // bits per digit
constexpr int DG_BM = 128, DG_BN = 64;   // output tile (rows of A x real rows of B)
constexpr int DG_BK = 32;                // BF16 elements per k-block (64 bytes)
constexpr int DG_CHUNK = 12;             // k-blocks per exact chunk (384 contraction steps)
constexpr int DG_STAGES = 2;
constexpr int DG_THREADS = 320;
constexpr int DG_HALF = DG_BN / 2;       // columns per epilogue warp
constexpr uint32_t DG_A_SL = DG_BM * 64, DG_B_SL = DG_BN * 64;
constexpr uint32_t DG_STAGE = DG_S * (DG_A_SL + DG_B_SL);
constexpr size_t DG_SMEM = (size_t)DG_STAGES * DG_STAGE + 1024;
constexpr int DG_GROUP = 16;             // row tiles that share a pass over the column tiles
constexpr int DG_NAN = 1 << 24;          // exponent of a row with an infinity or a NaN
static_assert(DG_S * DG_BN == 512, "the accumulators take the whole TMEM");
static_assert((long long)DG_CHUNK * DG_BK * (2 * 128 * 64 + (DG_S - 2) * 64 * 64) < (1ll << 24),
              "a chunk's sums are exact in FP32");

struct DgArgs {
    int Mr, Nc;              // rows of A, complex rows of B (per batch entry)
    int a_rows, b_rows;      // rows of one slice of A and of B (all batch entries)
    int a_batch, b_batch;    // rows between batch entries (0: shared)
    int nkb, splits;         // k-blocks; contraction splits
    int mt, nt, batch;       // row tiles, column tiles, batch entries
    const int* ea;           // [a_rows] exponents
    const int* eb;           // [b_rows]
    double2* C;              // C[z c_batch + n c_n + m c_m], z = batch entry or split
    long long c_batch, c_n, c_m;
    double2* acc;            // optional, same layout: acc = acc_in + C
    const double2* acc_in;
    double mul;              // C = mul (A B)
    // Gram form (gx >= 0): rows and columns stack gx alpha and gy beta entries;
    // the (alpha, alpha), (alpha, beta) and (beta, beta) blocks go to K[0..2]
    int gx, gy;
    double2* K[3];
    const int* eye;          // [Mr] or NULL: rows with eye[m] >= 0 are unit vectors
    const double2* live;     // [batch] with eye: entries z with live[z] = 0 are zero
    unsigned* err;
};

// hi 2^-35 + lo 2^-63 (the accumulators c = 2..5 and 6..9) times 2^e.
__device__ __forceinline__ double dg_value(long long hi, long long lo, int e)
{
    if (e >= DG_NAN / 2) return __longlong_as_double(0x7ff8000000000000ll);
    if (hi < (1ll << 38) && hi > -(1ll << 38))   // |value| < 8: one 64-bit integer of 2^-59
        return int_to_fp64((hi << 24) + ((lo + 8) >> 4), e - 59);
    return int_to_fp64_slow(hi, lo, e - 63);
}

struct DgTile { int m0, n0, z; };

__device__ __forceinline__ DgTile dg_tile(const DgArgs& a, int t)
{
    // row tiles in groups of DG_GROUP: a group's operand rows stay in L2 while
    // the column tiles pass
    const int per = a.mt * a.nt, z = t / per;
    int r = t - z * per;
    const int full = DG_GROUP * a.nt, g = r / full;
    r -= g * full;
    const int gm = min(DG_GROUP, a.mt - g * DG_GROUP);
    return {(g * DG_GROUP + r % gm) * DG_BM, (r / gm) * DG_BN, z};
}

// Tiles of the Gram form that hold only the (beta, alpha) block, which nobody
// reads.
__device__ __forceinline__ bool dg_skip(const DgArgs& a, const DgTile& t)
{
    return a.gx >= 0 && t.m0 >= a.gx && t.n0 + DG_BN <= 2 * a.gx;
}

__global__ void __launch_bounds__(DG_THREADS, 1)
k_tc_dgemm(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
           const __grid_constant__ DgArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[DG_STAGES], empty_bar[DG_STAGES];
    __shared__ __align__(8) uint64_t tfull, tempty[DG_S], drain_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntile = a.mt * a.nt * a.batch * a.splits;
    const uint64_t wb = wait_budget(a.err);

    if (threadIdx.x == 0) {
        for (int s = 0; s < DG_STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&tfull, 1);
        for (int c = 0; c < DG_S; ++c) mbar_init(&tempty[c], 8);
        mbar_init(&drain_bar, 1);
        fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(su32(&tmem_base_sh)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;
    volatile int* vfail = &fail;
    // k-blocks of a tile: all, or the split's share (z is then the split)
    auto kbeg = [&](int z) { return a.splits > 1 ? (int)((long long)a.nkb * z / a.splits) : 0; };
    auto kend = [&](int z) { return a.splits > 1 ? (int)((long long)a.nkb * (z + 1) / a.splits) : a.nkb; };

    if (warp == 0) {
        if (lane == 0) {
            // ---------------------------------------------------- TMA producer
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < ntile && ok; t += gridDim.x) {
                const DgTile q = dg_tile(a, t);
                if (dg_skip(a, q)) continue;
                const int bz = a.splits > 1 ? 0 : q.z, ke = kend(q.z);
                const int ra = bz * a.a_batch + q.m0, rb = bz * a.b_batch + q.n0;
                for (int kb = kbeg(q.z); kb < ke; ++kb, ++it) {
                    const int s = it % DG_STAGES;
                    if (!mbar_wait(&empty_bar[s], ((it / DG_STAGES) & 1) ^ 1, wb) || *vfail) { ok = false; break; }
                    uint8_t* st = smem + (size_t)s * DG_STAGE;
                    mbar_expect_tx(&full_bar[s], DG_STAGE);
#pragma unroll
                    for (int i = 0; i < DG_S; ++i) {
                        tma_load_2d(st + i * DG_A_SL, &ta, &full_bar[s], kb * DG_BK, i * a.a_rows + ra);
                        tma_load_2d(st + DG_S * DG_A_SL + i * DG_B_SL, &tb, &full_bar[s], kb * DG_BK, i * a.b_rows + rb);
                    }
                }
            }
            if (!ok) { *vfail = 1; atomicOr(a.err, MSD_DEV_ERR_TIMEOUT); }
            // the copies issued last must land before the CTA may exit
            for (int k = it - DG_STAGES < 0 ? 0 : it - DG_STAGES; k < it; ++k)
                mbar_drain(&full_bar[k % DG_STAGES], (k / DG_STAGES) & 1);
        }
    } else if (warp == 1) {
        // -------------------------------------------------------- MMA issuer
        // The whole warp runs the loop and one elected thread issues: the
        // descriptors stay in uniform registers (computed by a single diverged
        // lane, an MMA of 32 tensor clocks took 90 to issue).
        constexpr uint32_t idesc = idesc_bf16(DG_BM, DG_BN);
        const bool leader = elect_one();
        const uint64_t desc0 = sw64_desc(su32(smem));
        bool ok = true;
        int it = 0, unit = 0;   // unit: one chunk of one tile, one use of the accumulators
        for (int t = blockIdx.x; t < ntile && ok; t += gridDim.x) {
            const DgTile tl = dg_tile(a, t);
            if (dg_skip(a, tl)) continue;
            const int z = tl.z, k1 = kend(z);
            for (int c0 = kbeg(z); c0 < k1 && ok; c0 += DG_CHUNK, ++unit) {
                const int c1 = min(k1, c0 + DG_CHUNK);
                for (int kb = c0; kb < c1; ++kb, ++it) {
                    const int s = it % DG_STAGES;
                    const bool got = mbar_wait(&full_bar[s], (it / DG_STAGES) & 1, wb) && !*vfail;
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t dA = desc0 + (uint64_t)((uint32_t)s * DG_STAGE >> 4);
                    const uint64_t dB = dA + (uint64_t)(DG_S * DG_A_SL >> 4);
#pragma unroll
                    for (int kk = 0; kk < 2; ++kk) {   // 2 x 16 BF16 of K per k-block
                        if (kb == c0 && kk == 0) {
                            // first use of the accumulators: as the epilogue
                            // releases them, c ascending
#pragma unroll
                            for (int c = 0; c < DG_S; ++c) {   // accumulator c: i + j = c (digits from 0)
                                if (unit > 0) {
                                    const bool free_ = mbar_wait(&tempty[c], (unit - 1) & 1, wb);
                                    ok = __all_sync(0xffffffffu, free_) && ok;
                                    tc_fence_after();
                                }
                                if (ok && leader) {
#pragma unroll
                                    for (int i = 0; i <= c; ++i)
                                        mma_bf16(tmem + (uint32_t)(c * DG_BN), dA + (uint64_t)(i * (DG_A_SL >> 4)),
                                                 dB + (uint64_t)((c - i) * (DG_B_SL >> 4)), idesc, i == 0 ? 0u : 1u);
                                }
                            }
                        } else if (ok && leader) {
                            // consecutive products go to different accumulators
#pragma unroll
                            for (int i = 0; i < DG_S; ++i)
#pragma unroll
                                for (int c = DG_S - 1; c >= i; --c)
                                    mma_bf16(tmem + (uint32_t)(c * DG_BN), dA + (uint64_t)(i * (DG_A_SL >> 4) + kk * 2),
                                             dB + (uint64_t)((c - i) * (DG_B_SL >> 4) + kk * 2), idesc, 1u);
                        }
                    }
                    __syncwarp();
                    if (!ok) break;
                    if (leader) mma_commit(&empty_bar[s]);
                }
                if (!ok) break;
                if (leader) mma_commit(&tfull);
            }
        }
        if (leader) {
            if (!ok) { *vfail = 1; atomicOr(a.err, MSD_DEV_ERR_TIMEOUT); }
            // every product issued by this thread completes before TMEM is freed
            mma_commit(&drain_bar);
            mbar_drain(&drain_bar, 0);
        }
        __syncwarp();
    } else {
        // -------------------------------------------------------- epilogue
        const int q = warp & 3, hf = (warp - 2) >> 2;
        const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * DG_HALF);
        bool ok = true;
        int unit = 0;
        for (int t = blockIdx.x; t < ntile && ok; t += gridDim.x) {
            const DgTile tl = dg_tile(a, t);
            if (dg_skip(a, tl)) continue;
            long long hi[DG_HALF], lo[DG_HALF];
#pragma unroll
            for (int i = 0; i < DG_HALF; ++i) hi[i] = lo[i] = 0;
            const int k1 = kend(tl.z);
            for (int c0 = kbeg(tl.z); c0 < k1; c0 += DG_CHUNK, ++unit) {
                const bool got = mbar_wait(&tfull, unit & 1, wb) && !*vfail;
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
#pragma unroll
                for (int c = 0; c < DG_S; ++c) {
#pragma unroll
                    for (int h = 0; h < DG_HALF; h += 16) {
                        uint32_t r[16];
                        tmem_ld16_nowait(tbase + (uint32_t)(c * DG_BN + h), r);
                        tmem_wait_ld();
                        if (h + 16 == DG_HALF) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&tempty[c]);
                        }
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const int v = __float2int_rn(__uint_as_float(r[i]));
                            if (c < 4) hi[h + i] += (long long)v * (1 << (DG_BETA * (3 - c)));
                            else lo[h + i] += (long long)v * (1 << (DG_BETA * (7 - c)));
                        }
                    }
                }
            }
            if (!ok) break;
            const int m = tl.m0 + q * 32 + lane;
            if (m < a.Mr) {
                const int bz = a.splits > 1 ? 0 : tl.z;
                const int ea = a.ea[bz * a.a_batch + m];
                const int* ebp = a.eb + (size_t)bz * a.b_batch;
                const int unit_n = a.eye ? a.eye[m] : -1;
                const bool dead = a.eye && a.live[tl.z].x == 0.0 && a.live[tl.z].y == 0.0;
                const long long o0 = (long long)tl.z * a.c_batch + (long long)m * a.c_m;
#pragma unroll
                for (int i = 0; i < DG_HALF; i += 2) {
                    const int n2 = tl.n0 + hf * DG_HALF + i, n = n2 >> 1;
                    if (n < a.Nc) {
                        double2 v = make_double2(dg_value(hi[i], lo[i], ea + ebp[n2]),
                                                 dg_value(hi[i + 1], lo[i + 1], ea + ebp[n2 + 1]));
                        if (a.mul != 1.0) v = make_double2(v.x * a.mul, v.y * a.mul);
                        if (unit_n >= 0) v = make_double2(n == unit_n ? 1.0 : 0.0, 0.0);
                        if (dead) v = make_double2(0.0, 0.0);
                        if (a.gx >= 0) {
                            const int X = a.gx, Y = a.gy;
                            if (n >= X) {
                                if (m < X) a.K[1][((size_t)tl.z * X + m) * Y + n - X] = v;
                                else a.K[2][((size_t)tl.z * Y + m - X) * Y + n - X] = v;
                            } else if (m < X) {
                                a.K[0][((size_t)tl.z * X + m) * X + n] = v;
                            }
                            continue;
                        }
                        const long long o = o0 + (long long)n * a.c_n;
                        a.C[o] = v;
                        if (a.acc) {
                            const double2 p = a.acc_in[o];
                            a.acc[o] = make_double2(p.x + v.x, p.y + v.y);
                        }
                    }
                }
            }
        }
        if (!ok && lane == 0) { *vfail = 1; atomicOr(a.err, MSD_DEV_ERR_TIMEOUT); }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------- slicing
// Exponent e of a row with largest magnitude bits `top` (the sign-free high
// word of an FP64 value): every |x| < 2^e, -1021 for subnormal rows.
__device__ __forceinline__ int dg_exponent(unsigned top)
{
    const int f = (int)(top >> 20);
    return f == 0x7ff ? DG_NAN : max(f, 1) - 1022;
}

// The eight digits of eight fixed-point values as BF16: u[i] packs digit i (most
// significant first) of the eight.
__device__ __forceinline__ void dg_digits8(long long* q, uint4* u)
{
#pragma unroll
    for (int i = DG_S - 1; i >= 0; --i) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t h[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int v = 2 * j + k;
                int d;
                if (i > 0) {
                    d = (((int)q[v] & 127) ^ 64) - 64;
                    q[v] = (q[v] - d) >> DG_BETA;
                } else {
                    d = (int)q[v];
                }
                // d as a float through the integer part of 1.5 2^23 + d
                h[k] = __float_as_uint(__uint_as_float(0x4b400000u + (uint32_t)d) - 12582912.f);
            }
            w[j] = __byte_perm(h[0], h[1], 0x7632);
        }
        u[i] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ... stored at out[i * stride].
__device__ __forceinline__ void dg_store8(long long* q, __nv_bfloat16* out, size_t stride)
{
    uint4 u[DG_S];
    dg_digits8(q, u);
#pragma unroll
    for (int i = 0; i < DG_S; ++i) *reinterpret_cast<uint4*>(out + (size_t)i * stride) = u[i];
}

__device__ __forceinline__ unsigned dg_mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// Rows of a row-major matrix: src[r ld + k], real, or the two parts of a complex
// row as rows 2r, 2r + 1. LR lanes per row, each 8 consecutive elements of the
// row at a time (one 16-byte store per digit). SCALED: elements 2 k, 2 k + 1 of a real
// row times scale[r / rows][k].
template <bool CPLX, int LR, bool SCALED>
__global__ void __launch_bounds__(256)
k_dg_rows(long long R, int K, int Kp, const double* __restrict__ src, long long ld, __nv_bfloat16* __restrict__ S,
          int* __restrict__ ex, size_t stride, const double* __restrict__ scale, int rows)
{
    const long long r = ((long long)blockIdx.x * 256 + threadIdx.x) / LR;
    const int lane = threadIdx.x % LR;
    const bool live = r < R;
    const double* p = src + (CPLX ? 2 : 1) * (live ? r : 0) * ld;
    const double* sc = SCALED ? scale + (live ? r / rows : 0) * (K / 2) : nullptr;
    auto at = [&](int k) { return SCALED ? p[k] * sc[k >> 1] : p[k]; };
    unsigned t0 = 0, t1 = 0;
    if (live) {
        if (CPLX) {
            const double2* p2 = reinterpret_cast<const double2*>(p);
            for (int k = lane; k < K; k += LR) {
                const double2 v = p2[k];
                t0 = max(t0, dg_mag(v.x));
                t1 = max(t1, dg_mag(v.y));
            }
        } else {
            for (int k = lane; k < K; k += LR) t0 = max(t0, dg_mag(at(k)));
        }
    }
#pragma unroll
    for (int o = LR / 2; o; o >>= 1) {
        t0 = max(t0, __shfl_xor_sync(0xffffffffu, t0, o));
        if (CPLX) t1 = max(t1, __shfl_xor_sync(0xffffffffu, t1, o));
    }
    if (!live) return;
    const int e0 = dg_exponent(t0), e1 = dg_exponent(t1);
    if (lane == 0) {
        ex[(CPLX ? 2 : 1) * r] = e0;
        if (CPLX) ex[2 * r + 1] = e1;
    }
    __nv_bfloat16* o0 = S + (size_t)((CPLX ? 2 : 1) * r) * Kp;
    for (int k0 = lane * 8; k0 < Kp; k0 += 8 * LR) {
        long long q0[8], q1[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int k = k0 + j;
            if (CPLX) {
                const double2 v = k < K ? reinterpret_cast<const double2*>(p)[k] : make_double2(0, 0);
                q0[j] = fixed56(v.x, e0);
                q1[j] = fixed56(v.y, e1);
            } else {
                q0[j] = fixed56(k < K ? at(k) : 0.0, e0);
            }
        }
        dg_store8(q0, o0 + k0, stride);
        if (CPLX) dg_store8(q1, o0 + Kp + k0, stride);
    }
}

template <bool CPLX, bool SCALED = false>
void launch_dg_rows(long long R, int K, const double* src, long long ld, void* S, int* ex, size_t stride, cudaStream_t st,
                    const double* scale = nullptr, int rows = 1)
{
    const int Kp = dg_k_padded(K);
    // lanes per row: as many as have a group of 8 elements to write
    const int lr = Kp > 128 ? 32 : Kp > 64 ? 16 : Kp > 32 ? 8 : 4;
    const unsigned grid = (unsigned)((R * lr + 255) / 256);
    __nv_bfloat16* s = (__nv_bfloat16*)S;
    if (lr == 32) k_dg_rows<CPLX, 32, SCALED><<<grid, 256, 0, st>>>(R, K, Kp, src, ld, s, ex, stride, scale, rows);
    else if (lr == 16) k_dg_rows<CPLX, 16, SCALED><<<grid, 256, 0, st>>>(R, K, Kp, src, ld, s, ex, stride, scale, rows);
    else if (lr == 8) k_dg_rows<CPLX, 8, SCALED><<<grid, 256, 0, st>>>(R, K, Kp, src, ld, s, ex, stride, scale, rows);
    else k_dg_rows<CPLX, 4, SCALED><<<grid, 256, 0, st>>>(R, K, Kp, src, ld, s, ex, stride, scale, rows);
    msd_note_launch();
}

// Columns of a complex matrix src[z][k][c] (row stride ld, batch stride
// src_batch) as operand rows, one per column, batch entry z's rows from z *
// rows + row0 on. MODE 0 writes the row of a left operand, k' = 2 k + part
// (re, im interleaved), to Sa and the two rows of a right operand that make the
// real and the imaginary part of its complex product with such a row,
// (re, -im) and (im, re), to Sb; MODE 1 only the latter; MODE 2 the real and the
// imaginary part as plain rows (for a real left operand) to Sb. All rows of a
// column share its exponent. One block per 16 columns: a pass for the
// exponents, then tiles of 64 k staged in shared memory, so that reads run
// along c and the 16-byte digit stores along k.
template <int MODE>
__global__ void __launch_bounds__(256)
k_dg_cols(int K, int Kp, int nc, const double2* __restrict__ src, long long ld, long long src_batch, int row0, int rows,
          __nv_bfloat16* __restrict__ Sa, int* __restrict__ ea, size_t stride_a, __nv_bfloat16* __restrict__ Sb,
          int* __restrict__ eb, size_t stride_b)
{
    constexpr int TK = MODE == 2 ? 128 : 64;   // k per staged tile
    __shared__ double2 tile[TK][17];
    __shared__ unsigned top[16][17];
    __shared__ int ex[16];
    const int z = blockIdx.x, c0 = blockIdx.y * 16, t = threadIdx.x, cl = t & 15, kl = t >> 4;
    const double2* s = src + (size_t)z * src_batch;
    unsigned mx = 0;
    if (c0 + cl < nc)
        for (int k = kl; k < K; k += 16) {
            const double2 v = s[(size_t)k * ld + c0 + cl];
            mx = max(mx, max(dg_mag(v.x), dg_mag(v.y)));
        }
    top[kl][cl] = mx;
    __syncthreads();
    if (t < 16) {
        for (int i = 1; i < 16; ++i) mx = max(mx, top[i][t]);
        ex[t] = dg_exponent(mx);
        if (c0 + t < nc) {
            const size_t r = (size_t)z * rows + row0 + c0 + t;
            if (MODE == 0) ea[r] = ex[t];
            eb[2 * r] = eb[2 * r + 1] = ex[t];
        }
    }
    __syncthreads();
    // an item is 8 consecutive elements of an operand row: 4 complex k (modes 0,
    // 1) or 8 k of one part (mode 2)
    const int ci = t >> 4, gi = t & 15, e = ex[ci];
    const size_t r = (size_t)z * rows + row0 + c0 + ci;
    const int Kk = MODE == 2 ? Kp : Kp / 2;
    for (int k0 = 0; k0 < Kk; k0 += TK) {
        for (int kk = kl; kk < TK; kk += 16)
            tile[kk][cl] = (k0 + kk < K && c0 + cl < nc) ? s[(size_t)(k0 + kk) * ld + c0 + cl] : make_double2(0, 0);
        __syncthreads();
        if (c0 + ci < nc) {
            if (MODE == 2) {
                const int kb = gi * 8;
                if (k0 + kb < Kp)
                    for (int part = 0; part < 2; ++part) {
                        long long q[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) q[j] = fixed56(part ? tile[kb + j][ci].y : tile[kb + j][ci].x, e);
                        dg_store8(q, Sb + (2 * r + part) * Kp + k0 + kb, stride_b);
                    }
            } else {
                const int kb = gi * 4;
                if (2 * (k0 + kb) < Kp) {
                    long long q[8];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        q[2 * j] = fixed56(tile[kb + j][ci].x, e);
                        q[2 * j + 1] = fixed56(tile[kb + j][ci].y, e);
                    }
                    const size_t o = (size_t)2 * (k0 + kb);
                    uint4 u[DG_S];
                    dg_digits8(q, u);
#pragma unroll
                    for (int i = 0; i < DG_S; ++i) {
                        if (MODE == 0) *reinterpret_cast<uint4*>(Sa + i * stride_a + r * Kp + o) = u[i];
                        // (re, -im): the sign of the odd digits; (im, re): halves swapped
                        __nv_bfloat16* b = Sb + i * stride_b + 2 * r * Kp + o;
                        *reinterpret_cast<uint4*>(b) = make_uint4(u[i].x ^ 0x80000000u, u[i].y ^ 0x80000000u,
                                                                  u[i].z ^ 0x80000000u, u[i].w ^ 0x80000000u);
                        *reinterpret_cast<uint4*>(b + Kp) =
                            make_uint4(__byte_perm(u[i].x, 0, 0x1032), __byte_perm(u[i].y, 0, 0x1032),
                                       __byte_perm(u[i].z, 0, 0x1032), __byte_perm(u[i].w, 0, 0x1032));
                    }
                }
            }
        }
        __syncthreads();
    }
}

// out[r ldo + c] = sum over splits of part[split][r][c], in split order.
__global__ void k_dg_sum(int R, int Cc, int splits, const double2* __restrict__ part, double2* __restrict__ out,
                         long long ldo)
{
    const long long n = (long long)R * Cc, e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (e >= n) return;
    double2 s = part[e];
    for (int i = 1; i < splits; ++i) s = cadd(s, part[(size_t)i * n + e]);
    const long long r = e / Cc;
    out[r * ldo + (e - r * Cc)] = s;
}

}  // namespace

int dg_k_padded(int K) { return (K + DG_BK - 1) / DG_BK * DG_BK; }
size_t dg_row_bytes(int K) { return (size_t)DG_S * dg_k_padded(K) * sizeof(__nv_bfloat16) + sizeof(int); }

void dg_slice_real(long long R, int K, const double* src, long long ld, void* S, int* ex, cudaStream_t st,
                   const double* scale, int rows)
{
    const size_t stride = (size_t)R * dg_k_padded(K);
    if (scale) launch_dg_rows<false, true>(R, K, src, ld, S, ex, stride, st, scale, rows);
    else launch_dg_rows<false>(R, K, src, ld, S, ex, stride, st);
}

void dg_slice_complex(long long R, int K, const double2* src, long long ld, void* S, int* ex, cudaStream_t st)
{
    launch_dg_rows<true>(R, K, (const double*)src, ld, S, ex, (size_t)2 * R * dg_k_padded(K), st);
}

void dg_slice_columns(int mode, int K, int nc, int batch, const double2* src, long long ld, long long src_batch,
                      int row0, int rows, void* Sa, int* ea, void* Sb, int* eb, cudaStream_t st)
{
    if (nc <= 0 || batch <= 0) return;
    const int Kp = dg_k_padded(mode == 2 ? K : 2 * K);
    const size_t sa = (size_t)batch * rows * Kp, sb = 2 * sa;
    const dim3 grid(batch, (nc + 15) / 16);   // x: any number of walkers
    __nv_bfloat16 *a = (__nv_bfloat16*)Sa, *b = (__nv_bfloat16*)Sb;
    if (mode == 0) k_dg_cols<0><<<grid, 256, 0, st>>>(K, Kp, nc, src, ld, src_batch, row0, rows, a, ea, sa, b, eb, sb);
    else if (mode == 1) k_dg_cols<1><<<grid, 256, 0, st>>>(K, Kp, nc, src, ld, src_batch, row0, rows, a, ea, sa, b, eb, sb);
    else k_dg_cols<2><<<grid, 256, 0, st>>>(K, Kp, nc, src, ld, src_batch, row0, rows, a, ea, sa, b, eb, sb);
    msd_note_launch();
}

// Contraction splits: a long contraction with few rows of A (the force bias)
// leaves most SMs idle at small walker counts. At least one exact chunk per
// split; not a function of the walker count, so that a walker's rounding does
// not depend on its chunk.
int dg_splits(int Mr, int K)
{
    const int mt = (Mr + DG_BM - 1) / DG_BM, nkb = dg_k_padded(K) / DG_BK;
    return std::max(1, std::min(std::min(16, 64 / mt), nkb / DG_CHUNK));
}

int dg_gemm(const DgOperand& A, const DgOperand& B, const DgOut& o, int K, unsigned* err, cudaStream_t st)
{
    const int Kp = dg_k_padded(K);
    CUtensorMap ma, mb;
    if ((long long)DG_S * A.rows > 0x7fffffffll || (long long)DG_S * B.rows > 0x7fffffffll) return -1;
    if (tc_make_map(&ma, A.s, Kp, DG_S * A.rows, Kp, DG_BM, true, 64) ||
        tc_make_map(&mb, B.s, Kp, DG_S * B.rows, Kp, DG_BN, true, 64))
        return -1;
    if (cudaFuncSetAttribute(k_tc_dgemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DG_SMEM) != cudaSuccess)
        return -1;
    DgArgs a;
    a.Mr = o.Mr; a.Nc = o.Nc;
    a.a_rows = A.rows; a.b_rows = B.rows; a.a_batch = A.batch_rows; a.b_batch = B.batch_rows;
    a.nkb = Kp / DG_BK;
    a.splits = o.splits;
    a.mt = (o.Mr + DG_BM - 1) / DG_BM;
    a.nt = (2 * o.Nc + DG_BN - 1) / DG_BN;
    a.batch = o.batch;
    a.ea = A.e; a.eb = B.e;
    a.C = o.C; a.c_batch = o.c_batch; a.c_n = o.c_n; a.c_m = o.c_m;
    a.acc = o.acc; a.acc_in = o.acc_in; a.mul = o.mul; a.err = err;
    a.gx = o.gx; a.gy = o.gy; a.eye = o.eye; a.live = o.live;
    for (int i = 0; i < 3; ++i) a.K[i] = o.K[i];
    const long long tiles = (long long)a.mt * a.nt * a.batch * a.splits;
    if (tiles <= 0) return 0;
    if (tiles > 0x7fffffffll) return -1;
    k_tc_dgemm<<<(unsigned)std::min<long long>(tiles, msd_sm_count()), DG_THREADS, DG_SMEM, st>>>(ma, mb, a);
    msd_note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

void dg_sum_splits(int R, int Cc, int splits, const double2* part, double2* out, long long ldo, cudaStream_t st)
{
    const long long n = (long long)R * Cc;
    k_dg_sum<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(R, Cc, splits, part, out, ldo);
    msd_note_launch();
}
