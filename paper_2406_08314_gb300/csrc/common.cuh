// Shared device helpers and the internal launch interface of libmsd.
// Internal to the CUDA library; nothing outside csrc/ includes it.
#pragma once

#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

#define MSD_KMAX 6          // highest excitation level per spin
#define MSD_NMAX 64         // electrons per spin
#define MSD_XMAX 112        // n_h * n_p per spin (active hole x particle block)

// Row pitch (complex FP32 entries) of the mixed path's Lambda / Xi rows per
// (walker, Cholesky vector): X rounded up to 16 entries = 128 bytes, so that
// each row starts a cache line and is written in whole lines.
__host__ __device__ __forceinline__ int lam_pitch(int X) { return (X + 15) / 16 * 16; }

// Work decomposition of the per-determinant kernels: threads per block and
// strings (determinants) per thread. One block writes one partial-sum slot.
#define SE_THREADS 256
#define SE_PER_THREAD 4
#define PC_THREADS 256
#define PC_PER_THREAD 8
// The per-determinant terms take one launch for all their levels up to this many
// blocks per SM (a few resident waves of blocks); above, a launch per level with
// that level's registers.
#define ONE_LAUNCH_BLOCKS 6


// ---------------------------------------------------------------- complex
__host__ __device__ __forceinline__ double2 cz(double r, double i) { return make_double2(r, i); }
__host__ __device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }
// a + b * c
__host__ __device__ __forceinline__ double2 cfma(double2 b, double2 c, double2 a) {
    return make_double2(fma(b.x, c.x, fma(-b.y, c.y, a.x)), fma(b.x, c.y, fma(b.y, c.x, a.y)));
}
// a - b * c
__host__ __device__ __forceinline__ double2 cfms(double2 b, double2 c, double2 a) {
    return make_double2(fma(-b.x, c.x, fma(b.y, c.y, a.x)), fma(-b.x, c.y, fma(-b.y, c.x, a.y)));
}
__host__ __device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    // Smith's algorithm
    if (fabs(b.x) >= fabs(b.y)) {
        double r = b.y / b.x, d = b.x + b.y * r;
        return make_double2((a.x + a.y * r) / d, (a.y - a.x * r) / d);
    }
    double r = b.x / b.y, d = b.x * r + b.y;
    return make_double2((a.x * r + a.y) / d, (a.y * r - a.x) / d);
}
__host__ __device__ __forceinline__ double cabs1(double2 a) { return fabs(a.x) + fabs(a.y); }

__host__ __device__ __forceinline__ float2 fz(float r, float i) { return make_float2(r, i); }
__host__ __device__ __forceinline__ float2 fadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 fmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ float2 ffma(float2 b, float2 c, float2 a) {
    return make_float2(fmaf(b.x, c.x, fmaf(-b.y, c.y, a.x)), fmaf(b.x, c.y, fmaf(b.y, c.x, a.y)));
}

// Count of kernel launches made by the library (for launch accounting).
void msd_note_launch();
// Streaming multiprocessors of the current device (queried once per device).
int msd_sm_count();

// ------------------------------------------------------------ device state
// Error word bits set by kernels (read back by the host after a call).
#define MSD_DEV_ERR_SINGULAR 1u
#define MSD_DEV_ERR_TIMEOUT  2u
#define MSD_DEV_ERR_BOUNDS   4u
// The error word is four 32-bit words: [0] the flags above, [1] unused,
// [2..3] the budget of the tensor-core kernels' pipeline waits in
// nanoseconds (one 64-bit value; about 2 s unless the caller changes it).
#define MSD_ERR_WORDS 4
#define MSD_WAIT_DEFAULT_NS 2000000000ull
// Allocate and initialise an error word on the current device (0 or -1).
int msd_err_word_alloc(unsigned** out);

// Per-spin trial tables on the device.
struct SpinTables {
    int N;              // electrons
    int nh, np;         // active holes (orbitals of D0 ever vacated) / particles
    int n_str;          // distinct excitation strings, reference string first
    int bucket[MSD_KMAX + 2];   // strings of level k: [bucket[k], bucket[k+1])
    const int* occ0;    // [N]
    const int* pos0;    // [M] position of an orbital in occ0, or -1
    const int* hole_pos;   // [nh] position in occ0 of each hole orbital
    const int* part_orb;   // [np] orbital of each particle
    const uint4* str_hp;   // [n_str] one 16-byte record per string: hole indices (0..nh-1,
                           // ascending) in bytes 0..5, particle indices (0..np-1,
                           // ascending) in bytes 8..13, so one vector load fetches both
    const int* sub;        // [n_str][MSD_KMAX] of a level >= 4 string: the strings without its last hole
                           // and its j-th particle, (index << 1 | sign of the term), -1 first if one
                           // of them is not in the trial
    const int8_t* str_sign;    // [n_str] parity of the in-place -> sorted reordering
    const int* csr_off;    // [n_str+1] determinants containing each string
    const int* csr_other;  // [nnz] string of the opposite spin in that determinant
    const double* csr_c;   // [nnz] CI coefficient of that determinant
    const uint8_t* cmx;    // [sum_k k^2 n_k] x = p_i nh + h_j of entry (i, j) of each string's
                           // minor, bucket-major, a string's k^2 entries row-major (B's order)
    const uint8_t* kx;     // same layout: h_j np + p_i, the row/column of the Gram matrices
    const float* csr_cf;   // [nnz] csr_c in FP32
    long long b_off[MSD_KMAX + 2];  // per-walker offset (complex units) of each bucket's B block
    long long b_per_walker;         // sum_k b_stride(k) * (strings of level k)
    long long cmx_off[MSD_KMAX + 2];  // offset of each bucket's entries in cmx
};

// Complex entries per string in the inverse-minor arrays B: k^2 rounded up
// to even, so that in FP32 every string's block starts on a 16-byte boundary
// and two entries load as one 16-byte vector (the pad entry is zero).
__host__ __device__ __forceinline__ constexpr int b_stride(int k) { return k * k + (k & 1); }

// Index of the pair (a, b), a < b < n, among the n (n - 1) / 2 pairs in
// lexicographic order.
__host__ __device__ __forceinline__ int pair_index(int a, int b, int n) { return a * n - a * (a + 1) / 2 + (b - a - 1); }

// Hole / particle index i (< MSD_KMAX) of a string record.
__device__ __forceinline__ int rec_h(const uint4& r, int i) { return (int)(((i < 4 ? r.x : r.y) >> (8 * (i & 3))) & 0xffu); }
__device__ __forceinline__ int rec_p(const uint4& r, int i) { return (int)(((i < 4 ? r.z : r.w) >> (8 * (i & 3))) & 0xffu); }


#ifdef __CUDACC__
// 1 / m for m > 0: y <- y + y (1 - m y) (Newton-Raphson for f(y) = 1/y - m),
// two steps from the FP32 reciprocal (~2^-22 relative) reach FP64 rounding
// (2^-44, then below 2^-53 before rounding). Outside the FP32 normal range
// the quotient is taken directly.
__device__ __forceinline__ double recip_nr(double m)
{
    if (!(m > 1e-36 && m < 1e36)) return 1.0 / m;
    float yf;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"((float)m));
    double y = (double)yf;
    double e = fma(-m, y, 1.0);
    y = fma(y, e, y);
    e = fma(-m, y, 1.0);
    return fma(y, e, y);
}

__device__ __forceinline__ double2 crecip(double2 z)
{
    const double m2 = fma(z.x, z.x, z.y * z.y);
    if (!(m2 > 1e-280 && m2 < 1e280)) return cdiv(cz(1, 0), z);
    const double i = recip_nr(m2);
    return cz(z.x * i, -z.y * i);
}

// monotone in max(|Re v|, |Im v|) up to the low 32 bits of each mantissa
__device__ __forceinline__ int mag_key(double2 v)
{
    return max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
}

// x 2^-e (|x| < 2^e) as an integer of BITS fractional bits, rounded to nearest, ties to
// even (integer operations only: FP64 ones issue at a sixty-fourth of their rate). Ties are
// common: a value some bits below the scale drops that many bits, so halves upwards
// would bias every magnitude by up to 2^-53 of it.
template <int BITS>
__device__ __forceinline__ long long fixed_point(double x, int e)
{
    const long long b = __double_as_longlong(x);
    const int f = (int)((b >> 52) & 0x7ff);
    long long m = b & 0xfffffffffffffll;
    if (f) m |= 1ll << 52;
    const int sh = (f ? f : 1) - 1075 + BITS - e;   // below 63 (e >= -1073), m 2^sh below 2^BITS
    if (sh >= 0) m <<= sh;
    else m = sh > -56 ? (m + (1ll << (-sh - 1)) - 1 + ((m >> -sh) & 1)) >> -sh : 0;
    return b < 0 ? -m : m;
}
__device__ __forceinline__ long long fixed56(double x, int e) { return fixed_point<56>(x, e); }

// (hi 2^28 + lo) 2^s outside the fast path below (zeros, results beyond FP64's
// normal range, sums above 64 bits); a call, so that its FP64 conversions are not
// issued speculatively for every value.
static __device__ __noinline__ double int_to_fp64_slow(long long hi, long long lo, int s)
{
    return ldexp(fma((double)hi, 268435456.0, (double)lo), s);
}

// v 2^s rounded to FP64 (to nearest, ties to even) by integer operations (a conversion from 64 bits and a
// scaling are two operations of the FP64 unit, 2 per clock and SM).
__device__ __forceinline__ double int_to_fp64(long long v, int s)
{
    unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)u), ex = 1086 + s - lz;   // biased exponent of the leading bit
    if (u == 0 || ex < 1 || ex > 2045) return int_to_fp64_slow(0, v, s);
    u <<= lz;
    // the mantissa's leading bit adds one to the exponent field, a carry out of
    // the rounding another one
    unsigned long long m = u >> 11;
    m += (((unsigned)u & 2047u) + 1023u + ((unsigned)m & 1u)) >> 11;
    return __longlong_as_double((long long)((((unsigned long long)(ex - 1)) << 52) + m) | (v & (long long)(1ull << 63)));
}

// GELU of the control-variate network and its derivative.
__device__ __forceinline__ float net_gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float net_gelu_d(float z)
{
    return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// Sum of n partial sums by one warp (every lane returns it).
__device__ __forceinline__ double2 warp_sum_slots(const double2* __restrict__ p, int n, int lane)
{
    double2 a = make_double2(0, 0);
    for (int i = lane; i < n; i += 32) a = cadd(a, p[i]);
    for (int o = 16; o; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
    }
    return a;
}
#endif

// Pair (determinant) tables for the opposite-spin cross term.
struct PairTables {
    int n_det;
    int bucket[(MSD_KMAX + 1) * (MSD_KMAX + 1) + 1];  // by (ka, kb): index ka*(KMAX+1)+kb
    const int* a;       // [n_det] alpha string
    const int* b;       // [n_det] beta string
    const double* c;    // [n_det] coefficient
    const float* cf;    // [n_det] coefficient in FP32
    const int* det_index;  // [n_det] original position in the trial list
    // runs form of the opposite-spin term: per bucket 0 (per determinant),
    // 1 (runs sharing an alpha string) or 2 (runs sharing a beta string);
    // runs[run_off[b] ..] the first determinant of each run of bucket b
    int run_side[(MSD_KMAX + 1) * (MSD_KMAX + 1)];
    int run_off[(MSD_KMAX + 1) * (MSD_KMAX + 1) + 1];
    const int* runs;
};

// Workspace pointers for one chunk of walkers (nw walkers).
struct Work {
    int nw;             // walkers in this chunk
    int M;
    double2* Gr[2];     // [nw][N][M]     G[occ0_j][r] = Theta[r][j]
    double2* O0[2];     // [nw]           det(D0^dag phi)
    double2* Gact[2];   // [nw][nh][np]   G[h][p]
    double2* r[2];      // [nw][n_str]    ratio per string
    double2* B[2];      // [nw * b_per_walker] inverse minors (bucket-major, SoA within bucket)
    float2* Bf[2];      // FP32 copy for the mixed path (same layout)
    double2* wts[2];    // [nw][n_str]    r_s times the sum over dets containing the string of c * r_other
    double2* part;      // [nw][nslot]    per-block partial sums
    int nslot;
    unsigned* err;      // device error word
};
