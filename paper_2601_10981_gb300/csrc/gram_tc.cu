// Gram matrix G = W^T W of FP64 columns on GB300's fifth-generation tensor cores
// (tcgen05.mma, BF16 operands, FP32 accumulation in tensor memory), with FP64 accuracy.
//
// Step 1 of POD_Mode (Algorithm 1) forms the Gram matrix of the snapshots; its trailing
// eigenvalues (down to 1e-13 of the largest) decide the POD dimension, so the Gram must
// be as accurate as an FP64 one (~1e-15 relative).  A BF16 or TF32 product is not.  Here
// every FP64 value is cut, error-free, into integer digits that BF16 holds exactly, and
// the tensor core multiplies digits:
//
//   column i is aligned to its largest magnitude, 2^(e_i - 2) > max_p |W[p, i]|, and each
//   value is written as  W[p, i] = 2^e_i * sum_{s=1..8} d_s(p, i) 2^(-7 s)  (+ < 2^(e_i-56))
//   with balanced digits d_s in [-64, 63] (the value truncated to 2^-53 of the column's
//   largest magnitude; the headroom bit keeps the top digit from carrying out);
//   G[i, j] = 2^(e_i + e_j) * sum_{s,t} 2^(-7 (s + t)) sum_p d_s(p, i) d_t(p, j).
//
// A digit product is an integer of at most 2^12 in magnitude, so a sum of 4096 of them
// is an integer below 2^24 and exact in the FP32 accumulator.  Products of equal weight
// (equal s + t) share an accumulator: with the two slices s, s+1 (s odd) stacked as the
// 128 rows of the MMA's A operand and slice t as its B operand, the accumulator of tile c
// collects, in its top 64 lanes, the products with s + t = c and, in its bottom 64 lanes,
// those with s + t = c + 1, from at most four (s, t) pairs each.  Every 1024 points
// (4 x 1024 x 2^12 = 2^24) the eight tiles (c = 2..9, all pairs with s + t <= 9; the
// dropped ones weigh below 2^-58 of a leading product) are read back with tcgen05.ld and
// added, with their weights, into exact 96-bit integers, which are rounded once a chunk.
// The only other rounding is the 56-bit truncation of each value, so the result has the
// accuracy of an FP64 Gram.
//
// Two forms share the digit scheme: the wide one described here (up to 64 columns,
// gram_tc_kernel) and a narrow, warp-specialised one for up to 32 columns
// (gram_tc32_kernel, described at its definition), which sums exactly and rounds once.
//
// Wide form.  A persistent grid, one CTA per SM (the eight tiles fill the SM's 512 TMEM
// columns); a CTA takes work units (batch item, chunk of points) in turn and, per stage
// of 64 points, 512 threads cut eight values each (loaded a stage ahead) into digits and
// store them into a ring of two stages in the MMA operands' layout; a seventeenth warp issues the MMAs.  Slices
// follow one another in a stage, so one B operand spans four of them (N = 256) and a K-step
// is six MMAs.  Every wait on an mbarrier is bounded: on time-out the kernel records
// PR_ERR_TIMEOUT, waits (bounded) for its MMAs in flight, frees its tensor memory and
// returns.  Column maxima come from a pre-pass (colmax_kernel).
// Four windows of 64 columns on 128^3: 6.5 -> 2.4 ms (one: 1.72 -> 0.60 ms, the tensor pipe 71 %
// busy, it was 22; a POD call 18.2 -> 12.9 ms).
#include "pr_internal.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <stdint.h>

namespace pr {

namespace {

constexpr int TC_PROD = 512;          // producer threads: four warps for each tensor-memory lane quarter
constexpr int TC_THREADS = TC_PROD + 32;   // + the MMA warp
constexpr int TC_N = 64;             // columns handled (K <= 64)
constexpr int TC_PTS = 64;           // points per shared-memory stage
constexpr int TC_SLICES = 8;         // digits per value
constexpr int TC_TILES = 8;          // accumulator tiles c = 2..9
constexpr int TC_WIN = 1024;         // points per accumulation window
constexpr int TC_TMEM_COLS = TC_TILES * TC_N;   // 512: all of an SM's tensor memory
// operand layout: K-major with the 128-byte swizzle.  A digit row (one slice of one column of W)
// holds a stage's 64 points in 128 bytes; its 16-byte chunk g (8 points) sits at chunk
// g ^ (row % 8), so that the eight chunks of a row, stored by eight neighbouring threads, hit
// distinct banks; groups of 8 rows are SBO = 1024 bytes apart.  Slices follow one another, so B
// operands of 2 or 4 slices (N = 128, 256) are one descriptor.  The order of the points within a
// row is free (the same for all rows): thread g's chunk holds the point pairs g, g + 8, g + 16
// and g + 24 of the stage, and a warp's loads take whole 128-byte lines.
constexpr int TC_SBO = 1024;
constexpr int TC_STAGE_BYTES = TC_SLICES * 8 * TC_SBO;   // 64 KiB
constexpr int TC_NS = 2;                                 // stages in the digit ring
constexpr int TC_SMEM = TC_NS * TC_STAGE_BYTES + 48 * TC_PROD * 4;   // + the exact sums
constexpr long long TC_SPIN_LIMIT = 1LL << 24;   // polls of an mbarrier (~1 s with the sleeps)

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

// UMMA shared-memory matrix descriptor (K-major, 128-byte swizzle = 2 at bit 61): start address
// and stride (8-row group) byte offset, each >> 4; descriptor version 1 at bit 46.  A K-step of
// 16 points advances the start by 32 bytes.
__device__ __forceinline__ uint64_t umma_desc(unsigned saddr) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(TC_SBO >> 4) << 32) | (1ull << 46) |
           (2ull << 61);
}

// Instruction descriptor of kind::f16: D FP32 (bits 4-5 = 1), A and B BF16 (bits 7-9 and
// 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
constexpr unsigned tc_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(n >> 3) << 17) | ((unsigned)(128 >> 4) << 24);
}

template <int N>
__device__ __forceinline__ void mma_bf16(unsigned tmem_d, uint64_t adesc, uint64_t bdesc, unsigned accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(tc_idesc(N)), "r"(accum));
}

__device__ __forceinline__ void mma_commit(unsigned mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

// Bounded wait for phase `parity` of the mbarrier (non-blocking test, short sleeps: about
// a second at most with the default limit); false on time-out.
__device__ __forceinline__ bool mbar_wait(unsigned mbar, unsigned parity, long long limit = TC_SPIN_LIMIT) {
    for (long long it = 0; it <= limit; ++it) {
        unsigned ok = 0;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (it >= 64) __nanosleep(64);
    }
    return false;
}

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float (&v)[8]) {
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[e]);
}

}  // namespace

// colmax[b * ld + i] = bit pattern of max_p |W_b[p, i]| (non-negative doubles order like
// their bit patterns), by atomicMax from each CTA's chunk; the buffer starts at zero.
// Eight columns at a time, two points a load where the columns are 16-byte aligned (eight
// independent 16-byte loads in flight per thread), per-warp maxima in shared memory, one
// barrier and one atomic per column and CTA.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__device__ __forceinline__ unsigned long long umax64(unsigned long long x, unsigned long long y) {
    return x > y ? x : y;
}
__global__ void __launch_bounds__(256) colmax_kernel(GramArgs a, long long CH, unsigned long long* colmax,
                                                     int ld) {
    const int b = blockIdx.y;
    const int K = a.KA[b];
    const long long p_lo = (long long)blockIdx.x * CH, p_hi = min(a.Ng, p_lo + CH);
    const void* const* cols = a.colsA + (size_t)b * a.ldcols;
    __shared__ unsigned long long red[8][64];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < K; i0 += 8) {
        const double* c[8];
        unsigned long long m[8];
        bool al = (p_lo & 1) == 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {   // columns past K read column i0 again (never stored)
            c[j] = reinterpret_cast<const double*>(cols[i0 + j < K ? i0 + j : i0]);
            m[j] = 0ull;
            al = al && ((reinterpret_cast<uintptr_t>(c[j]) & 15u) == 0);
        }
        long long p = p_lo + (al ? 2 * (long long)threadIdx.x : (long long)threadIdx.x);
        if (al) {
            for (; p + 1 < p_hi; p += 2 * (long long)blockDim.x) {
                double2 v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = *reinterpret_cast<const double2*>(c[j] + p);
#pragma unroll
                for (int j = 0; j < 8; ++j) m[j] = umax64(m[j], umax64(abs_bits(v[j].x), abs_bits(v[j].y)));
            }
        }
        // the remaining single points (an odd tail, or every point of unaligned columns)
        for (; p < p_hi; p += (al ? 2 * (long long)blockDim.x : (long long)blockDim.x)) {
#pragma unroll
            for (int j = 0; j < 8; ++j) m[j] = umax64(m[j], abs_bits(c[j][p]));
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) m[j] = umax64(m[j], __shfl_xor_sync(0xffffffffu, m[j], off));
            if (lane == 0 && i0 + j < K) red[warp][i0 + j] = m[j];
        }
    }
    __syncthreads();
    if (threadIdx.x < K) {
        unsigned long long t = 0ull;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = umax64(t, red[w][threadIdx.x]);
        if (t) atomicMax(colmax + (size_t)b * ld + threadIdx.x, t);
    }
}

namespace {

// ---------------------------------------------------------------------------------------
// Narrow form, K <= 32 columns: one M = 128 x N = 256 x K = 16 MMA per 16 points.
//
// The digit rows of a stage are slice s (0 = most significant) x 32 columns, 256 rows in
// all.  A is rows 0..127 (slices 0..3), B all 256 rows (slices 0..7), so one MMA forms
// every product D_s^T D_t with s <= 3: accumulator lane 32 s + i, column 32 t + j holds
// P_st[i, j] = sum_p d_s(p, i) d_t(p, j).  The Gram needs the pairs with min(s, t) <= 3
// (the pairs with both s, t >= 4 weigh below 2^-58 of 2^(e_i + e_j); the wide form above
// drops more); those with s >= 4 are transposes of computed ones, P_st = P_ts^T, so
//   G = sum_{s<=3, t} w_st P_st + (sum_{s<=3, t>=4} w_st P_st)^T,  w_st = 2^(-7 (s+t+2)).
// Each accumulator position takes one digit product a point, so a window of 4096 points
// stays below 2^24 (exact in FP32); the tensor memory holds two windows (2 x 256 columns)
// and the MMAs of one run while the other is read back.
//
// Warp roles: warps 0-7 load the FP64 values (one stage ahead, in registers), cut them
// into digits, store them into a ring of four shared-memory stages, and read back the
// accumulators of finished windows; warp 8 issues the MMAs (one thread) and owns the
// tensor memory.  They meet only at mbarriers (stage full / stage free / window done /
// window read), every wait bounded.  Read-back is integer: each (s, i, j) folds its eight
// tiles into two exact 64-bit integers H (t <= 3) and L (t >= 4), kept in shared memory
// over the windows of a work unit; at the unit's end the 12 terms of each output are
// summed exactly in 128-bit integers and stored as the unit's partial; the last unit of
// an item adds the partials (exact) and rounds once to FP64.  The result is the exactly
// rounded value of the digit sum: reproducible bit for bit, whatever the chunking.
constexpr int N2_PROD = 256;                     // producer threads (warps 0-7)
constexpr int N2_THREADS = N2_PROD + 32;         // + the MMA warp
constexpr int N2_COLS = 32;
constexpr int N2_PTS = 64;                       // points per stage
constexpr int N2_NS = 3;                         // stages in the digit ring
constexpr int N2_DEPTH = 3;                      // stages of FP64 values in flight (cp.async)
constexpr int N2_STG_BYTES = N2_PTS * N2_COLS * 8;   // 16 KiB of FP64 values a stage
constexpr int N2_STAGE_BYTES = TC_SLICES * N2_COLS * N2_PTS * 2;   // 32 KiB
constexpr int N2_WIN = 4096;                     // points per accumulation window (2^12)
constexpr int N2_TMEM_COLS = 512;                // two windows of 256 FP32 columns
constexpr int N2_XP = 33;                        // 64-bit row pitch of the exchange arrays
constexpr int N2_XWORDS = 4 * 32 * N2_XP;        // per array (H or L)
constexpr int N2_SMEM = N2_NS * N2_STAGE_BYTES + (N2_DEPTH + 1) * N2_STG_BYTES + 2 * N2_XWORDS * 8;
static_assert(N2_SMEM + 256 <= 227 * 1024, "shared memory of the narrow form");
constexpr unsigned N2_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(256 >> 3) << 17) |
                              ((unsigned)(128 >> 4) << 24);
// B = sum_{k=0..7} 64 * 128^k: z = y + B has the unsigned base-128 digits u_k = d_k + 64
constexpr unsigned long long N2_BIAS = 0x0081020408102040ull;

__device__ __forceinline__ unsigned long long shr64_clamp(unsigned long long x, unsigned r) {
    unsigned long long y;
    asm("shr.b64 %0, %1, %2;" : "=l"(y) : "l"(x), "r"(r));   // r >= 64 gives 0
    return y;
}

// Digit field bp of z (bits bp .. bp + 6 of the 56-bit z = zh:zl) for two points, packed
// as a BF16 pair of the digits u - 64: the halves hold 128 + u (bits 0x4300 | u), and one
// packed BF16 subtraction of 192 leaves u - 64 exactly.
template <int BP>
__device__ __forceinline__ unsigned digit_pair(unsigned zla, unsigned zha, unsigned zlb, unsigned zhb) {
    unsigned fa, fb16;
    if constexpr (BP + 7 <= 32) {
        fa = zla >> BP;
        fb16 = (BP <= 16) ? (zlb << (16 - BP)) : (zlb >> (BP - 16));
    } else if constexpr (BP >= 32) {
        fa = zha >> (BP - 32);
        fb16 = (BP - 32 <= 16) ? (zhb << (16 - (BP - 32))) : (zhb >> (BP - 32 - 16));
    } else {
        fa = __funnelshift_r(zla, zha, BP);
        fb16 = __funnelshift_r(zlb, zhb, BP) << 16;
    }
    const unsigned w = (fa & 0x7Fu) | (fb16 & 0x7F0000u) | 0x43004300u;
    __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162*>(&w);
    const unsigned c192 = 0x43404340u;
    v = __hsub2(v, *reinterpret_cast<const __nv_bfloat162*>(&c192));
    return *reinterpret_cast<const unsigned*>(&v);
}

// z = 2^(56 - e) x truncated toward zero, plus the bias, as two 32-bit words; ce = e + 1020.
// Zero and subnormal x take the effective exponent 1 (no implicit bit).
__device__ __forceinline__ void cut56(double x, int ce, unsigned& zl, unsigned& zh) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(bits >> 32), lo = (unsigned)bits;
    const unsigned exf = hi & 0x7FF00000u;
    const unsigned imp = min(exf, 0x100000u);
    const int exe = (int)(max(exf, 0x100000u) >> 20);
    const unsigned long long m = ((unsigned long long)((hi & 0xFFFFFu) | imp) << 32) | lo;
    const unsigned long long y = shr64_clamp(m << 1, (unsigned)(ce - exe));   // ce >= exe
    const unsigned long long sg = (unsigned long long)(long long)((int)hi >> 31);
    const unsigned long long z = (N2_BIAS - sg) + (y ^ sg);
    zl = (unsigned)z;
    zh = (unsigned)(z >> 32);
}

// Bounded mbarrier wait that also gives up once another thread has recorded a failure.
// try_wait suspends the thread (at most ~1 us a try, by its time hint) instead of
// spinning, so waiting warps leave the issue slots to the others; `limit` tries (the
// context's spin limit, 2^22 ~ a few seconds by default).  limit 0: one non-blocking
// test, so that a wait not already complete gives up at once.
__device__ __forceinline__ bool mbar_wait_f(unsigned mbar, unsigned parity, volatile int* fail, long long limit) {
    if (limit == 0) {
        if (mbar_wait(mbar, parity, 0)) return true;
        *fail = 1;
        return false;
    }
    for (long long it = 0; it <= limit; ++it) {
        unsigned ok = 0;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(ok)
            : "r"(mbar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 15) == 15 && *fail) return false;
    }
    *fail = 1;
    return false;
}
__device__ __forceinline__ void mbar_arrive(unsigned mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

__device__ __forceinline__ void prod_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

__device__ __forceinline__ void mma_n256(unsigned tmem_d, uint64_t desc, unsigned accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %1, %2, p;\n\t}\n" ::"r"(tmem_d),
        "l"(desc), "r"(N2_IDESC), "r"(accum));
}

// the exponent e of a column (2^(e - 2) > max |W[:, i]|) from its column-maximum bits
__device__ __forceinline__ int col_exp(unsigned long long m) {
    return m ? (int)((m >> 52) & 0x7FF) - 1023 + 3 : 0;
}

// a column that holds an infinity or a NaN: its digits mean nothing, its products are NaN
__device__ __forceinline__ bool col_bad(unsigned long long m) { return m >= 0x7FF0000000000000ull; }

// 2^sc * S, rounded once to the nearest double (ties to even)
__device__ __forceinline__ double i128_to_double(__int128 S, int sc) {
    if (S == 0) return 0.0;
    const bool neg = S < 0;
    const unsigned __int128 u = neg ? (unsigned __int128)(-S) : (unsigned __int128)S;
    const unsigned long long hi = (unsigned long long)(u >> 64), lo = (unsigned long long)u;
    unsigned long long v = lo;
    int sh = 0;
    if (hi != 0) {
        sh = 64 - __clzll((long long)hi);   // 1..64: the bits above the low word
        const unsigned long long rest = sh == 64 ? lo : (lo << (64 - sh));
        v = (sh == 64 ? hi : ((hi << (64 - sh)) | (lo >> sh))) | (rest != 0 ? 1ull : 0ull);   // sticky bit
    }
    const double d = __ull2double_rn(v);
    // times 2^(sh + sc) in two exact power-of-two factors (each exponent within the normal range)
    const int k = sh + sc, k1 = max(-1022, min(1023, k / 2)), k2 = max(-1022, min(1023, k - k / 2));
    const double f1 = __longlong_as_double((long long)(k1 + 1023) << 52);
    const double f2 = __longlong_as_double((long long)(k2 + 1023) << 52);
    return (neg ? -d : d) * f1 * f2;
}

}  // namespace

// 9 warps: three share one SM sub-partition's 16K registers, so at most 168 a thread
__global__ void __launch_bounds__(N2_THREADS, 1) gram_tc32_kernel(GramArgs a, long long U, int chunks,
                                                                  const unsigned long long* colmax, int ld,
                                                                  int* err, long long limit) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long s_bar[2 * N2_NS + 5];
    __shared__ unsigned s_tmem;
    __shared__ volatile int s_fail;
    __shared__ int s_last;
    unsigned char* stg = smem_raw + N2_NS * N2_STAGE_BYTES;   // FP64 staging ring, N2_DEPTH + 1 slots
    long long* sH = reinterpret_cast<long long*>(stg + (N2_DEPTH + 1) * N2_STG_BYTES);
    long long* sL = sH + N2_XWORDS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned full0 = smem_u32(&s_bar[0]);            // [N2_NS], 256 arrivals
    const unsigned empty0 = smem_u32(&s_bar[N2_NS]);       // [N2_NS], MMA commit
    const unsigned tfull0 = smem_u32(&s_bar[2 * N2_NS]);   // [2], MMA commit
    const unsigned tempty0 = tfull0 + 16;                  // [2], 256 arrivals
    const unsigned done = tfull0 + 32;                     // MMA commit at exit
    const unsigned stage_s = smem_u32(smem_raw);

    if (tid == 0) {
        for (int q = 0; q < N2_NS; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8u * q), "r"(N2_PROD) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty0 + 8u * q) : "memory");
        }
        for (int h = 0; h < 2; ++h) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tfull0 + 8u * h) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tempty0 + 8u * h), "r"(N2_PROD) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    // zero the stage ring once (digit rows of columns >= K then only ever hold digits of
    // earlier items, which reach no output read back)
    for (int e = tid; e < N2_NS * N2_STAGE_BYTES / 16; e += N2_THREADS)
        reinterpret_cast<uint4*>(smem_raw)[e] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == 8) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(N2_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    const int units = a.B * chunks;
    auto unit_lo = [&](int u) -> long long { return (long long)(u % chunks) * U; };
    auto unit_hi = [&](int u) -> long long { return min(a.Ng, (long long)(u % chunks) * U + U); };

    if (warp == 8) {
        // ---------------- MMA issue (one thread) ----------------
        if (lane == 0) {
            int gs = 0, gw = 0;
            bool bad = false;
            for (int u = blockIdx.x; u < units; u += gridDim.x) {
                const long long lo = unit_lo(u), hi = unit_hi(u);
                for (long long w0 = lo; w0 < hi; w0 += N2_WIN, ++gw) {
                    const long long w1 = min(hi, w0 + N2_WIN);
                    const int h = gw & 1;
                    if (!bad && !mbar_wait_f(tempty0 + 8u * h, ((gw >> 1) & 1) ^ 1, &s_fail, limit)) bad = true;
                    const unsigned td = tmem + (unsigned)(h * 256);
                    for (long long p0 = w0; p0 < w1; p0 += N2_PTS, ++gs) {
                        const int q = gs % N2_NS;
                        if (!bad && !mbar_wait_f(full0 + 8u * q, (gs / N2_NS) & 1, &s_fail, limit)) bad = true;
                        if (!bad) {
                            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                            const unsigned sb = stage_s + q * N2_STAGE_BYTES;
#pragma unroll
                            for (int k = 0; k < N2_PTS / 16; ++k)
                                mma_n256(td, umma_desc(sb + k * 32), (p0 == w0 && k == 0) ? 0u : 1u);
                        }
                        mma_commit(empty0 + 8u * q);
                    }
                    mma_commit(tfull0 + 8u * h);
                }
            }
            mma_commit(done);
            mbar_wait(done, 0);   // every MMA of this CTA has completed (bounded; also after a failure)
        }
        __syncwarp();
    } else {
        // ---------------- producers / read-back (warps 0-7) ----------------
        const int col = tid >> 3, g8 = tid & 7;   // this thread's column and chunk of a stage
        const int qd = warp & 3, ch = warp >> 2;   // read-back: lane quarter (slice s) and column half
        bool bad = false;
        int gw = 0;
        // one pending read-back: window pw of unit pu (its first / last window?)
        int pu = -1, pw = 0;
        bool pfirst = false, plast = false;

        // Position in the CTA's sequence of stages, with the unit's values kept in registers
        // (no divisions per stage): unit u (item b, K columns, points lo .. hi), stage at p0,
        // and this thread's column pointer (null for col >= K).
        struct Pos {
            int u, b, K;
            long long lo, hi, p0;
            const double* c;
        };
        auto set_unit = [&](Pos& P, int u) {
            P.u = u;
            if (u >= units) return;
            P.b = u / chunks;
            P.K = a.KA[P.b];
            P.lo = (long long)(u - P.b * chunks) * U;
            P.hi = min(a.Ng, P.lo + U);
            P.p0 = P.lo;
            P.c = col < P.K ? reinterpret_cast<const double*>(a.colsA[(size_t)P.b * a.ldcols + col]) : nullptr;
        };
        auto advance = [&](Pos& P) {
            P.p0 += N2_PTS;
            if (P.p0 >= P.hi) set_unit(P, P.u + gridDim.x);
        };
        // this thread's 8 values of a stage, copied by cp.async into its own 16-byte chunks of a
        // staging slot: chunk k (the point pair g8 + 8 k) at (k * 256 + tid) * 16, so that a warp's reads hit distinct banks; points past the
        // unit are zero-filled (source size 0 reads nothing).  Columns >= K are neither
        // copied nor cut: their digit rows reach no output that is read back.
        const unsigned stg_s = smem_u32(stg) + (unsigned)tid * 16u;
        auto issue = [&](const Pos& P, int slot) {
            if (P.c == nullptr) return;
            const long long pb = P.p0 + 2 * g8;
            const unsigned d0 = stg_s + (unsigned)(slot * N2_STG_BYTES);
            if (P.p0 + N2_PTS <= P.hi && ((reinterpret_cast<uintptr_t>(P.c) & 15u) == 0)) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d0 + (unsigned)(k * 256 * 16)),
                                 "l"(P.c + pb + 16 * k)
                                 : "memory");
                return;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {   // 8-byte copies (ragged tail or 8-byte aligned columns)
                const long long pk = pb + 16 * (k >> 1) + (k & 1);
                const bool v = pk < P.hi;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d0 + (unsigned)((k >> 1) * 256 * 16 + (k & 1) * 8)),
                             "l"(v ? P.c + pk : P.c), "r"(v ? 8u : 0u)
                             : "memory");
            }
        };

        auto readback = [&]() {
            const int h = pw & 1;
            if (!bad && !mbar_wait_f(tfull0 + 8u * h, (pw >> 1) & 1, &s_fail, limit)) bad = true;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const unsigned base = tmem + ((unsigned)(32 * qd) << 16) + (unsigned)(h * 256 + 16 * ch);
            long long* hrow = sH + (qd * 32 + lane) * N2_XP + 16 * ch;
            long long* lrow = sL + (qd * 32 + lane) * N2_XP + 16 * ch;
#pragma unroll 1
            for (int j0 = 0; j0 < 16; j0 += 8) {   // two passes of 8 columns (fewer live registers)
                long long H[8], L[8];
#pragma unroll
                for (int e2 = 0; e2 < 8; ++e2) H[e2] = L[e2] = 0ll;
#pragma unroll
                for (int t = 0; t < TC_SLICES; ++t) {
                    float v[8];
                    tmem_ld8(base + (unsigned)(t * 32 + j0), v);
#pragma unroll
                    for (int e2 = 0; e2 < 8; ++e2) {
                        const long long x = (long long)__float2int_rn(v[e2]);   // an exact integer
                        if (t < 4) H[e2] += x << (7 * (3 - t));
                        else L[e2] += x << (7 * (7 - t));
                    }
                }
#pragma unroll
                for (int e2 = 0; e2 < 8; ++e2) {
                    hrow[j0 + e2] = pfirst ? H[e2] : hrow[j0 + e2] + H[e2];
                    lrow[j0 + e2] = pfirst ? L[e2] : lrow[j0 + e2] + L[e2];
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(tempty0 + 8u * h);
            if (!plast) return;
            // ---- the unit's partial: 12 exact terms per output (i <= j), in 128-bit integers
            prod_sync();
            const int b = pu / chunks, chunk = pu - b * chunks;
            const int K = a.KA[b];
            const int mk = a.maxKA;
            __int128* mypart =
                reinterpret_cast<__int128*>(a.part) + ((size_t)b * chunks + chunk) * (size_t)mk * mk;
            for (int o = tid; o < K * K; o += N2_PROD) {
                const int i = o / K, j = o - i * K;
                if (j < i) continue;
                __int128 S = 0;
#pragma unroll
                for (int s = 0; s < 4; ++s) {
                    S += ((__int128)sH[(s * 32 + i) * N2_XP + j]) << (7 * (7 - s));
                    S += ((__int128)(sL[(s * 32 + i) * N2_XP + j] + sL[(s * 32 + j) * N2_XP + i])) << (7 * (3 - s));
                }
                mypart[(size_t)i * mk + j] = S;
            }
            __threadfence();
            prod_sync();
            if (tid == 0) {
                const unsigned ticket = atom_add_acq_rel_u32(a.counter + b, 1u);
                s_last = (ticket == (unsigned)chunks - 1u);
            }
            prod_sync();
            if (s_last) {
                __threadfence();
                const __int128* bpart = reinterpret_cast<const __int128*>(a.part) + (size_t)b * chunks * mk * mk;
                double* Gb = a.G + (size_t)b * a.ldG_b;
                for (int o = tid; o < K * K; o += N2_PROD) {
                    const int i = o / K, j = o - i * K;
                    if (j < i) continue;
                    // the chunk partials in batches of 16 independent loads (a chain of
                    // dependent loads here held the CTA for tens of microseconds)
                    const __int128* src = bpart + (size_t)i * mk + j;
                    const size_t cs = (size_t)mk * mk;
                    __int128 S = 0;
                    int cc = 0;
                    for (; cc + 16 <= chunks; cc += 16) {
                        __int128 v[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) v[e] = src[(size_t)(cc + e) * cs];
#pragma unroll
                        for (int e = 0; e < 16; ++e) S += v[e];
                    }
                    for (; cc < chunks; ++cc) S += src[(size_t)cc * cs];
                    const int sc = col_exp(colmax[(size_t)b * ld + i]) + col_exp(colmax[(size_t)b * ld + j]) - 84;
                    const bool bad = col_bad(colmax[(size_t)b * ld + i]) || col_bad(colmax[(size_t)b * ld + j]);
                    const double g = bad ? nan("") : i128_to_double(S, sc);
                    Gb[(size_t)i * a.ldG + j] = g;
                    Gb[(size_t)j * a.ldG + i] = g;
                }
                if (tid == 0) st_relaxed_u32(a.counter + b, 0u);
            }
            prod_sync();
        };

        // the stages in order; the copies run N2_DEPTH stages ahead of the digit cut
        Pos P, I;
        set_unit(P, blockIdx.x);
        I = P;
        for (int d = 0; d < N2_DEPTH; ++d) {
            if (I.u < units) {
                issue(I, d);
                advance(I);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
        int ce = 0;
        int q = 0, slot = 0;             // digit stage gs % N2_NS, staging slot gs % (N2_DEPTH + 1)
        unsigned eph = 1u;               // parity to wait for on the digit stage's free barrier
        while (P.u < units) {
            if (I.u < units) {
                issue(I, slot == 0 ? N2_DEPTH : slot - 1);   // slot (gs + N2_DEPTH) % (N2_DEPTH + 1)
                advance(I);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            if (P.p0 == P.lo)   // a new unit: this thread's column exponent
                ce = col_exp(P.c ? colmax[(size_t)P.b * ld + col] : 0ull) + 1020;
            asm volatile("cp.async.wait_group %0;" ::"n"(N2_DEPTH) : "memory");   // this stage's copies
            if (!bad && !mbar_wait_f(empty0 + 8u * q, eph, &s_fail, limit)) bad = true;
            if (P.c) {
                double xc[8];
                const unsigned char* sp = stg + (size_t)slot * N2_STG_BYTES + (size_t)tid * 16;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const double2 v = *reinterpret_cast<const double2*>(sp + k * 256 * 16);
                    xc[2 * k] = v.x;
                    xc[2 * k + 1] = v.y;
                }
                unsigned zl[8], zh[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) cut56(xc[k], ce, zl[k], zh[k]);
                // slice s holds digit k = 7 - s (bits 7k .. 7k + 6 of z); row 32 s + col
                unsigned char* rowp = smem_raw + q * N2_STAGE_BYTES + col * 128 + ((g8 ^ (col & 7)) << 4);
#define N2_SLICE(S)                                                                                        \
    *reinterpret_cast<uint4*>(rowp + (S) * 4 * 1024) =                                                     \
        make_uint4(digit_pair<7 * (7 - (S))>(zl[0], zh[0], zl[1], zh[1]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[2], zh[2], zl[3], zh[3]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[4], zh[4], zl[5], zh[5]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[6], zh[6], zl[7], zh[7]));
                N2_SLICE(0) N2_SLICE(1) N2_SLICE(2) N2_SLICE(3) N2_SLICE(4) N2_SLICE(5) N2_SLICE(6) N2_SLICE(7)
#undef N2_SLICE
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            mbar_arrive(full0 + 8u * q);
            // the end of a window: read back the previous one, this one becomes pending
            const long long wend = min(P.hi, P.lo + (((P.p0 - P.lo) >> 12) + 1) * N2_WIN);
            if (P.p0 + N2_PTS >= wend) {
                if (pu >= 0) readback();
                pu = P.u;
                pw = gw;
                pfirst = (P.p0 - P.lo) < N2_WIN;
                plast = (wend == P.hi);
                ++gw;
            }
            if (++q == N2_NS) {
                q = 0;
                eph ^= 1u;
            }
            slot = (slot == N2_DEPTH) ? 0 : slot + 1;
            advance(P);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (pu >= 0) readback();
    }
    if (s_fail && tid == 0) record_error(err, DERR_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 8) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(N2_TMEM_COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------------------
// Wide form, K <= 64 columns (see the head of this file).

namespace {

// four columns of two accumulator tiles
__device__ __forceinline__ void tmem_ld4(unsigned taddr, int (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

__device__ __forceinline__ void tc_prod_sync() { asm volatile("bar.sync 1, 512;" ::: "memory"); }

// (w0, w1, w2) += the 96-bit integer H 2^28 + L
__device__ __forceinline__ void add96(unsigned (&w)[3], long long H, long long L) {
    const unsigned long long h = (unsigned long long)H << 28;
    const unsigned h2 = (unsigned)(int)(H >> 36), l2 = (unsigned)(int)(L >> 63);
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(w[0]), "+r"(w[1]), "+r"(w[2])
        : "r"((unsigned)h), "r"((unsigned)(h >> 32)), "r"(h2));
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(w[0]), "+r"(w[1]), "+r"(w[2])
        : "r"((unsigned)L), "r"((unsigned)((unsigned long long)L >> 32)), "r"(l2));
}

}  // namespace

// 17 warps: five share one SM sub-partition's 16K registers, so at most 96 a thread (the bound of
// 640 threads says so); the exact sums, touched once a window, live in shared memory
__global__ void __launch_bounds__(640, 1) gram_tc_kernel(GramArgs a, int CH, int chunks, int SH, int nsub,
                                                                const unsigned long long* colmax, int ld,
                                                                int* err, long long limit) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long s_bar[2 * TC_NS + 3];
    __shared__ unsigned s_tmem;
    __shared__ volatile int s_fail;
    __shared__ int s_last;
    unsigned* sv = reinterpret_cast<unsigned*>(smem_raw + TC_NS * TC_STAGE_BYTES);   // [16 x 3][TC_PROD]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const unsigned full0 = smem_u32(&s_bar[0]);          // [TC_NS], TC_PROD arrivals
    const unsigned empty0 = smem_u32(&s_bar[TC_NS]);     // [TC_NS], MMA commit
    const unsigned tfull = smem_u32(&s_bar[2 * TC_NS]);  // MMA commit of a window
    const unsigned tempty = tfull + 8;                   // TC_PROD arrivals: a window is read back
    const unsigned done = tfull + 16;                    // MMA commit at exit
    const unsigned stage_s = smem_u32(smem_raw);
    if (tid == 0) {
        for (int q = 0; q < TC_NS; ++q) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full0 + 8u * q), "r"(TC_PROD) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty0 + 8u * q) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tfull) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tempty), "r"(TC_PROD) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(done) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    // zero the ring once (digit rows of columns >= K then only ever hold digits of earlier
    // items, which reach no output read back)
    for (int e = tid; e < TC_NS * TC_STAGE_BYTES / 16; e += TC_THREADS)
        reinterpret_cast<uint4*>(smem_raw)[e] = make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == 16) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = s_tmem;
    // An item's points are cut into chunks of CH, whose sums are rounded, and these into nsub units of
    // SH points (fewer in the last chunk), whose sums stay exact where a chunk has several
    const int Ng = (int)a.Ng;
    const int upi = (chunks - 1) * nsub + (Ng - (chunks - 1) * CH + SH - 1) / SH, units = a.B * upi;
    auto span = [&](int r, int& lo, int& hi) {   // unit r of an item
        const int c = min(r / nsub, chunks - 1);
        lo = c * CH + (r - c * nsub) * SH;
        hi = min(min(Ng, (c + 1) * CH), lo + SH);
    };

    if (warp == 16) {
        // ---------------- MMA issue (one thread) ----------------
        if (lane == 0) {
            int gs = 0, gw = 0;
            bool bad = false;
            for (int u = blockIdx.x; u < units; u += gridDim.x) {
                int lo, hi;
                span(u % upi, lo, hi);
                const int len = hi - lo;
                for (int rel = 0; rel < len; rel += TC_PTS, ++gs) {
                    const bool first = rel % TC_WIN == 0;
                    if (first && !bad && !mbar_wait_f(tempty, (gw & 1) ^ 1, &s_fail, limit)) bad = true;
                    const int q = gs % TC_NS;
                    if (!bad && !mbar_wait_f(full0 + 8u * q, (gs / TC_NS) & 1, &s_fail, limit)) bad = true;
                    if (!bad) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                        for (int k = 0; k < TC_PTS / 16; ++k) {
                            // slices sa, sa + 1 (A) times slices t .. (B) into the tiles from sa + t; the
                            // pairs of slices 0, 1 reach every tile and overwrite it at a window's start
                            const uint64_t d0 = umma_desc(stage_s + q * TC_STAGE_BYTES + 32 * k);
                            const uint64_t sl = (8 * TC_SBO) >> 4;   // next slice, in descriptor units
                            const unsigned acc = (k == 0 && first) ? 0u : 1u;
                            mma_bf16<256>(tmem, d0, d0, acc);
                            mma_bf16<256>(tmem + 4 * TC_N, d0, d0 + 4 * sl, acc);
                            mma_bf16<256>(tmem + 2 * TC_N, d0 + 2 * sl, d0, 1u);
                            mma_bf16<128>(tmem + 6 * TC_N, d0 + 2 * sl, d0 + 4 * sl, 1u);
                            mma_bf16<256>(tmem + 4 * TC_N, d0 + 4 * sl, d0, 1u);
                            mma_bf16<128>(tmem + 6 * TC_N, d0 + 6 * sl, d0, 1u);
                        }
                    }
                    mma_commit(empty0 + 8u * q);
                    if ((rel + TC_PTS) % TC_WIN == 0 || rel + TC_PTS >= len) {
                        mma_commit(tfull);
                        ++gw;
                    }
                }
            }
            mma_commit(done);
            mbar_wait(done, 0);   // every MMA of this CTA has completed (bounded; also after a failure)
        }
        __syncwarp();
    } else {
    // ---------------- producers / read-back (warps 0-15) ----------------
    const int col = tid >> 3, g8 = tid & 7;   // this thread's column and chunk of a stage
    // read-back: lane quarter warp % 4, columns 16 (warp / 4) .. + 15; accumulator rows r < 64
    // hold the products with s + t = c (top), rows r >= 64 those with s + t = c + 1 (bottom)
    const int irow = (32 * (warp & 3) + lane) & 63, cq = warp >> 2;
    const bool top = (warp & 3) < 2;
    bool bad = false;

    // the stage whose values are in flight: unit u, points p0 .. of lo .. hi, this thread's column
    int u = blockIdx.x, hi = 0, p0 = 0, lo = 0;
    const double* c = nullptr;
    auto set_unit = [&]() {
        if (u >= units) return;
        const int b = u / upi;
        span(u - b * upi, lo, hi);
        p0 = lo;
        c = col < a.KA[b] ? reinterpret_cast<const double*>(a.colsA[(size_t)b * a.ldcols + col]) : nullptr;
    };
    double x[8];
    auto load = [&]() {   // columns >= K are neither read nor cut
        if (u >= units || c == nullptr) return;
        const int pb = p0 + 2 * g8;
        if (p0 + TC_PTS <= hi && ((reinterpret_cast<uintptr_t>(c) & 15u) == 0)) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double2 v = *reinterpret_cast<const double2*>(c + pb + 16 * k);
                x[2 * k] = v.x;
                x[2 * k + 1] = v.y;
            }
            return;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[2 * k] = pb + 16 * k < hi ? c[pb + 16 * k] : 0.0;
            x[2 * k + 1] = pb + 16 * k + 1 < hi ? c[pb + 16 * k + 1] : 0.0;
        }
    };
    // this thread's 16 outputs: exact 96-bit sums over the unit's windows, word w of output j at
    // sv[(3 j + w) TC_PROD + tid]
    int pu = -1, gw = 0;   // unit of the window to read back, windows read back so far
    bool pfirst = false, plast = false;
    auto readback = [&]() {
        if (!bad && !mbar_wait_f(tfull, gw & 1, &s_fail, limit)) bad = true;
        ++gw;
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const unsigned base = tmem + ((unsigned)(32 * (warp & 3)) << 16) + (unsigned)(16 * cq);
#pragma unroll
        for (int j0 = 0; j0 < 16; j0 += 4) {
            int v[TC_TILES][4];
#pragma unroll
            for (int t = 0; t < TC_TILES; ++t) tmem_ld4(base + (unsigned)(t * TC_N + j0), v[t]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                long long h[4];
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    h[t] = (long long)__float2int_rn(__int_as_float(v[2 * t][e])) * 128 +
                           __float2int_rn(__int_as_float(v[2 * t + 1][e]));   // exact integers
                unsigned* v3 = sv + 3 * (j0 + e) * TC_PROD + tid;
                unsigned w[3] = {0u, 0u, 0u};
                if (!pfirst) {
#pragma unroll
                    for (int t = 0; t < 3; ++t) w[t] = v3[t * TC_PROD];
                }
                add96(w, (h[0] << 14) + h[1], (h[2] << 14) + h[3]);
#pragma unroll
                for (int t = 0; t < 3; ++t) v3[t * TC_PROD] = w[t];
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(tempty);   // the tiles may be overwritten
        if (!plast) return;
        // ---- the unit's partial: 2^7 top + bottom (64 rows, two warps on); a chunk rounded once, or,
        // of several units a chunk, the upper triangle in 128-bit integers, row by row
        tc_prod_sync();
        const int b = pu / upi, unit = pu - b * upi;
        const int K = a.KA[b];
        const int mk = a.maxKA;
        const size_t outsz = (size_t)mk * a.maxKB, tri = (size_t)mk * (mk + 1) / 2;
        double* mypart = a.part + ((size_t)b * chunks + unit) * outsz;
        __int128* bexact = reinterpret_cast<__int128*>(a.part) + (size_t)b * upi * tri;
        auto at = [&](int i, int j) { return (size_t)(i * mk - i * (i - 1) / 2 + (j - i)); };
        auto rounded = [&](__int128 S, int i, int j) {
            return i128_to_double(S, col_exp(colmax[(size_t)b * ld + i]) + col_exp(colmax[(size_t)b * ld + j]) - 70);
        };
        if (top && irow < K) {
#pragma unroll 1
            for (int j = 0; j < 16; ++j) {
                const int jj = 16 * cq + j;
                if (jj < irow || jj >= K) continue;
                const unsigned* v = sv + 3 * j * TC_PROD + tid;
                auto word = [&](int o) {
                    return ((__int128)(int)v[2 * TC_PROD + o] << 64) |
                           ((unsigned long long)v[TC_PROD + o] << 32 | v[o]);
                };
                const __int128 S = (word(0) << 7) + word(64);
                if (nsub == 1) mypart[(size_t)irow * a.maxKB + jj] = rounded(S, irow, jj);
                else bexact[unit * tri + at(irow, jj)] = S;
            }
        }
        // the last unit of item b sums the chunk partials in chunk order
        __threadfence();
        tc_prod_sync();
        if (tid == 0) {
            const unsigned ticket = atom_add_acq_rel_u32(a.counter + b, 1u);
            s_last = (ticket == (unsigned)upi - 1u);
        }
        tc_prod_sync();
        if (s_last) {
            __threadfence();
            const double* bpart = a.part + (size_t)b * chunks * outsz;
            double* Gb = a.G + (size_t)b * a.ldG_b;
            for (int o = tid; o < K * K; o += TC_PROD) {
                const int i = o / K, j = o - i * K;
                if (j < i) continue;
                // chunk order (reproducible), loads in batches of 8 independent ones
                const double* src = bpart + (size_t)i * a.maxKB + j;
                double sum = 0.0;
                int cc = 0;
                if (nsub > 1) {   // the same chunk sums
                    const __int128* se = bexact + at(i, j);
                    for (int r = 0; cc < chunks; ++cc) {
                        __int128 S = 0;
                        for (const int r1 = min(upi, (cc + 1) * nsub); r < r1; ++r) S += se[r * tri];
                        sum += rounded(S, i, j);
                    }
                }
                for (; cc + 8 <= chunks; cc += 8) {
                    double v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = src[(size_t)(cc + e) * outsz];
#pragma unroll
                    for (int e = 0; e < 8; ++e) sum += v[e];
                }
                for (; cc < chunks; ++cc) sum += src[(size_t)cc * outsz];
                if (col_bad(colmax[(size_t)b * ld + i]) || col_bad(colmax[(size_t)b * ld + j])) sum = nan("");
                Gb[(size_t)i * a.ldG + j] = sum;
                Gb[(size_t)j * a.ldG + i] = sum;
            }
            if (tid == 0) st_relaxed_u32(a.counter + b, 0u);
        }
        tc_prod_sync();
    };

    set_unit();
    load();
    int gs = 0, ce = 0;
    while (u < units) {
        const int q = gs % TC_NS;
        const bool mine = c != nullptr;
        const int cu = u, rel = p0 - lo, len = hi - lo;   // the stage at hand
        if (rel == 0) ce = col_exp(mine ? colmax[(size_t)(u / upi) * ld + col] : 0ull) + 1020;
        unsigned zl[8], zh[8];
        if (mine) {
#pragma unroll
            for (int k = 0; k < 8; ++k) cut56(x[k], ce, zl[k], zh[k]);
        }
        // the next stage's values travel while this one's digits are stored
        p0 += TC_PTS;
        if (p0 >= hi) {
            u += gridDim.x;
            set_unit();
        }
        load();
        if (!bad && !mbar_wait_f(empty0 + 8u * q, ((gs / TC_NS) & 1) ^ 1, &s_fail, limit)) bad = true;
        if (mine) {
            unsigned char* rowp = smem_raw + q * TC_STAGE_BYTES + col * 128 + ((g8 ^ (col & 7)) << 4);
#define TC_SLICE(S)                                                                                        \
    *reinterpret_cast<uint4*>(rowp + (S) * 8 * TC_SBO) =                                                   \
        make_uint4(digit_pair<7 * (7 - (S))>(zl[0], zh[0], zl[1], zh[1]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[2], zh[2], zl[3], zh[3]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[4], zh[4], zl[5], zh[5]),                                  \
                   digit_pair<7 * (7 - (S))>(zl[6], zh[6], zl[7], zh[7]));
            TC_SLICE(0) TC_SLICE(1) TC_SLICE(2) TC_SLICE(3) TC_SLICE(4) TC_SLICE(5) TC_SLICE(6) TC_SLICE(7)
#undef TC_SLICE
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        mbar_arrive(full0 + 8u * q);
        ++gs;
        // A finished window is read back a stage later, which waits in the ring meanwhile (one
        // set of tiles fills the tensor memory).
        const bool wlast = (rel + TC_PTS) % TC_WIN == 0 || rel + TC_PTS >= len;
        if (pu >= 0) {
            readback();
            pu = -1;
        }
        if (wlast) {
            pu = cu;
            pfirst = rel < TC_WIN;
            plast = rel + TC_PTS >= len;
        }
    }
    if (pu >= 0) readback();
    }
    if (s_fail && tid == 0) record_error(err, DERR_TIMEOUT);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 16) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                     : "memory");
    }
}

int gram_tc_max_cols() { return TC_N; }

cudaError_t launch_gram_tc(const GramArgs& a, unsigned long long* colmax, int ld, int* err, long long spin_limit,
                           cudaStream_t st) {
    if (!a.sym || a.maxKA > TC_N || a.maxKA <= 0 || !colmax || !err || ld < a.maxKA) return cudaErrorInvalidValue;
    if (a.B <= 0) return cudaSuccess;
    // the chunks of the other Gram kernels, so that the partial buffer (gram_part_doubles)
    // fits; any chunk length works for this kernel
    const int chunks = gram_chunks(a.Ng);
    const long long CH = ((a.Ng + chunks - 1) / chunks + TC_PTS - 1) / TC_PTS * TC_PTS;
    cudaError_t e = cudaMemsetAsync(colmax, 0, sizeof(unsigned long long) * (size_t)a.B * ld, st);
    if (e != cudaSuccess) return e;
    colmax_kernel<<<dim3(chunks, a.B), 256, 0, st>>>(a, CH, colmax, ld);
    ++g_launch_count;
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    // Units of about 16384 points, as many as fill whole waves of the grid, but one wave at least
    // (short units pay a read-back, the partials' fences and the last CTA's sum over them: 16
    // windows of 33 columns on 32^3, 791 us in units of 320 points, 230 us in one wave; 16 of 54
    // on 64^3, 2.64 and 1.22 ms)
    auto units = [&](long long items) {
        const long long waves = std::max<long long>(1, items * a.Ng / 16384 / std::max(1, sms));
        return (int)std::min<long long>(chunks, std::max<long long>(1, waves * sms / items));
    };
    if (a.maxKA <= N2_COLS && chunks >= 2) {
        // narrow form: at most one unit for two partial slots of the other Gram kernels, since a
        // unit's partial is K x K 128-bit integers
        const int ctc = std::min(units(a.B), chunks / 2);
        const long long U2 = ((a.Ng + ctc - 1) / ctc + N2_PTS - 1) / N2_PTS * N2_PTS;
        const int chunks2 = (int)((a.Ng + U2 - 1) / U2);
        e = cudaFuncSetAttribute((const void*)gram_tc32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 N2_SMEM);
        if (e != cudaSuccess) return e;
        const int grid2 = std::max(1, std::min(sms, a.B * chunks2));
        gram_tc32_kernel<<<grid2, N2_THREADS, N2_SMEM, st>>>(a, U2, chunks2, colmax, ld, err, spin_limit);
        ++g_launch_count;
        return cudaGetLastError();
    }
    // wide form, one CTA an SM (the tiles take all 512 tensor-memory columns).  It rounds a chunk's
    // sums, and an item's Gram may not depend on how many items share the call: chunks of the context's
    // items.  (Exact sums over an item, rounded at the end, would allow any chunks, but Grams of windows
    // with fewer modes than columns, so rounded, take the Jacobi iteration more sweeps: four windows
    // of 64 on 128^3, 13.8 -> 15.4 ms a POD call.)
    const int cw = units(std::max(1, a.items));
    const int CHw = (int)(((a.Ng + cw - 1) / cw + TC_PTS - 1) / TC_PTS * TC_PTS);
    const int chunksw = (int)((a.Ng + CHw - 1) / CHw);
    // A call of fewer items cuts the chunks into units that stay exact (one window of 54 on 64^3 in a
    // context of 16: 0.97 -> 0.27 ms); their partials are K (K + 1) doubles where the other kernels'
    // are K^2.
    const int most = std::min(units(a.B), (int)((long long)chunks * a.maxKA / (a.maxKA + 1)));
    const int want = std::max(1, most / chunksw);
    const int SH = ((CHw + want - 1) / want + TC_PTS - 1) / TC_PTS * TC_PTS;
    const int nsub = (CHw + SH - 1) / SH;
    e = cudaFuncSetAttribute((const void*)gram_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    if (e != cudaSuccess) return e;
    const int grid = std::max(1, std::min(sms, a.B * chunksw * nsub));
    gram_tc_kernel<<<grid, TC_THREADS, TC_SMEM, st>>>(a, CHw, chunksw, SH, nsub, colmax, ld, err, spin_limit);
    ++g_launch_count;
    return cudaGetLastError();
}

}  // namespace pr
