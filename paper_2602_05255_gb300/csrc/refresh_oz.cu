// From-scratch FP64 inverse with the trailing updates on the tensor cores.
//
// The refresh (Sec. 2.3 init_det_carrier; Sec. 1 advises double precision) is
// a blocked Gauss-Jordan inversion of M = A^T, n^3 FMAs per walker, and
// GB300's FP64 pipe runs at about 1/64 of its FP32 rate.  Panels of OZ_B = 64
// columns are eliminated in four 16-column sub-panels (eight 8-column ones for
// n > 1024): each in FP64 (refresh.cu: n * 16^2 FMAs), its update of the
// panel's other columns as the split product below with one K-step of 16;
// then the update of every other column by the panel,
//     M[i, j] += sum_c (Pan - E)[i, c] * S[c, j],   S = rows k0 .. k0+63 of M,
// (n^2 * 64 FMAs per panel: 94% of the work at n = 1024) also runs as an
// error-free split product on the BF16 tensor cores, the scheme of Ozaki,
// Ogita, Oishi and Rump (Numer. Algorithms 59, 2012):
//   - every 64-vector (a row of Pan - E, a column of S) is scaled by a power
//     of two 2^E with |x| < 2^E and rounded to a multiple of 2^(E-56), then
//     written exactly as 7 signed base-256 digits, x = 2^E sum_t d_t 2^(-8(t+1))
//     (|d_0| <= 256, |d_t| <= 128), each digit times its power a BF16 value;
//     this uses integer operations only;
//   - the product of digit t of S and digit u of Pan has level l = t + u + 2:
//     an integer times 2^(-8l).  Summed over the 64-wide inner dimension, all
//     products of one level stay below 2^23 in magnitude, so the FP32
//     accumulation of tcgen05.mma is exact for each of the levels 2 .. 6,
//     each in its own TMEM accumulator; levels 7..10 (below 2^(-40) of level
//     2, summed with FP32 rounding) share a sixth; levels above 10 (below
//     2^(-66) of the scale) are dropped.  Levels 7..10 are kept because the
//     row scaling measures errors against the row maxima: a level dropped at
//     2^-56 of the maxima of two rows whose large entries do not meet costs
//     far more than 2^-53 of the products actually summed;
//   - the epilogue recovers the five exact levels as integers, rounds the
//     tail to a multiple of 2^-56, adds all six exactly in int64, converts
//     once to double with the scale 2^(E_i + E_j) folded into the exponent
//     (integer operations), and adds it to M: one FP64 add per element, and
//     the rounding of an FP64 update, at tensor-core speed.
// The output tile is 128 columns j (TMEM lanes, so the FP64 read-modify-write
// of row-major M is coalesced) x 64 rows i; TMA stages the 7 S slices of a
// column block once (112 KiB) and the 7 Pan slices of each row tile (two stages
// of 56 KiB; SWIZZLE_128B, no multicast).  Every wait is bounded as in the
// delayed flush.  (At 32 rows, where two full accumulator sets fit, the MMAs,
// whose operands are re-read from shared memory per instruction, become the
// bound.)
#include <algorithm>
#include <cuda.h>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "tcgen05.cuh"

namespace lru {

constexpr int OZ_TJ = 128;                        // output columns j per tile (MMA M)
constexpr int OZ_TI = 64;                         // output rows i per tile (MMA N)
constexpr int OZ_SLICE_A = OZ_TJ * 128;           // bytes of one S slice tile (128 rows x 128 B)
constexpr int OZ_SLICE_B = OZ_TI * 128;           // bytes of one Pan slice tile (64 rows x 128 B)
constexpr int OZ_GROUPS = 6;                      // accumulators: levels 2, 3, 4, 5, 6 (exact), 7..10
constexpr int OZ_MAXLV = 8;                       // products t + u <= 8 (levels up to 10) are kept
constexpr uint32_t OZ_TMEM_COLS = 512;            // 6 x 64 columns, rounded to a power of two
constexpr uint32_t OZ_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(OZ_TI >> 3) << 17) |
                              ((uint32_t)(OZ_TJ >> 4) << 24);   // BF16 x BF16 -> F32, K-major, 128 x 64

struct OzMaps {
    CUtensorMap S, P;
};

// ---- exact splitting (integer operations only) --------------------------------

__device__ __forceinline__ int oz_bexp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

// X = round(x * 2^(56 - E)) for |x| < 2^E: |X| < 2^56.  Zero and subnormal x give 0.
__device__ __forceinline__ long long oz_fixed(double x, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int eb = (int)((b >> 52) & 0x7FF);
    if (eb == 0) return 0;
    const long long m = (long long)((b & 0xFFFFFFFFFFFFFull) | (1ull << 52));
    const int sh = eb - 1075 + 56 - E;   // <= 3 because |x| < 2^E
    long long X;
    if (sh >= 0) X = m << sh;
    else if (sh > -60) X = (m + (1ll << (-sh - 1))) >> (-sh);
    else X = 0;
    return (b >> 63) ? -X : X;
}

// digit t of X (signed, rounded): X = sum_t d_t 2^(48 - 8t); BF16 bits of d_t * 2^(-8(t+1))
__device__ __forceinline__ void oz_digits(long long X, uint16_t (&h)[OZ_S]) {
#pragma unroll
    for (int t = 0; t < OZ_S; ++t) {
        const int sh = 48 - 8 * t;
        const long long q = sh > 0 ? ((X + (1ll << (sh - 1))) >> sh) : X;
        X -= q << sh;
        // |q| <= 256: exact in FP32 via the 1.5 * 2^23 offset, exact in BF16 (8 significant bits)
        const float f = (__int_as_float(0x4B400000 + (int)q) - 12582912.0f) * __int_as_float((127 - 8 * (t + 1)) << 23);
        h[t] = (uint16_t)(__float_as_uint(f) >> 16);
    }
}

// A walker's working matrix M has nr rows of nc doubles: nc = nr for real
// scalars and 2 nr for complex ones (CX = 2: re, im interleaved).  A complex
// update sum_c p_c s_c is two real ones of the interleaved row (re p, im p):
// against (re s, -im s) for the real part, (im s, re s) for the imaginary one.
// So the panel rows are sliced as they lie, the S columns twice, and the same
// 64-wide products serve 64 real or 32 complex panel columns.

// Rows of (Pan - E) from row i_lo: the width (<= 64) doubles c0 .. of M's row i,
// minus 1 at the diagonal; columns past the width are zero.  One warp per row;
// lane covers c = lane and lane + 32.
__global__ void __launch_bounds__(256) k_oz_slice_P(int nr, int nc, int cx, int i_lo, int c0, int width, OzWork Z,
                                                    const uint8_t* mask) {
    const int w = blockIdx.y;
    if (mask && !mask[w]) return;
    const int lane = threadIdx.x & 31;
    const int i = i_lo + blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= nr) return;
    const double* row = Z.M + (long long)w * nr * nc + (long long)i * nc + c0;
    double a = lane < width ? row[lane] : 0.0, b = lane + 32 < width ? row[lane + 32] : 0.0;
    if (lane < width && i * cx == c0 + lane) a -= 1.0;
    if (lane + 32 < width && i * cx == c0 + lane + 32) b -= 1.0;
    const int mx = __reduce_max_sync(0xffffffffu, max(oz_bexp(a), oz_bexp(b)));
    const int E = mx > 0 ? mx - 1022 : 0;
    uint16_t ha[OZ_S], hb[OZ_S];
    oz_digits(oz_fixed(a, E), ha);
    oz_digits(oz_fixed(b, E), hb);
#pragma unroll
    for (int t = 0; t < OZ_S; ++t) {
        uint16_t* dst = Z.Pb + (((long long)w * OZ_S + t) * nr + i) * OZ_B;
        dst[lane] = ha[t];
        dst[lane + 32] = hb[t];
    }
    if (lane == 0) Z.eP[(long long)w * nr + i] = E;
}

// The same rows for a sub-panel (16 doubles or fewer): half a warp per row, lane c
// of the half covering column c, so no lane splits a zero.  Such a width feeds a
// single K-step of 16, which reads only the first 16 columns of each slice row,
// so only those are written.  nr - i_lo is a multiple of 16.
__global__ void __launch_bounds__(256) k_oz_slice_P16(int nr, int nc, int cx, int i_lo, int c0, int width, OzWork Z,
                                                      const uint8_t* mask) {
    const int w = blockIdx.y;
    if (mask && !mask[w]) return;
    const int c = threadIdx.x & 15;
    const int i = i_lo + blockIdx.x * 16 + (threadIdx.x >> 4);
    const unsigned hmask = 0xFFFFu << (threadIdx.x & 16);   // this half of the warp
    const bool ok = i < nr;
    const double* row = Z.M + (long long)w * nr * nc + (long long)i * nc + c0;
    double a = (ok && c < width) ? row[c] : 0.0;
    if (c < width && i * cx == c0 + c) a -= 1.0;
    int mx = oz_bexp(a);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(hmask, mx, o));
    const int E = mx > 0 ? mx - 1022 : 0;
    uint16_t ha[OZ_S];
    oz_digits(oz_fixed(a, E), ha);
    if (!ok) return;
#pragma unroll
    for (int t = 0; t < OZ_S; ++t) Z.Pb[(((long long)w * OZ_S + t) * nr + i) * OZ_B + c] = ha[t];
    if (c == 0) Z.eP[(long long)w * nr + i] = E;
}

// Columns of S = the rows r0 .. r0 + rows - 1 of M (rows * CX <= 64), zero past
// them: 64 doubles of each row per CTA (column blocks jb0, jb0 + 1, ..) through
// shared memory (stored transposed), then one warp per real column j.  At most
// 16 doubles write only the first 16 entries of each slice row.
template <int CX>
__global__ void __launch_bounds__(256) k_oz_slice_S(int nr, int nc, int r0, int rows, int jb0, OzWork Z,
                                                    const uint8_t* mask) {
    __shared__ double sT[64][65];   // sT[j][c] = S[c][j0 + j]
    const int w = blockIdx.y;
    if (mask && !mask[w]) return;
    const int j0 = (jb0 + blockIdx.x) * 64, width = rows * CX;
    if (j0 >= nc) return;
    const double* M = Z.M + (long long)w * nr * nc;
    for (int e = threadIdx.x; e < 64 * 64 / CX; e += 256) {
        const int c = e >> 6, j = e & 63;
        const double v = c < rows ? M[(long long)(r0 + c) * nc + j0 + j] : 0.0;
        if constexpr (CX == 1) {
            sT[j][c] = v;
        } else {
            sT[j][2 * c] = v;                              // re: (re s, .); im: (im s, .)
            sT[j ^ 1][2 * c + 1] = (j & 1) ? -v : v;       // (., -im s) and (., re s)
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < 64; j += 8) {
        const double a = sT[j][lane], b = sT[j][lane + 32];
        const int mx = __reduce_max_sync(0xffffffffu, max(oz_bexp(a), oz_bexp(b)));
        const int E = mx > 0 ? mx - 1022 : 0;
        uint16_t ha[OZ_S], hb[OZ_S];
        oz_digits(oz_fixed(a, E), ha);
        oz_digits(oz_fixed(b, E), hb);
#pragma unroll
        for (int t = 0; t < OZ_S; ++t) {
            uint16_t* dst = Z.Sb + (((long long)w * OZ_S + t) * nc + j0 + j) * OZ_B;
            if (width > 16 || lane < 16) dst[lane] = ha[t];
            if (width > 16) dst[lane + 32] = hb[t];
        }
        if (lane == 0) Z.eS[(long long)w * nc + j0 + j] = E;
    }
}

__device__ __forceinline__ void oz_mma(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t acc) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(dtmem), "l"(a), "l"(b), "r"(OZ_IDESC), "r"(acc)
        : "memory");
}

// Levels 2 .. 6 of one element are integers N_l 2^(-8l), |N_l| < 2^23 (a float holds
// them exactly), and the tail (levels 7 .. 10) is rounded to a multiple of 2^-56:
// their sum F in units of 2^-56, |F| < 2^62, exactly, as two words.  A level that
// stays within 2^22 comes out of the mantissa of x * scale + 1.5 * 2^23, which
// holds no more: N_2 and N_3 always, the tail of a single K-step (below 2^21 +
// 2^14).  N_4 .. N_6 and the tail of more (up to 2^23 + 2^16 at 64) take the
// conversion unit.
__device__ __forceinline__ void oz_sum2(float a2, float a3, int& hi) {
    constexpr float magic = 12582912.0f;
    const int n2 = __float_as_int(__fmaf_rn(a2, 65536.0f, magic)), n3 = __float_as_int(__fmaf_rn(a3, 16777216.0f, magic));
    hi = n2 * 256 + n3 - (int)(0x4B400000u * 257u);
}
__device__ __forceinline__ void oz_sum4(float a4, float a5, int& hi, uint32_t& lo) {
    const int b = __float2int_rn(a4 * 4294967296.0f) * 256 + __float2int_rn(a5 * 1099511627776.0f);
    lo = (uint32_t)b << 16;
    hi += b >> 16;
}
template <bool ONE_STEP>
__device__ __forceinline__ void oz_sum6(float a6, float tail, int& hi, uint32_t& lo) {
    constexpr float unit = 72057594037927936.0f;   // 2^56
    const int t = ONE_STEP ? __float_as_int(__fmaf_rn(tail, unit, 12582912.0f)) - 0x4B400000 : __float2int_rn(tail * unit);
    const int c = __float2int_rn(a6 * 281474976710656.0f) * 256 + t;
    const uint32_t l = lo + (uint32_t)c;
    hi += (c >> 31) + (l < lo ? 1 : 0);
    lo = l;
}

// F * 2^(e - 56) as a double, rounded to nearest even (products of 53-bit values have
// many ties), by integer operations
// (results below the normal range become zero; the callers keep away from the upper end).  The
// mantissa with its leading one is added to the exponent field less one, so a
// rounding that carries out of it needs no case of its own.
__device__ __forceinline__ double oz_to_double(int hi, uint32_t lo, int e) {
    const int s = hi >> 31;
    const unsigned long long F = ((unsigned long long)(uint32_t)hi << 32) | lo;
    const unsigned long long sx = ((unsigned long long)(uint32_t)s << 32) | (uint32_t)s;
    const unsigned long long a = (F ^ sx) - sx;   // |F|
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
    const int lz = __clz((int)(ah ? ah : al)) + (ah ? 0 : 32);
    const unsigned long long v = a << ((lz - 1) & 63);           // leading one at bit 62 (|F| < 2^63)
    const unsigned long long mant = (v + (0x1FFu + ((uint32_t)(v >> 10) & 1u))) >> 10;
    const uint32_t rh = (uint32_t)(mant >> 32) + ((uint32_t)(1029 + e - lz) << 20);
    const bool nz = a != 0 && 1029 + e - lz > 0;   // below the normal range: zero
    return __hiloint2double(nz ? (int)(rh | ((uint32_t)s & 0x80000000u)) : 0, nz ? (int)(uint32_t)mant : 0);
}

// M[i][j] += 2^(E_i + E_j) sum_c Pan[i][c] S[c][j] as a split product, with
// NKS K-steps of 16 (4 for a 64-column panel, 1 for a sub-panel or the K = 16
// flush), written only for the columns cols selects.  Persistent CTAs take
// (walker, 128-column block) units: the 7 S slices of the block are loaded
// once, then the 64-row tiles i stream through.
//
// Run one after the other, the MMAs of a tile (with the wait for its slices) took
// 36 ms and its epilogue 32 ms of the 66 ms that the trailing updates of a refresh
// of 512 walkers, n = 1024 cost.  So the roles are split over warps: one thread
// loads (two stages of Pan slices), one issues MMAs, 16 warps run the epilogue of
// tile T while the MMAs of tile T + 1 run.  Two sets of six accumulators do not fit
// the 512 TMEM columns; but 29 of the 39 slice products go to two of the six
// accumulators (level 6, and the levels 7 .. 10 together), and two sets of those
// fit beside one of the levels 2 .. 5.  The MMA thread does these 29 first and only
// then waits for the epilogue to have read levels 2 .. 5 of the tile before, which
// it does at once, into 64-bit sums in registers: 66 -> 46 ms (the sub-panel
// products 27 -> 20 ms, the K = 16 flush of 1024 walkers 5.7 -> 4.9 ms).  A full
// overlap would end at the 36 ms of the MMAs.
constexpr int OZ_EPI_WARPS = 16;  // 4 per TMEM lane quarter, each 16 of the 64 rows i
constexpr int OZ_THREADS = 32 * (OZ_EPI_WARPS + 2);
constexpr size_t OZ_GEMM_SMEM = 1024 + (size_t)OZ_S * (OZ_SLICE_A + 2 * OZ_SLICE_B);

// accumulator g (level g + 2; 5: the tail) of tile T
__device__ __forceinline__ uint32_t oz_acc(uint32_t tmem, int g, uint32_t T) {
    return tmem + 64u * (g < 4 ? (uint32_t)g : 4u + 2u * (uint32_t)(g - 4) + (T & 1u));
}

// bounded wait that also ends when another role has given up
__device__ __forceinline__ bool oz_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
    for (int i = 0; i < (1 << 20); ++i) {
        if (mbar_try(bar, parity)) return true;
        if (i > 64) {
            __nanosleep(256);
            if (*abort) return false;
        }
    }
    return false;
}

// the products of tile T for accumulators g_lo .. g_hi - 1
template <int NKS, int G_LO, int G_HI>
__device__ __forceinline__ void oz_issue(uint32_t tmem, uint32_t T, uint64_t a0, uint64_t b0) {
    // fully unrolled: descriptor offsets and accumulate flags are compile-time, so
    // the issuing thread streams back-to-back MMAs
    uint32_t started = 0;   // bit g: accumulator g holds a partial sum
#pragma unroll
    for (int t = 0; t < OZ_S; ++t)
#pragma unroll
        for (int u = 0; u < OZ_S; ++u) {
            const int g = t + u < OZ_GROUPS - 1 ? t + u : OZ_GROUPS - 1;   // level t+u+2: 2 .. 6, then 7..10
            if (u + t > OZ_MAXLV || g < G_LO || g >= G_HI) continue;
            const uint64_t a = a0 + (uint64_t)((t * OZ_SLICE_A) >> 4), b = b0 + (uint64_t)((u * OZ_SLICE_B) >> 4);
#pragma unroll
            for (int ks = 0; ks < NKS; ++ks) {
                const uint64_t adv = (uint64_t)(ks * 32) >> 4;   // 16 BF16 along K per MMA
                oz_mma(oz_acc(tmem, g, T), a + adv, b + adv, (started >> g) & 1u);
                started |= 1u << g;
            }
        }
}

template <int NKS, bool EDGE>   // EDGE: M has fewer rows than the slices (a flush with n % 64 != 0)
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(const __grid_constant__ OzMaps maps, int W, int nr, int nc, OzCols cols, OzWork Z,
              const uint8_t* mask, int* err) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* sm = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    unsigned char* sA = sm;                               // OZ_S slices of S, 128 rows each
    unsigned char* sB = sA + OZ_S * OZ_SLICE_A;           // two stages of OZ_S slices of Pan, 64 rows each
    constexpr uint32_t STAGE = (uint32_t)OZ_S * OZ_SLICE_B;
    __shared__ __align__(8) unsigned long long mbar[8];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const uint32_t m_sfull = smem_u32(&mbar[0]);          // S slices of a unit have landed
    const uint32_t m_pfull = smem_u32(&mbar[1]);          // [2] Pan slices of a tile have landed
    const uint32_t m_pfree = smem_u32(&mbar[3]);          // [2] the MMAs of a stage's tile are done
    const uint32_t m_full = smem_u32(&mbar[5]);           // the accumulators of a tile are complete
    const uint32_t m_free = smem_u32(&mbar[6]);           // the epilogue warps have read them
    const uint32_t m_drain = smem_u32(&mbar[7]);          // (giving up) MMAs in flight are done
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(OZ_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < 8; ++i) mbar_init(smem_u32(&mbar[i]), i == 6 ? OZ_EPI_WARPS : 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_abort = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const uint32_t bytes_a = (uint32_t)OZ_S * OZ_SLICE_A, bytes_b = STAGE;
    const int ntj = cols.jt_hi - cols.jt_lo, nti = nr / OZ_TI;
    const int rs = cols.rsplit, ntr = nti - cols.it_lo;   // row tiles of a unit: an rs-th of the block's
    const long long units = (long long)W * ntj * rs;
    auto walker = [&](long long un) { return (int)(un / (ntj * rs)); };
    auto block = [&](long long un) { return (cols.jt_lo + (int)(un % ntj)) * OZ_TJ; };
    auto first = [&](long long un) { return cols.it_lo + (int)(un / ntj % rs) * ntr / rs; };
    auto past = [&](long long un) { return cols.it_lo + ((int)(un / ntj % rs) + 1) * ntr / rs; };
    uint32_t T = 0, U = 0;   // tiles and units done; every role walks the same ones
    auto give_up = [&]() {
        set_dev_error(err, DEV_ERR_TIMEOUT);
        s_abort = 1;
    };
    if (warp == OZ_EPI_WARPS) {
        // ---- loads; the other lanes prefetch the tile's M into L2, two tiles
        //      ahead of the epilogue that reads it (registers for a second set of
        //      M values, and shared memory for one, are not to be had; 0.3% of a refresh
        //      of 512 walkers, n = 1024, 0.9% of a Pfaffian sweep) ----
        bool ok = true;
        for (long long un = blockIdx.x; un < units && ok; un += gridDim.x) {
            const int w = walker(un);
            if (mask && !mask[w]) continue;
            const int j0 = block(un), end = past(un);
            const int p0 = max(j0, cols.c_lo), p1 = min(j0 + OZ_TJ, cols.c_hi);   // multiples of 64
            const double* Mp = Z.M + (long long)w * cols.rows * cols.ld + p0;
            // rows past the walker's last column (a 128-wide tile at nc % 128 == 64) are
            // the next slice's or zero, and their products are not kept
            const int ys = (int)((long long)w * OZ_S * nc) + j0;
            const int yp = (int)((long long)w * OZ_S * nr);
            if (lane == 0) {
                if (T > 0) ok = oz_wait(m_pfree + 8 * ((T - 1) & 1), ((T - 1) >> 1) & 1, &s_abort);   // the last unit's MMAs
                if (ok) {
                    mbar_expect_tx(m_sfull, bytes_a);
                    for (int t = 0; t < OZ_S; ++t)
                        tma_load_2d(smem_u32(sA + t * OZ_SLICE_A), &maps.S, 0, ys + t * nc, m_sfull);
                    ++U;
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            for (int it = first(un); it < end && ok; ++it) {
                if (lane == 0) {
                    const uint32_t st = T & 1;
                    if (T >= 2) ok = oz_wait(m_pfree + 8 * st, ((T - 2) >> 1) & 1, &s_abort);
                    if (ok) {
                        mbar_expect_tx(m_pfull + 8 * st, bytes_b);
                        for (int t = 0; t < OZ_S; ++t)
                            tma_load_2d(smem_u32(sB + st * STAGE + t * OZ_SLICE_B), &maps.P, 0,
                                        yp + t * nr + it * OZ_TI, m_pfull + 8 * st);
                        ++T;
                    }
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (ok && p1 > p0 && ((cols.ld | p1) & 1) == 0)   // 16-byte rows
                    for (int r = it * OZ_TI + lane; r < min(it * OZ_TI + OZ_TI, cols.rows); r += 32)
                        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(Mp + (long long)r * cols.ld),
                                     "r"((uint32_t)(p1 - p0) * 8u)
                                     : "memory");
            }
        }
        if (lane == 0) {
            if (!ok) give_up();
            // let copies in flight land before leaving, also when it is another role
            // that has given up and does not wait for them
            if (U > 0) mbar_wait(m_sfull, (U - 1) & 1);
            if (T >= 1) mbar_wait(m_pfull + 8 * ((T - 1) & 1), ((T - 1) >> 1) & 1);
            if (T >= 2) mbar_wait(m_pfull + 8 * (T & 1), ((T - 2) >> 1) & 1);
        }
    } else if (warp == OZ_EPI_WARPS + 1) {
        // ---- MMAs ----
        const uint64_t a0 = desc_sw128(smem_u32(sA));
        bool ok = true;
        for (long long un = blockIdx.x; un < units && ok && lane == 0; un += gridDim.x) {
            if (mask && !mask[walker(un)]) continue;
            ok = oz_wait(m_sfull, U & 1, &s_abort);
            ++U;
            const int tiles = past(un) - first(un);
            for (int it = 0; it < tiles && ok; ++it, ++T) {
                const uint32_t st = T & 1;
                ok = oz_wait(m_pfull + 8 * st, (T >> 1) & 1, &s_abort);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint64_t b0 = desc_sw128(smem_u32(sB + st * STAGE));
                oz_issue<NKS, 4, 6>(tmem, T, a0, b0);
                if (T > 0) ok = oz_wait(m_free, (T - 1) & 1, &s_abort);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                oz_issue<NKS, 0, 4>(tmem, T, a0, b0);
                mma_commit(m_pfree + 8 * st);
                mma_commit(m_full);
            }
        }
        // MMAs in flight end before the TMEM goes back, whichever role gave up
        if (lane == 0) {
            if (!ok) {
                give_up();
                mma_commit(m_drain);
                mbar_wait(m_drain, 0);
            } else if (T > 0) {
                mbar_wait(m_full, (T - 1) & 1);
            }
        }
    } else {
        // ---- epilogue: warp q reads TMEM lanes 32 (q % 4) .. +31 (columns j) and
        //      rows i0 + 16 (q / 4) .. +15 ----
        const int quad = warp & 3, part = warp >> 2;
        const uint32_t lanes = (uint32_t)(32 * quad) << 16;
        bool ok = true;
        for (long long un = blockIdx.x; un < units && ok; un += gridDim.x) {
            const int w = walker(un), end = past(un);
            if (mask && !mask[w]) continue;
            const int j = block(un) + 32 * quad + lane;   // this thread's column
            const bool keep = j >= cols.c_lo && j < cols.c_hi && !(j >= cols.s_lo && j < cols.s_hi);
            const bool wact = __any_sync(0xffffffffu, keep);   // a warp with no column to write only keeps step
            const int eSj = j < nc ? Z.eS[(long long)w * nc + j] : 0;
            for (int it = first(un); it < end; ++it, ++T) {
                const int i0 = it * OZ_TI + 16 * part;
                double* Mj = Z.M + ((long long)w * cols.rows + i0) * cols.ld + j;
                // this thread writes row c
                auto mine = [&](int c) { return EDGE ? keep && i0 + c < cols.rows : keep; };
                const int* eP = Z.eP + (long long)w * nr + i0;
                // this thread's 16 values of M: the loads overlap the MMAs
                double m[16];
#pragma unroll
                for (int c = 0; c < 16; ++c) m[c] = mine(c) ? Mj[(long long)c * cols.ld] : 0.0;
                // the lanes leave together: the TMEM loads below take the whole warp
                ok = __all_sync(0xffffffffu, oz_wait(m_full, T & 1, &s_abort));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                // the six accumulators into one exact sum per element, then the
                // accumulators are free
                int fh[16];
                uint32_t fl[16];
                if (wact) {
#pragma unroll
                    for (int ch = 0; ch < 2; ++ch) {
                        float x[8], y[8];
                        const uint32_t c0 = (uint32_t)(16 * part + 8 * ch);
                        tmem_ld8(oz_acc(tmem, 0, T) + lanes + c0, x);
                        tmem_ld8(oz_acc(tmem, 1, T) + lanes + c0, y);
#pragma unroll
                        for (int c = 0; c < 8; ++c) oz_sum2(x[c], y[c], fh[8 * ch + c]);
                        tmem_ld8(oz_acc(tmem, 2, T) + lanes + c0, x);
                        tmem_ld8(oz_acc(tmem, 3, T) + lanes + c0, y);
#pragma unroll
                        for (int c = 0; c < 8; ++c) oz_sum4(x[c], y[c], fh[8 * ch + c], fl[8 * ch + c]);
                        tmem_ld8(oz_acc(tmem, 4, T) + lanes + c0, x);
                        tmem_ld8(oz_acc(tmem, 5, T) + lanes + c0, y);
#pragma unroll
                        for (int c = 0; c < 8; ++c) oz_sum6<NKS == 1>(x[c], y[c], fh[8 * ch + c], fl[8 * ch + c]);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(m_free);
                if (wact) {
#pragma unroll
                    for (int c = 0; c < 16; ++c) {
                        const double d = oz_to_double(fh[c], fl[c], eP[c] + eSj);
                        if (mine(c)) Mj[(long long)c * cols.ld] = m[c] + d;
                    }
                }
            }
        }
        if (!ok && lane == 0) give_up();
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS)
                     : "memory");
    }
}

// ---- the delayed flush as a split product ------------------------------------

// Everything before the product, one CTA per walker that flushes (persistent
// over walkers; on a step where none does every block leaves after reading tau):
//   - the flush flag Z.go;
//   - the column balance.  Every row is written as digits of one power-of-two
//     scale (its largest entry), so a slot column much larger than the others (the
//     step of a near-node update) would cost the other entries of the row their low
//     bits.  Column c of P is scaled by 2^s_c and column c of Q by 2^-s_c, with s_c
//     half the exponent gap of the two columns' maxima: P Q^T is unchanged exactly,
//     and the entries of a row span a far smaller range;
//   - the slices and exponents of the rows of P (complex: two rows each, see
//     k_oz_slice_S) and of sgnQ Q, the cu columns of the tau filled slots (of the
//     walker's own rank each, kv; the row stride is the handle's rank's), zeros after.
// A walker with slots above 2^480, where a product of scales could leave the
// exponent range, is folded here in FP64 instead and not flagged.
// One launch in place of four (flags, balance, two slicings): a step without a
// flush costs one launch less than the time of three.
__device__ __forceinline__ double oz_pow2(int k) { return __hiloint2double((1023 + k) << 20, 0); }

template <typename T>
__global__ void __launch_bounds__(256) k_oz_flush_slices(int W, int n, int nr, int K, int kk, const int* kv, const T* P,
                                                         const T* Q, double sgnQ, const int* tau, const uint8_t* force,
                                                         OzWork Z) {
    constexpr int CX = traits<T>::is_complex ? 2 : 1;
    __shared__ int sp[4][OZ_B], sq[4][OZ_B], s_big;
    __shared__ double s_fp[OZ_B], s_fq[OZ_B];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int c = threadIdx.x % OZ_B, g = threadIdx.x / OZ_B;   // 64 columns x 4 row groups
    const int ldx = K * kk * CX, nc = nr * CX;
    for (int w = blockIdx.x; w < W; w += gridDim.x) {
        const int t = tau[w];
        const bool due = force ? (force[w] && t > 0) : t >= K;
        if (threadIdx.x == 0) {
            Z.go[w] = due ? 1 : 0;
            s_big = 0;
        }
        if (!due) continue;
        const int slots = t * (kv ? kv[w] : kk), cu = slots * CX;   // filled columns, and their doubles
        const double* Pw = reinterpret_cast<const double*>(P) + (long long)w * n * ldx;
        const double* Qw = reinterpret_cast<const double*>(Q) + (long long)w * n * ldx;
        int ep = 0, eq = 0;
        if (c < cu)
#pragma unroll 4
            for (int r = g; r < n; r += 4) {
                ep = max(ep, oz_bexp(Pw[(long long)r * ldx + c]));
                eq = max(eq, oz_bexp(Qw[(long long)r * ldx + c]));
            }
        __syncthreads();
        sp[g][c] = ep;
        sq[g][c] = eq;
        __syncthreads();
        if (g == 0) {
            ep = eq = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int x = 0; x < CX; ++x) {   // both parts of a complex column share its scale
                    ep = max(ep, sp[q][c ^ x]);
                    eq = max(eq, sq[q][c ^ x]);
                }
            const int cs = (ep > 0 && eq > 0) ? (eq - ep) / 2 : 0;
            s_fp[c] = c < cu ? oz_pow2(cs) : 0.0;
            s_fq[c] = c < cu ? sgnQ * oz_pow2(-cs) : 0.0;
            if (max(ep, eq) > 1023 + 480) s_big = 1;
        }
        __syncthreads();
        if (s_big) {
            T* G = reinterpret_cast<T*>(Z.M) + (long long)w * n * n;
            for (long long e = threadIdx.x; e < (long long)n * n; e += 256) {
                const int l = (int)(e / n), j = (int)(e - (long long)l * n);
                T d = s_zero(T());
                for (int q = 0; q < slots; ++q)
                    d = s_fma(P[((long long)w * n + j) * K * kk + q], Q[((long long)w * n + l) * K * kk + q], d);
                G[e] = sgnQ < 0 ? G[e] - d : G[e] + d;
            }
            if (threadIdx.x == 0) Z.go[w] = 0;
            __syncthreads();
            continue;
        }
        const double pa = s_fp[lane], pb = s_fp[lane + 32], qa = s_fq[lane], qb = s_fq[lane + 32];
        const bool second = ldx > 32;
        for (int r = wid; r < 2 * n; r += 8) {
            const bool isq = r >= n;
            const int i = isq ? r - n : r;
            const double* row = (isq ? Qw : Pw) + (long long)i * ldx;
            double a = lane < cu ? (isq ? qa : pa) * row[lane] : 0.0;
            double b = lane + 32 < cu ? (isq ? qb : pb) * row[lane + 32] : 0.0;
            const int mx = __reduce_max_sync(0xffffffffu, max(oz_bexp(a), oz_bexp(b)));
            const int E = mx > 0 ? mx - 1022 : 0;
            const int outs = CX == 2 && !isq ? 2 : 1;
            for (int o = 0; o < outs; ++o) {
                if (CX == 2 && !isq) {
                    if (o == 0) {
                        if (lane & 1) { a = -a; b = -b; }            // (re, -im)
                    } else {
                        if (lane & 1) { a = -a; b = -b; }
                        a = __shfl_xor_sync(0xffffffffu, a, 1);      // (im, re)
                        b = __shfl_xor_sync(0xffffffffu, b, 1);
                    }
                }
                const int ro = isq ? i : i * CX + o, rows = isq ? nr : nc;
                uint16_t* plane = (isq ? Z.Pb : Z.Sb) + (long long)w * OZ_S * rows * OZ_B;
                uint16_t ha[OZ_S], hb[OZ_S];
                oz_digits(oz_fixed(a, E), ha);
                if (second) oz_digits(oz_fixed(b, E), hb);
#pragma unroll
                for (int q = 0; q < OZ_S; ++q) {
                    uint16_t* d = plane + ((long long)q * rows + ro) * OZ_B;
                    d[lane] = ha[q];
                    if (second) d[lane + 32] = hb[q];
                }
                if (lane == 0) (isq ? Z.eP : Z.eS)[(long long)w * rows + ro] = E;
            }
        }
    }
}

// ---- host side ----------------------------------------------------------------

int oz_rows(int n) { return n <= 1024 ? (n + 63) / 64 * 64 : (n + 127) / 128 * 128; }

size_t oz_work_layout(OzWork* Z, void* base, int W, int nr, int cx, bool with_M) {
    const size_t Wr = (size_t)W * nr, Wc = Wr * cx;
    size_t off = 0;
    auto take = [&](size_t x) {
        unsigned char* q = base ? (unsigned char*)base + off : nullptr;
        off += (x + 255) / 256 * 256;
        return q;
    };
    OzWork z{};
    z.perm = (int*)take(Wr * sizeof(int));
    z.sing = (int*)take((size_t)W * sizeof(int));
    z.Sb = (uint16_t*)take(Wc * OZ_S * OZ_B * sizeof(uint16_t));
    z.Pb = (uint16_t*)take(Wr * OZ_S * OZ_B * sizeof(uint16_t));
    z.eS = (int*)take(Wc * sizeof(int));
    z.eP = (int*)take(Wr * sizeof(int));
    z.go = (uint8_t*)take((size_t)W);
    z.odd = (uint8_t*)take((size_t)W);
    z.piv = (double*)take(Wc * sizeof(double));
    z.rmax = (int*)take(Wr * sizeof(int));
    if (with_M) z.M = (double*)take(Wr * nr * cx * sizeof(double));
    if (Z) *Z = z;
    return off;
}

// rows x 64 BF16 matrix, box 64 x box_rows, SWIZZLE_128B
static bool oz_map(CUtensorMap* m, const void* base, long long rows, int box_rows) {
    EncodeTiled enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)OZ_B, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)OZ_B * 2};
    cuuint32_t box[2] = {(cuuint32_t)OZ_B, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Parts into which the row tiles of a column block are cut: few blocks (the
// sub-panel products have one per walker) leave SMs idle or a last wave nearly
// empty; a part loads the block's S slices again (about 2 us), so it keeps four
// tiles (about 6 us each) or more.  Sub-panel products of a refresh of 512 walkers,
// n = 1024: 20.5 -> 17.8 ms.
static int oz_rsplit(int blocks, int tiles, int nsm) {
    int rs = 1;
    while (blocks * rs < 6 * nsm && tiles / (2 * rs) >= 4) rs *= 2;
    return rs;
}

// Gauss-Jordan elimination of the W matrices Z.M (nr rows, nr % 64 == 0 up to
// 1024, % 128 above) of the walkers with mask[w] (NULL: all): the row exchanges
// stay in Z.perm, the pivots in Z.piv.  lu: rows above a panel and columns left
// of it are left alone (a third of the work), enough for the determinant.
template <typename T>
bool oz_eliminate(int W, int nr, const OzWork& Z, const uint8_t* mask, bool lu, int* err, cudaStream_t st,
                  void (*hook)(void*, int, int), void* hctx) {
    constexpr int CX = traits<T>::is_complex ? 2 : 1, PB = OZ_B / CX;
    const int nc = nr * CX;
    const long long rows = (long long)W * OZ_S * nc;
    if (rows >= (1ll << 31) || W > 65535) return false;
    OzMaps maps;
    if (!oz_map(&maps.S, Z.Sb, rows, OZ_TJ) || !oz_map(&maps.P, Z.Pb, (long long)W * OZ_S * nr, OZ_TI)) return false;
    const size_t dyn = OZ_GEMM_SMEM;
    if (cudaFuncSetAttribute(k_oz_gemm<OZ_B / 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) !=
            cudaSuccess ||
        cudaFuncSetAttribute(k_oz_gemm<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int dev = 0, nsm = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int SW = oz_subpanel_width<T>(nr);   // sub-panel width
    const int ntj = (nc + OZ_TJ - 1) / OZ_TJ;
    for (int k0 = 0; k0 < nr; k0 += PB) {
        if (hook) hook(hctx, 4, 1);
        // sub-panels: FP64 elimination, then the update of the other panel
        // columns as a one-K-step split product on the panel's 128-column tile
        const int c0 = k0 * CX, jt = c0 / OZ_TJ;
        const int it0 = lu ? k0 / OZ_TI : 0, i0 = it0 * OZ_TI;
        for (int sp = 0; sp < PB / SW; ++sp) {
            const int ks = k0 + SW * sp;
            launch_oz_subpanel<T>(W, nr, k0, sp, lu, Z, mask, st);
            k_oz_slice_P16<<<dim3((nr - i0) / 16, W), 256, 0, st>>>(nr, nc, CX, i0, ks * CX, SW * CX, Z, mask);
            k_oz_slice_S<CX><<<dim3(1, W), 256, 0, st>>>(nr, nc, ks, SW, c0 / 64, Z, mask);
            const OzCols inner{c0, c0 + OZ_B, ks * CX, (ks + SW) * CX, jt, jt + 1, it0, nr, nc, oz_rsplit(W, nr / OZ_TI - it0, nsm)};
            k_oz_gemm<1, false><<<nsm, OZ_THREADS, dyn, st>>>(maps, W, nr, nc, inner, Z, mask, err);
        }
        if (hook) { hook(hctx, 4, 0); hook(hctx, 5, 1); }
        const int kn = k0 + PB, itn = lu ? kn / OZ_TI : 0, in = itn * OZ_TI, cl = lu ? kn * CX : 0;
        if (!lu || kn < nr) {
            k_oz_slice_P<<<dim3((nr - in) / 8, W), 256, 0, st>>>(nr, nc, CX, in, c0, OZ_B, Z, mask);
            k_oz_slice_S<CX><<<dim3((nc - cl) / 64, W), 256, 0, st>>>(nr, nc, k0, PB, cl / 64, Z, mask);
            const OzCols outer{cl, nc, c0, c0 + OZ_B, cl / OZ_TJ, ntj, itn, nr, nc,
                               oz_rsplit(W * (ntj - cl / OZ_TJ), nr / OZ_TI - itn, nsm)};
            k_oz_gemm<OZ_B / 16, false><<<nsm, OZ_THREADS, dyn, st>>>(maps, W, nr, nc, outer, Z, mask, err);
        }
        if (hook) hook(hctx, 5, 0);
    }
    return true;
}

template bool oz_eliminate<double>(int, int, const OzWork&, const uint8_t*, bool, int*, cudaStream_t,
                                   void (*)(void*, int, int), void*);
template bool oz_eliminate<c128>(int, int, const OzWork&, const uint8_t*, bool, int*, cudaStream_t,
                                 void (*)(void*, int, int), void*);

// The whole refresh of the selected walkers: M = A^T, n / 64 panels, then the
// column permutation and log|det|.  in_state: Z.M is the state's A^{-1} storage
// and tau is reset; otherwise launch_oz_store does both.
// Needs n % 128 == 0, 128 <= n <= 2048 and W <= 65535 (checked by the caller).
bool launch_refresh_oz(int W, int n, const double* A, const OzWork& Z, const DevState<double>& S,
                       const uint8_t* mask, bool delayed, bool in_state, int* err, cudaStream_t st,
                       void (*hook)(void*, int, int), void* hctx) {
    launch_oz_load<double>(W, n, n, A, true, false, Z, mask, st);
    if (!oz_eliminate<double>(W, n, Z, mask, false, err, st, hook, hctx)) return false;
    launch_oz_finish<double>(W, n, n, true, Z, mask, S.logabs, S.sgn, S.pst,
                             delayed && in_state ? S.tau : nullptr, st);
    return true;
}

// A_0^{-1} -= P Q^T (Sec. 2.3, Eq. delayed_Ainv) for the walkers that flush:
// with M = the stored A_0^{-1} (row l of storage = column l of A_0^{-1}),
// M[l][j] += sum_c (-Q)[l][c] P[j][c]: the P rows take the place of the S
// columns, the -Q rows that of the panel rows, no column is skipped.  The slices
// are padded to a multiple of 64 rows, the state is not.
template <typename T>
bool launch_flush_split(int W, int n, int K, int kk, const int* kv, const T* P, const T* Q, double sgnQ, const int* tau,
                        const uint8_t* force, const OzWork& Z, int* err, cudaStream_t st) {
    constexpr int CX = traits<T>::is_complex ? 2 : 1;
    const int kw = K * kk * CX, nr = oz_flush_rows(n), nc = nr * CX;
    if (kw < 1 || kw > OZ_B) return false;
    const long long rows = (long long)W * OZ_S * nc;
    if (rows >= (1ll << 31)) return false;
    static thread_local OzMaps maps;
    static thread_local const void* cached[2] = {nullptr, nullptr};
    static thread_local long long cached_rows[2] = {-1, -1};
    const long long prow = (long long)W * OZ_S * nr;
    if (cached[0] != Z.Sb || cached[1] != Z.Pb || cached_rows[0] != rows || cached_rows[1] != prow) {
        cached[0] = nullptr;
        if (!oz_map(&maps.S, Z.Sb, rows, OZ_TJ) || !oz_map(&maps.P, Z.Pb, prow, OZ_TI)) return false;
        cached[0] = Z.Sb;
        cached[1] = Z.Pb;
        cached_rows[0] = rows;
        cached_rows[1] = prow;
    }
    const bool edge = n != nr;
    auto kern = edge ? k_oz_gemm<1, true> : k_oz_gemm<1, false>;
    switch ((kw + 15) / 16) {
        case 2: kern = edge ? k_oz_gemm<2, true> : k_oz_gemm<2, false>; break;
        case 3: kern = edge ? k_oz_gemm<3, true> : k_oz_gemm<3, false>; break;
        case 4: kern = edge ? k_oz_gemm<4, true> : k_oz_gemm<4, false>; break;
        default: break;
    }
    // on every call: the limit belongs to the current device, not to the thread
    const size_t dyn = OZ_GEMM_SMEM;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    int dev = 0, nsm = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    k_oz_flush_slices<T><<<std::min(W, 8 * nsm), 256, 0, st>>>(W, n, nr, K, kk, kv, P, Q, sgnQ, tau, force, Z);
    const OzCols all{0, n * CX, -1, -1, 0, (nc + OZ_TJ - 1) / OZ_TJ, 0, n, n * CX, 1};
    kern<<<nsm, OZ_THREADS, dyn, st>>>(maps, W, nr, nc, all, Z, Z.go, err);
    return true;
}

template bool launch_flush_split<double>(int, int, int, int, const int*, const double*, const double*, double, const int*,
                                         const uint8_t*, const OzWork&, int*, cudaStream_t);
template bool launch_flush_split<c128>(int, int, int, int, const int*, const c128*, const c128*, double, const int*,
                                       const uint8_t*, const OzWork&, int*, cudaStream_t);

// Exact skew symmetry of the flushed walkers' A_0^{-1}, after the Pfaffian
// split-product flush A_0^{-1} += P Q^T: the product of the rounded slots
// (P = a M^{-1}, Q = a) is skew only up to that rounding, so the upper
// triangle (each entry one rounding of an exact product) is kept and the
// lower triangle is written as its exact negative (a sign flip, no FP64
// arithmetic), the diagonal as zero -- the same rule as the FP64 skew flush.
// Reads the upper half, writes the lower half.  One CTA per (walker, upper tile).  A walker folded in FP64 (k_oz_flush_slices) is mirrored too:
// the test is the slots', not the product's flag.
// Tiles of 512-byte rows, every load of a thread in flight before the barrier.
template <typename T> constexpr int skew_tw() { return sizeof(T) == 16 ? 32 : 64; }

template <typename T>
__global__ void __launch_bounds__(256) k_skew_project(int n, int K, T* G, const int* tau, const uint8_t* force) {
    constexpr int TW = skew_tw<T>(), NH = TW / 32, NQ = TW / 8;
    __shared__ T sU[TW][TW + 1];
    const int w = blockIdx.y, t = tau[w];
    if (!(force ? (force[w] && t > 0) : t >= K)) return;
    const int nt = (n + TW - 1) / TW;
    int r = 0, rem = (int)blockIdx.x;
    while (rem >= nt - r) { rem -= nt - r; ++r; }
    const int j0 = TW * r, l0 = TW * (r + rem);
    T* Gw = G + (long long)w * n * n;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    // sU[l][j] = G(j0 + j, l0 + l), stored at Gw[(l0 + l) * n + j0 + j]
    T v[NQ][NH];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const int l = l0 + ty + 8 * q, j = j0 + tx + 32 * h;
            v[q][h] = l < n && j < n ? Gw[(long long)l * n + j] : s_zero(T());
        }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int h = 0; h < NH; ++h) sU[ty + 8 * q][tx + 32 * h] = v[q][h];
    __syncthreads();
    // the mirrored block: G(l0 + l, j0 + j) = -G(j0 + j, l0 + l), stored at
    // Gw[(j0 + j) * n + l0 + l]; in a diagonal tile the entries below the diagonal
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const int a = ty + 8 * q, x = tx + 32 * h;   // j within the tile, l within the tile
            if (j0 + a >= n || l0 + x >= n || (rem == 0 && x < a)) continue;
            Gw[(long long)(j0 + a) * n + l0 + x] = rem == 0 && x == a ? s_zero(T()) : s_neg(sU[x][a]);
        }
}

template <typename T>
void launch_skew_project(int W, int n, int K, T* G, const int* tau, const uint8_t* force, cudaStream_t st) {
    const int nt = (n + skew_tw<T>() - 1) / skew_tw<T>();
    k_skew_project<T><<<dim3(nt * (nt + 1) / 2, W), 256, 0, st>>>(n, K, G, tau, force);
}
template void launch_skew_project<double>(int, int, int, double*, const int*, const uint8_t*, cudaStream_t);
template void launch_skew_project<c128>(int, int, int, c128*, const int*, const uint8_t*, cudaStream_t);

}  // namespace lru
