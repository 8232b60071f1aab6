// The two streaming passes over A^{-1} that a proposal of rank k needs, as
// device functions of a PASS_T-thread CTA:
//   dense_x_rows : X = A^{-1} U for XT rows of the dense columns of U
//   dense_y_cols : Y = V A^{-1} for YC columns of A^{-1} and the dense rows of V
// Both read each element of A^{-1} once for up to KB vectors, in 16-byte loads
// where the walker's matrix allows it, and cut a walker into many CTAs: a CTA
// per walker leaves most of the chip idle as soon as sizes differ or walkers
// are few, and rereads A^{-1} once for every four vectors.
#pragma once
#include "common.cuh"
#include "internal.h"

namespace lru {

constexpr int PASS_T = 256;
constexpr int XT = STEP_X_ROWS;   // rows of X per tile
constexpr int YC = 32;         // columns of Y per call (4 per warp)
constexpr int PASS_KK = 16;    // vector slots per update

// Single-precision handles sum in one fixed order on every path (rows: one
// accumulator over l; dot products: one lane per residue of j modulo 32, then
// the butterfly), so that a ratio, whose logarithm is accumulated in double,
// has the same bits from the persistent step, the separate calls and a handle
// of another layout.  They are bound by memory either way.  The double types,
// bound by the FP64 pipe, split the sums as the pass likes.
template <typename T> constexpr bool ordered() { return sizeof(typename traits<T>::real) == 4; }

// Vectors per pass over A^{-1}: with four, the double types are bound by the
// FP64 pipe; single precision goes on gaining to eight, as far as registers go.
template <typename T> constexpr int kb_max() { return ordered<T>() ? 8 : 4; }

// elements of a 16-byte load
template <typename T> constexpr int vec_n() { return 16 / (int)sizeof(T); }
template <typename T, int N> struct alignas(N * sizeof(T)) vecN { T e[N]; };

// matrices whose rows of n elements all start on a 16-byte boundary
template <typename T>
__device__ __forceinline__ bool rows_aligned(const T* G, int n) {
    return ((reinterpret_cast<uintptr_t>(G) | ((size_t)n * sizeof(T))) & 15u) == 0;
}

// Sums N values per lane over the warp with N - 1 exchanges and additions
// instead of 5 N: at each level the lane keeps the half of the values its bit
// selects.  The levels are those of warp_sum (16, 8, .. 1), so every total has
// the bits that warp_sum gives.  Value i ends in v[0] of the 32 / N lanes with
// spread_index<N>() == i.  N a power of two <= 32.
template <int N> __device__ __forceinline__ int spread_index() { return (int)(threadIdx.x & 31) / (32 / N); }
template <int N> __device__ __forceinline__ bool spread_owner() { return (threadIdx.x & 31) % (32 / N) == 0; }

template <typename T> __device__ __forceinline__ T shfl_xor(T v, int m) {
    if constexpr (traits<T>::is_complex) {
        v.re = __shfl_xor_sync(0xffffffffu, v.re, m);
        v.im = __shfl_xor_sync(0xffffffffu, v.im, m);
        return v;
    } else {
        return __shfl_xor_sync(0xffffffffu, v, m);
    }
}

template <int N, typename T>
__device__ __forceinline__ void warp_sum_spread(T (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int m = 16;
#pragma unroll
    for (int h = N / 2; h >= 1; h /= 2, m /= 2) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const T give = up ? v[i] : v[i + h];
            const T keep = up ? v[i + h] : v[i];
            v[i] = keep + shfl_xor(give, m);
        }
    }
#pragma unroll
    for (int o = 16 / N; o >= 1; o /= 2) v[0] = v[0] + shfl_xor(v[0], o);
}

// ---- X = A^{-1} U ---------------------------------------------------------------

template <typename T>
struct XSmem {
    T red[PASS_T / 32][XT];
};

// X[slot_b][j] = sum_l G[l n + j] u_b[l] for rows j0 .. j0 + XT - 1 and the
// columns slot[0 .. nb) of U (nb <= KB).  The warps take the columns l of
// A^{-1} in turn, a lane VR rows of each, so a load instruction reads 512
// contiguous bytes; the warps' sums meet in shared memory.  The rate is the
// FP64 pipe's for the double types (KB FMAs per element) and HBM's otherwise.
template <typename T, int KB, bool VEC>
__device__ void dense_x_group(const T* G, int n, int j0, const T* U, const int* slot, int nb, T* X, XSmem<T>& sm) {
    constexpr int VR = VEC ? vec_n<T>() : 1;
    constexpr int LJ = XT / VR < 32 ? XT / VR : 32;   // lanes along the rows
    constexpr int LL = 32 / LJ;                       // columns of A^{-1} per warp and load
    constexpr int NG = XT / (LJ * VR);
    constexpr int NW = PASS_T / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int lj = (lane % LJ) * VR, ll = lane / LJ;
    T acc[NG][VR][KB];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int r = 0; r < VR; ++r)
#pragma unroll
            for (int b = 0; b < KB; ++b) acc[g][r][b] = s_zero(T());
    const T* ub[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b) ub[b] = U + (size_t)slot[b < nb ? b : 0] * n;
#pragma unroll 4
    for (int l = wid * LL + ll; l < n; l += NW * LL) {
        vecN<T, VR> g[NG];
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            const int j = j0 + q * LJ * VR + lj;
            if (j < n) {
                g[q] = *reinterpret_cast<const vecN<T, VR>*>(G + (size_t)l * n + j);
            } else {
#pragma unroll
                for (int r = 0; r < VR; ++r) g[q].e[r] = s_zero(T());
            }
        }
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const T u = ub[b][l];
#pragma unroll
            for (int q = 0; q < NG; ++q)
#pragma unroll
                for (int r = 0; r < VR; ++r) acc[q][r][b] = s_fma(g[q].e[r], u, acc[q][r][b]);
        }
    }
#pragma unroll
    for (int b = 0; b < KB; ++b) {
        if (b >= nb) break;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
            for (int r = 0; r < VR; ++r) {
                T v = acc[q][r][b];
                if constexpr (LL == 2) v = v + shfl(v, (lane & 15) | ((lane & 16) ^ 16));
                if (ll == 0) sm.red[wid][q * LJ * VR + lj + r] = v;
            }
        __syncthreads();
        if (threadIdx.x < XT && j0 + (int)threadIdx.x < n) {
            T s = sm.red[0][threadIdx.x];
#pragma unroll
            for (int q = 1; q < NW; ++q) s = s + sm.red[q][threadIdx.x];
            X[(size_t)slot[b] * n + j0 + threadIdx.x] = s;
        }
    }
    __syncthreads();
}

// The ordered form: a warp takes the XT rows for itself, two per lane, and walks
// the columns l_lo .. l_hi - 1 in order; a batch of columns is in flight while
// the one before is multiplied.
template <typename T, int KB, bool VEC>
__device__ void dense_x_warp(const T* G, int n, int j0, int l_lo, int l_hi, const T* U, const int* slot, int nb,
                             T (&acc)[2][KB], int (&row)[2]) {
    constexpr int NR = VEC ? 1 : 2, VR = VEC ? 2 : 1;   // loads per column, rows per load
    constexpr int BL = KB > 4 ? 4 : 8;                  // columns per batch
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int b = 0; b < KB; ++b) acc[r][b] = s_zero(T());
    int off[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b) off[b] = slot[b < nb ? b : 0] * n;
#pragma unroll
    for (int r = 0; r < 2; ++r) row[r] = VEC ? j0 + 2 * lane + r : j0 + lane + 32 * r;
    const T* at[NR];   // rows past n are read as row j0 and not stored
#pragma unroll
    for (int q = 0; q < NR; ++q) at[q] = G + (row[q] < n ? row[q] : j0);
    using V = vecN<T, VR>;
    auto load = [&](V (&g)[BL][NR], int l) {
#pragma unroll
        for (int i = 0; i < BL; ++i)
#pragma unroll
            for (int q = 0; q < NR; ++q) g[i][q] = *reinterpret_cast<const V*>(at[q] + (size_t)(l + i) * n);
    };
    auto multiply = [&](const V (&g)[NR], int l) {
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const T u = U[off[b] + l];
#pragma unroll
            for (int r = 0; r < 2; ++r) acc[r][b] = s_fma(g[r / VR].e[r % VR], u, acc[r][b]);
        }
    };
    int l = l_lo;
    if (l + BL <= l_hi) {
        V g[BL][NR];
        load(g, l);
        for (; l + 2 * BL <= l_hi; l += BL) {
            V h[BL][NR];
            load(h, l + BL);
#pragma unroll
            for (int i = 0; i < BL; ++i) multiply(g[i], l + i);
#pragma unroll
            for (int i = 0; i < BL; ++i)
#pragma unroll
                for (int q = 0; q < NR; ++q) g[i][q] = h[i][q];
        }
#pragma unroll
        for (int i = 0; i < BL; ++i) multiply(g[i], l + i);
        l += BL;
    }
    for (; l < l_hi; ++l) {
        V g[NR];
#pragma unroll
        for (int q = 0; q < NR; ++q) g[q] = *reinterpret_cast<const V*>(at[q] + (size_t)l * n);
        multiply(g, l);
    }
}

template <typename T>
__device__ __forceinline__ bool pairs_aligned(const T* G, int n) {
    return ((reinterpret_cast<uintptr_t>(G) | ((size_t)n * sizeof(T))) & (2 * sizeof(T) - 1)) == 0;
}

// XT rows of X for all dense columns, by one warp
template <typename T, int KBM>
__device__ void dense_x_rows_warp(const T* G, int n, int j0, const T* U, unsigned onehot, int kk, T* X) {
    int slot[PASS_KK], nd = 0;
    for (int a = 0; a < kk; ++a)
        if (!((onehot >> a) & 1u)) slot[nd++] = a;
    const bool vec = pairs_aligned(G, n);
    for (int b0 = 0; b0 < nd; b0 += KBM) {
        const int nb = min(KBM, nd - b0);
#define LRU_XW(KB)                                                                         \
    if constexpr (KB <= KBM) {                                                             \
        T acc[2][KB];                                                                      \
        int row[2];                                                                        \
        if (vec) dense_x_warp<T, KB, true>(G, n, j0, 0, n, U, slot + b0, nb, acc, row);    \
        else dense_x_warp<T, KB, false>(G, n, j0, 0, n, U, slot + b0, nb, acc, row);       \
        _Pragma("unroll") for (int b = 0; b < KB; ++b)                                     \
            _Pragma("unroll") for (int r = 0; r < 2; ++r)                                  \
                if (b < nb && row[r] < n) X[(size_t)slot[b0 + b] * n + row[r]] = acc[r][b]; \
    }
        if (nb > 4) { LRU_XW(8) }
        else if (nb > 2) { LRU_XW(4) }
        else if (nb == 2) { LRU_XW(2) }
        else { LRU_XW(1) }
#undef LRU_XW
    }
}

// One dense column in slot a by a pair of warps, each summing half of the range
// of l (half 0 also the last of an odd n): few rows and one vector leave a warp
// little to overlap, so the pair keeps twice the columns in flight.  sm: 64
// values of the pair.
template <typename T>
__device__ void dense_x_halves(const T* G, int n, int j0, const T* U, int a, int half, bool active, T* X, T* sm) {
    T acc[2][1];
    int row[2] = {n, n};
    const int h = n / 2;
    if (active) {
        const int lo = half ? h : 0, hi = half ? 2 * h : h;
        if (pairs_aligned(G, n)) dense_x_warp<T, 1, true>(G, n, j0, lo, hi, U, &a, 1, acc, row);
        else dense_x_warp<T, 1, false>(G, n, j0, lo, hi, U, &a, 1, acc, row);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (half) sm[(threadIdx.x & 31) * 2 + r] = acc[r][0];
            else if ((n & 1) && row[r] < n)
                acc[r][0] = s_fma(G[(size_t)(n - 1) * n + row[r]], U[(size_t)a * n + n - 1], acc[r][0]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 2; ++r)
        if (active && !half && row[r] < n) X[(size_t)a * n + row[r]] = acc[r][0] + sm[(threadIdx.x & 31) * 2 + r];
}

// All dense columns of one walker (kk slots; bit a of onehot set: not dense),
// KBM, .. four, two or one at a time.  G, U and X are the walker's own.
template <typename T, int KBM>
__device__ void dense_x_rows(const T* G, int n, int j0, const T* U, unsigned onehot, int kk, T* X, XSmem<T>& sm) {
    int slot[PASS_KK], nd = 0;
    for (int a = 0; a < kk; ++a)
        if (!((onehot >> a) & 1u)) slot[nd++] = a;
    const bool vec = rows_aligned(G, n);
    for (int b0 = 0; b0 < nd; b0 += KBM) {
        const int nb = min(KBM, nd - b0);
#define LRU_XG(KB)                                                                         \
    if constexpr (KB <= KBM) {                                                             \
        if (vec) dense_x_group<T, KB, true>(G, n, j0, U, slot + b0, nb, X, sm);            \
        else dense_x_group<T, KB, false>(G, n, j0, U, slot + b0, nb, X, sm);               \
    }
        if (nb > 4) { LRU_XG(8) }
        else if (nb > 2) { LRU_XG(4) }
        else if (nb == 2) { LRU_XG(2) }
        else { LRU_XG(1) }
#undef LRU_XG
    }
}

// ---- Y = V A^{-1} ---------------------------------------------------------------

template <typename T>
struct YSmem {
    T y[PASS_KK][YC];
};

// columns a warp keeps in flight, so that KB * CW accumulators stay in registers
template <typename T, int KB> constexpr int y_cw() { return KB * (int)sizeof(T) > 64 ? 2 : 4; }

// sm.y[slot_b][c] = sum_j v_b[j] G[(l0 + c) n + j] for c < nc (<= YC).  A warp
// streams CW columns at once, so that a load of V from L1 serves CW elements
// of A^{-1}.
template <typename T, int KB, bool VEC>
__device__ void dense_y_group(const T* G, int n, int l0, int nc, const T* V, const int* slot, int nb, YSmem<T>& sm) {
    constexpr int VR = VEC && !ordered<T>() ? vec_n<T>() : 1;
    constexpr int CW = y_cw<T, KB>();
    constexpr int NV = CW * KB;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const T* vb[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b) vb[b] = V + (size_t)slot[b < nb ? b : 0] * n;
    for (int c0 = wid * CW; c0 < nc; c0 += (PASS_T / 32) * CW) {
        const T* col[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) col[c] = G + (size_t)(l0 + min(c0 + c, nc - 1)) * n;
        T acc[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] = s_zero(T());
#pragma unroll 2
        for (int j = lane * VR; j < n; j += 32 * VR) {
            vecN<T, VR> g[CW];
#pragma unroll
            for (int c = 0; c < CW; ++c) g[c] = *reinterpret_cast<const vecN<T, VR>*>(col[c] + j);
#pragma unroll
            for (int b = 0; b < KB; ++b) {
                const vecN<T, VR> v = *reinterpret_cast<const vecN<T, VR>*>(vb[b] + j);
#pragma unroll
                for (int c = 0; c < CW; ++c)
#pragma unroll
                    for (int r = 0; r < VR; ++r) acc[c * KB + b] = s_fma(v.e[r], g[c].e[r], acc[c * KB + b]);
            }
        }
        warp_sum_spread<NV>(acc);
        const int i = spread_index<NV>(), c = c0 + i / KB, b = i % KB;   // the value this lane holds now
        if (spread_owner<NV>() && c < nc && b < nb) sm.y[slot[b]][c] = acc[0];
    }
}

// Y of columns l0 .. l0 + nc - 1 (nc <= YC) for all kk slots of V: the dense
// ones by the pass above, one-hot ones e_{iv} by reading element iv of each
// column.  Every thread of the CTA calls it; the result is visible after the
// barrier it ends with.
template <typename T, int KBM>
__device__ void dense_y_cols(const T* G, int n, int l0, int nc, const T* V, const int* siv, int kk, YSmem<T>& sm) {
    int slot[PASS_KK], nd = 0;
    for (int a = 0; a < kk; ++a)
        if (siv[a] < 0) slot[nd++] = a;
    const bool vec = rows_aligned(G, n) && (nd == 0 || rows_aligned(V, n));
    __syncthreads();
    for (int b0 = 0; b0 < nd; b0 += KBM) {
        const int nb = min(KBM, nd - b0);
#define LRU_YG(KB)                                                                         \
    if constexpr (KB <= KBM) {                                                             \
        if (vec) dense_y_group<T, KB, true>(G, n, l0, nc, V, slot + b0, nb, sm);           \
        else dense_y_group<T, KB, false>(G, n, l0, nc, V, slot + b0, nb, sm);              \
    }
        if (nb > 4) { LRU_YG(8) }
        else if (nb > 2) { LRU_YG(4) }
        else if (nb == 2) { LRU_YG(2) }
        else { LRU_YG(1) }
#undef LRU_YG
    }
    if (nd < kk)
        for (int e = threadIdx.x; e < kk * nc; e += PASS_T) {
            const int a = e / nc, c = e - a * nc;
            if (siv[a] >= 0) sm.y[a][c] = G[(size_t)(l0 + c) * n + siv[a]];
        }
    __syncthreads();
}

// y -= (V P) Q[l,:]^T for the nc columns l0 .. and kk rows in sm (VP: rows of
// 64, Q the walker's slot rows of ld); ends with a barrier.
template <typename T>
__device__ void slot_correct_y(const T* Q, int ld, int cu, int l0, int nc, const T* VP, int kk, YSmem<T>& sm) {
    if constexpr (ordered<T>()) {
        // a warp per column: the lanes split the slots
        const int lane = threadIdx.x & 31;
        for (int c = threadIdx.x >> 5; c < nc; c += PASS_T / 32) {
            const T* qrow = Q + (size_t)(l0 + c) * ld;
            const T q0 = lane < cu ? qrow[lane] : s_zero(T()), q1 = lane + 32 < cu ? qrow[lane + 32] : s_zero(T());
            for (int b0 = 0; b0 < kk; b0 += 4) {
                T v[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    v[b] = s_zero(T());
                    if (b0 + b < kk) {
                        if (lane < cu) v[b] = s_fma(VP[(b0 + b) * 64 + lane], q0, v[b]);
                        if (lane + 32 < cu) v[b] = s_fma(VP[(b0 + b) * 64 + lane + 32], q1, v[b]);
                    }
                }
                warp_sum_spread<4>(v);
                const int b = b0 + spread_index<4>();
                if (spread_owner<4>() && b < kk) sm.y[b][c] = sm.y[b][c] - v[0];
            }
        }
    } else {
        for (int e = threadIdx.x; e < kk * nc; e += PASS_T) {
            const int c = e / kk, b = e - c * kk;
            const T* qrow = Q + (size_t)(l0 + c) * ld;
            T y = sm.y[b][c];
            for (int q = 0; q < cu; ++q) y = s_fms(VP[b * 64 + q], qrow[q], y);
            sm.y[b][c] = y;
        }
    }
    __syncthreads();
}

// ---- products with the delay slots ------------------------------------------------

template <typename T>
struct SlotSmem {
    T red[PASS_T / 32][4][32];
};

// store(c, slot_b, sum_j M[j ld + c] v_b[j]) for c < cu and nb <= KB vectors.
// The lanes lie along the slot columns of a row, so the rows of M are read
// whole (a warp per column touches one sector of every row per element).
template <typename T, int KB, typename F>
__device__ void slot_dot_group(const T* M, int ld, int cu, int n, const T* V, const int* slot, int nb, SlotSmem<T>& sm,
                               F store) {
    constexpr int NW = PASS_T / 32;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const T* vb[KB];
#pragma unroll
    for (int b = 0; b < KB; ++b) vb[b] = V + (size_t)slot[b < nb ? b : 0] * n;
    for (int c0 = 0; c0 < cu; c0 += 32) {
        const int cw = min(32, cu - c0);
        int sh = 5;                                   // 2^sh lanes along the columns
        while (sh > 0 && (1 << (sh - 1)) >= cw) --sh;
        const int c = lane & ((1 << sh) - 1), r = lane >> sh, rows = 32 >> sh;
        T acc[KB];
#pragma unroll
        for (int b = 0; b < KB; ++b) acc[b] = s_zero(T());
        if (c < cw) {
            const T* m = M + c0 + c;
#pragma unroll 4
            for (int j = wid * rows + r; j < n; j += NW * rows) {
                const T x = m[(size_t)j * ld];
#pragma unroll
                for (int b = 0; b < KB; ++b) acc[b] = s_fma(vb[b][j], x, acc[b]);
            }
        }
        for (int o = 1 << sh; o < 32; o *= 2)
#pragma unroll
            for (int b = 0; b < KB; ++b) acc[b] = acc[b] + shfl(acc[b], lane ^ o);
        __syncthreads();
        if (lane < cw)
#pragma unroll
            for (int b = 0; b < KB; ++b) sm.red[wid][b][lane] = acc[b];
        __syncthreads();
        for (int e = threadIdx.x; e < nb * cw; e += PASS_T) {
            const int b = e / cw, q = e - b * cw;
            T s = sm.red[0][b][q];
#pragma unroll
            for (int w = 1; w < NW; ++w) s = s + sm.red[w][b][q];
            store(c0 + q, slot[b], s);
        }
    }
}

// 4 vectors x 8 slot columns per thread or lane, the ordered form's block
template <typename T, bool V_FIRST>
__device__ __forceinline__ void slot_block(const T* mrow, int cw, const T* const (&vb)[4], int j, T (&acc)[32]) {
    T v[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) v[b] = vb[b][j];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const T x = c < cw ? mrow[c] : s_zero(T());
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[c * 4 + b] = V_FIRST ? s_fma(v[b], x, acc[c * 4 + b]) : s_fma(x, v[b], acc[c * 4 + b]);
    }
}

// Ordered forms.  BY_WARP: a warp sums one block over all j (lane t: j = t, t +
// 32, ..), the order of the V P products; otherwise the CTA does (thread t: j =
// t, t + PASS_T, .., then the warps in turn), the order of Q^T U.
template <typename T, bool BY_WARP, typename F>
__device__ void slot_dot_ordered(const T* M, int ld, int cu, int n, const T* V, const int* slot, int nd,
                                 SlotSmem<T>& sm, F store) {
    const int wid = threadIdx.x >> 5, nbg = (nd + 3) / 4, ncg = (cu + 7) / 8;
    for (int p = BY_WARP ? wid : 0; p < nbg * ncg; p += BY_WARP ? PASS_T / 32 : 1) {
        const int b0 = (p % nbg) * 4, c0 = (p / nbg) * 8, cw = min(8, cu - c0);
        const T* vb[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) vb[b] = V + (size_t)slot[min(b0 + b, nd - 1)] * n;
        T acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = s_zero(T());
        constexpr int STEP = BY_WARP ? 32 : PASS_T;
        for (int j = threadIdx.x & (STEP - 1); j < n; j += STEP)
            slot_block<T, BY_WARP>(M + (size_t)j * ld + c0, cw, vb, j, acc);
        warp_sum_spread<32>(acc);
        const int i = threadIdx.x & 31, c = i / 4, b = b0 + i % 4;
        if constexpr (BY_WARP) {
            if (c < cw && b < nd) store(c0 + c, slot[b], acc[0]);
        } else {
            __syncthreads();
            sm.red[wid][0][i] = acc[0];
            __syncthreads();
            if (wid == 0 && c < cw && b < nd) {
                T s = s_zero(T());
#pragma unroll
                for (int w = 0; w < PASS_T / 32; ++w) s = s + sm.red[w][0][i];
                store(c0 + c, slot[b], s);
            }
        }
    }
    __syncthreads();
}

// store(c, slot_b, ..) for the nd vectors slot[0 .. nd) of V; ends with a barrier.
template <typename T, bool BY_WARP, typename F>
__device__ void slot_dot(const T* M, int ld, int cu, int n, const T* V, const int* slot, int nd, SlotSmem<T>& sm,
                         F store) {
    if constexpr (ordered<T>()) {
        slot_dot_ordered<T, BY_WARP>(M, ld, cu, n, V, slot, nd, sm, store);
        return;
    }
    for (int b0 = 0; b0 < nd; b0 += 4) {
        const int nb = min(4, nd - b0);
        if (nb > 2) slot_dot_group<T, 4>(M, ld, cu, n, V, slot + b0, nb, sm, store);
        else if (nb == 2) slot_dot_group<T, 2>(M, ld, cu, n, V, slot + b0, nb, sm, store);
        else slot_dot_group<T, 1>(M, ld, cu, n, V, slot + b0, nb, sm, store);
    }
    __syncthreads();
}

// s[b] += sum_c prow[c] q[c * PASS_KK + b] for b < NB (prow: the slot row of one j)
template <typename T, int NB, bool VEC>
__device__ __forceinline__ void slot_row(const T* prow, int cu, const T* q, T (&s)[NB]) {
    constexpr int VR = VEC ? vec_n<T>() : 1;
    int c = 0;
    for (; c + VR <= cu; c += VR) {
        const vecN<T, VR> p = *reinterpret_cast<const vecN<T, VR>*>(prow + c);
#pragma unroll
        for (int r = 0; r < VR; ++r)
#pragma unroll
            for (int b = 0; b < NB; ++b) s[b] = s_fma(p.e[r], q[(c + r) * PASS_KK + b], s[b]);
    }
    for (; c < cu; ++c)
#pragma unroll
        for (int b = 0; b < NB; ++b) s[b] = s_fma(prow[c], q[c * PASS_KK + b], s[b]);
}

// X_a[j] -/+= (P q_a)[j] for the columns a0 .. a0 + NB - 1 of X (rows of P: ld)
template <typename T, int NB>
__device__ void slot_correct(const T* P, int ld, int cu, int n, const T* q, bool add, T* X) {
    const bool vec = (((size_t)ld * sizeof(T)) & 15u) == 0 && (reinterpret_cast<uintptr_t>(P) & 15u) == 0;
    for (int j = threadIdx.x; j < n; j += PASS_T) {
        T s[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) s[b] = s_zero(T());
        const T* prow = P + (size_t)j * ld;
        if (vec) slot_row<T, NB, true>(prow, cu, q, s);
        else slot_row<T, NB, false>(prow, cu, q, s);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            T* x = X + (size_t)b * n + j;
            *x = add ? (*x + s[b]) : (*x - s[b]);
        }
    }
}

}  // namespace lru
