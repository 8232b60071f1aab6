// From-scratch inverse, log|det| and Pfaffian of the walker matrices: the
// initial carrier (Sec. 2.3 init_det_carrier, Sec. 3.3 init_pf_carrier) and
// the periodic refresh that bounds the drift of the update chain (Sec. 2.1
// advises double precision against accumulated error).  Always run in the
// handle dtype (FP64 / complex128 for the double types).
#include "common.cuh"
#include "internal.h"

#include <algorithm>
#include <type_traits>

namespace lru {

constexpr int RT = 256;   // threads per matrix
constexpr int GB = 16;    // Gauss-Jordan panel width

__device__ void block_argmax(double v, int i, double* sv, int* si, double& bv, int& bi) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        double ov = __shfl_xor_sync(0xffffffffu, v, o);
        int oi = __shfl_xor_sync(0xffffffffu, i, o);
        if (ov > v || (ov == v && oi >= 0 && (i < 0 || oi < i))) { v = ov; i = oi; }
    }
    if (lane == 0) { sv[wid] = v; si[wid] = i; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double b = sv[0];
        int ib = si[0];
        for (int q = 1; q < RT / 32; ++q)
            if (sv[q] > b || (sv[q] == b && si[q] >= 0 && (ib < 0 || si[q] < ib))) { b = sv[q]; ib = si[q]; }
        sv[0] = b;
        si[0] = ib;
    }
    __syncthreads();
    bv = sv[0];
    bi = si[0];
    __syncthreads();
}

// Loads M = A^T (A row-major n x n) through 32 x 32 shared-memory tiles.
template <typename T>
__device__ void load_transposed(T* M, const T* A, int n, T (*tile)[33]) {
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int b0 = 0; b0 < n; b0 += 32)
        for (int b1 = 0; b1 < n; b1 += 32) {
            for (int q = ty; q < 32; q += RT / 32) {
                const int r = b0 + q, c = b1 + tx;
                if (r < n && c < n) tile[q][tx] = A[(long long)r * n + c];
            }
            __syncthreads();
            for (int q = ty; q < 32; q += RT / 32) {
                const int r = b1 + q, c = b0 + tx;   // M[r][c] = A[c][r]
                if (r < n && c < n) M[(long long)r * n + c] = tile[tx][q];
            }
            __syncthreads();
        }
}

// In-place Gauss-Jordan inversion with partial pivoting of the row-major n x n
// matrix M, blocked in panels of GB columns: each panel is eliminated with the
// row exchanges restricted to it, then the exchanges and the panel's
// accumulated transform T = I + sum_c (panel_c - e_c) e_c^T are applied to the
// other columns as one rank-GB update (a GEMM).  Row exchanges turn into
// column exchanges of the inverse, undone at the end.  Returns log|det M| and
// its sign/phase; *singular is set when a pivot is exactly zero.
template <typename T>
struct GJSmem {
    T sS[GB][64];
    T sPan[64][GB + 1];
    T tile[32][33];
};

// Eliminates columns [c_lo, c_hi) of M (all rows) in panels of GB columns,
// applying each panel's row exchanges and rank-GB transform to the other
// columns of [j_lo, j_hi) only.  Pivot rows go to perm[k]; log|pivot| and the
// sign/phase accumulate into the shared s_log / s_sgn, a zero pivot sets
// s_sing.  The full inverse is c = j = [0, n).
template <typename T>
__device__ void gj_columns(T* M, int n, int c_lo, int c_hi, int j_lo, int j_hi, int* perm, double& s_log, T& s_sgn,
                           int& s_sing, GJSmem<T>& sm) {
    __shared__ double s_v[32];
    __shared__ int s_i[32];
    __shared__ T s_rowk[GB];
    auto& sS = sm.sS;
    auto& sPan = sm.sPan;
    const int tid = threadIdx.x;

    for (int k0 = c_lo; k0 < c_hi; k0 += GB) {
        const int bw = min(GB, c_hi - k0);
        // ---- panel ----
        for (int kc = 0; kc < bw; ++kc) {
            const int k = k0 + kc;
            double best = -1.0;
            int bi = -1;
            for (int i = k + tid; i < n; i += RT) {
                double v = (double)s_abs2(M[(long long)i * n + k]);
                if (v > best) { best = v; bi = i; }
            }
            double bv;
            int p;
            block_argmax(best, bi, s_v, s_i, bv, p);
            if (!(bv > 0.0) || p < 0) {
                if (tid == 0) { perm[k] = k; s_sing = 1; }
                __syncthreads();
                continue;
            }
            if (tid == 0) perm[k] = p;
            if (p != k && tid < bw) {
                T a = M[(long long)k * n + k0 + tid];
                M[(long long)k * n + k0 + tid] = M[(long long)p * n + k0 + tid];
                M[(long long)p * n + k0 + tid] = a;
            }
            __syncthreads();
            const T piv = M[(long long)k * n + k];
            const T ipiv = s_recip(piv);
            if (tid < bw) {
                T v = (tid == kc) ? make_real<T>(1.0) : M[(long long)k * n + k0 + tid];
                v = v * ipiv;
                s_rowk[tid] = v;
                M[(long long)k * n + k0 + tid] = v;
            }
            if (tid == 0) {
                s_log += log(s_absd(piv));
                T sg = s_sgn * s_unit(piv);
                s_sgn = (p != k) ? s_neg(sg) : sg;
            }
            __syncthreads();
            for (int i = tid; i < n; i += RT) {
                if (i == k) continue;
                T* row = M + (long long)i * n + k0;
                const T f = row[kc];
                for (int c = 0; c < bw; ++c) {
                    T v = (c == kc) ? s_zero(T()) : row[c];
                    row[c] = s_fms(f, s_rowk[c], v);
                }
            }
            __syncthreads();
        }
        // ---- the panel's row exchanges on the other columns ----
        for (int kc = 0; kc < bw; ++kc) {
            const int k = k0 + kc, p = perm[k];
            if (p != k)
                for (int j = j_lo + tid; j < j_hi; j += RT) {
                    if (j >= k0 && j < k0 + bw) continue;
                    T a = M[(long long)k * n + j];
                    M[(long long)k * n + j] = M[(long long)p * n + j];
                    M[(long long)p * n + j] = a;
                }
            __syncthreads();
        }
        // ---- rank-bw update of the other columns: M += (panel - E) S ----
        const int tx = tid & 15, ty = tid >> 4;   // 16 x 16 threads, 4 x 4 outputs each
        for (int j0 = j_lo; j0 < j_hi; j0 += 64) {
            for (int e = tid; e < GB * 64; e += RT) {
                const int c = e / 64, jj = e % 64;
                sS[c][jj] = (c < bw && j0 + jj < j_hi) ? M[(long long)(k0 + c) * n + j0 + jj] : s_zero(T());
            }
            __syncthreads();
            for (int i0 = 0; i0 < n; i0 += 64) {
                for (int e = tid; e < 64 * GB; e += RT) {
                    const int ii = e / GB, c = e % GB;
                    const int i = i0 + ii;
                    T v = s_zero(T());
                    if (c < bw && i < n) {
                        v = M[(long long)i * n + k0 + c];
                        if (i == k0 + c) v = v - make_real<T>(1.0);
                    }
                    sPan[ii][c] = v;
                }
                __syncthreads();
                T acc[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[r][c] = s_zero(T());
                for (int cc = 0; cc < bw; ++cc) {
                    T a[4], b[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) a[r] = sPan[ty * 4 + r][cc];
#pragma unroll
                    for (int c = 0; c < 4; ++c) b[c] = sS[cc][tx * 4 + c];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[r][c] = s_fma(a[r], b[c], acc[r][c]);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int i = i0 + ty * 4 + r;
                    if (i >= n) continue;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int j = j0 + tx * 4 + c;
                        if (j >= j_hi || (j >= k0 && j < k0 + bw)) continue;
                        M[(long long)i * n + j] = M[(long long)i * n + j] + acc[r][c];
                    }
                }
                __syncthreads();
            }
        }
    }
}

// In-place Gauss-Jordan inverse of M (see gj_columns), exchanges undone.
template <typename T>
__device__ void gj_invert(T* M, int n, int* perm, double* logabs_out, T* sgn_out, int* singular, GJSmem<T>& sm) {
    __shared__ double s_log;
    __shared__ T s_sgn;
    __shared__ int s_sing;
    const int tid = threadIdx.x;
    if (tid == 0) { s_log = 0.0; s_sgn = make_real<T>(1.0); s_sing = 0; }
    __syncthreads();
    gj_columns(M, n, 0, n, 0, n, perm, s_log, s_sgn, s_sing, sm);
    // ---- undo the exchanges as column exchanges, last first ----
    for (int k = n - 1; k >= 0; --k) {
        const int p = perm[k];
        if (p != k)
            for (int i = tid; i < n; i += RT) {
                T a = M[(long long)i * n + k];
                M[(long long)i * n + k] = M[(long long)i * n + p];
                M[(long long)i * n + p] = a;
            }
        __syncthreads();
    }
    if (tid == 0) {
        *logabs_out = s_sing ? -INFINITY : s_log;
        *sgn_out = s_sing ? s_zero(T()) : s_renorm(s_sgn);
        *singular = s_sing;
    }
    __syncthreads();
}

// One CTA per (selected) walker.  target: ws slot of the CTA when ws != null
// (refresh with drift), else the state G itself.
template <typename T>
__global__ void __launch_bounds__(RT) k_refresh(DevLayout L, DevState<T> S, const T* A, const uint8_t* mask,
                                                 T* ws, int nws, double* drift, bool pf, bool delayed,
                                                 bool write_logdet) {
    extern __shared__ __align__(16) unsigned char dsm[];
    GJSmem<T>& sm = *reinterpret_cast<GJSmem<T>*>(dsm);
    __shared__ int perm[2048];
    __shared__ double s_l;
    __shared__ T s_s;
    __shared__ int s_sing;
    __shared__ double s_red[2][32];
    for (int w = blockIdx.x; w < L.W; w += gridDim.x) {
        if (mask && !mask[w]) continue;
        const int n = L.nw(w);
        T* G = S.G + L.mo(w);
        T* M = ws ? ws + (long long)blockIdx.x * (long long)L.n_max * L.n_max : G;
        load_transposed(M, A + L.mo(w), n, sm.tile);
        __syncthreads();
        gj_invert(M, n, perm, &s_l, &s_s, &s_sing, sm);
        if (pf) {
            // the inverse of a skew matrix is skew: keep it exactly so
            for (long long e = threadIdx.x; e < (long long)n * n; e += RT) {
                const int i = (int)(e / n), j = (int)(e % n);
                if (i < j) {
                    T h = s_half(M[(long long)i * n + j] - M[(long long)j * n + i]);
                    M[(long long)i * n + j] = h;
                    M[(long long)j * n + i] = s_neg(h);
                } else if (i == j) {
                    M[e] = s_zero(T());
                }
            }
            __syncthreads();
        }
        if (ws) {
            // drift of the tracked inverse, then replace it
            double num = 0.0, den = 0.0;
            const int kk = L.kv(w);
            const int cu = delayed ? S.tau[w] * kk : 0;
            const long long vo = L.vo(w);
            for (long long e = threadIdx.x; e < (long long)n * n; e += RT) {
                const int l = (int)(e / n), j = (int)(e % n);   // memory [l*n + j] = (A^{-1})_{jl}
                T tr = G[e];
                if (cu) {
                    const T* pr = S.P + (vo + j) * L.Kc;
                    const T* qr = S.Q + (vo + l) * L.Kc;
                    T s = s_zero(T());
                    for (int c = 0; c < cu; ++c) s = s_fma(pr[c], qr[c], s);
                    tr = pf ? tr + s : tr - s;
                }
                T f = M[e];
                num += (double)s_abs2(tr - f);
                den += (double)s_abs2(f);
                G[e] = f;
            }
            num = warp_sum(num);
            den = warp_sum(den);
            if ((threadIdx.x & 31) == 0) { s_red[0][threadIdx.x >> 5] = num; s_red[1][threadIdx.x >> 5] = den; }
            __syncthreads();
            if (threadIdx.x == 0) {
                double a = 0, b = 0;
                for (int q = 0; q < RT / 32; ++q) { a += s_red[0][q]; b += s_red[1][q]; }
                if (drift) drift[w] = b > 0 ? sqrt(a / b) : 0.0;
            }
        }
        if (threadIdx.x == 0) {
            if (write_logdet) {
                S.logabs[w] = s_l;
                S.sgn[w] = s_s;
            }
            if (delayed) S.tau[w] = 0;
            S.pst[w] = s_sing ? 1 : 5;   // 5: fresh, no pending proposal
        }
        __syncthreads();
    }
}

// Pfaffian of a skew n x n matrix (row-major copy in M) by Parlett-Reid
// elimination with pivoting (see small_pf for the step), one CTA per matrix.
template <typename T>
__device__ void pr_pfaffian(T* M, int n, double* logabs, T* sgn, T* s_tau, T* s_row) {
    __shared__ double s_v[32];
    __shared__ int s_i[32];
    __shared__ double s_log;
    __shared__ T s_sg;
    __shared__ int s_zero_pf;
    const int tid = threadIdx.x;
    if (tid == 0) { s_log = 0.0; s_sg = make_real<T>(1.0); s_zero_pf = (n & 1); }
    __syncthreads();
    for (int k = 0; k + 1 < n && !s_zero_pf; k += 2) {
        double best = -1.0;
        int bi = -1;
        for (int i = k + 1 + tid; i < n; i += RT) {
            double v = (double)s_abs2(M[(long long)i * n + k]);
            if (v > best) { best = v; bi = i; }
        }
        double bv;
        int p;
        block_argmax(best, bi, s_v, s_i, bv, p);
        if (!(bv > 0.0) || p < 0) {
            if (tid == 0) s_zero_pf = 1;
            __syncthreads();
            break;
        }
        if (p != k + 1) {
            // swap rows k+1, p, then columns k+1, p
            for (int j = tid; j < n; j += RT) {
                T a = M[(long long)(k + 1) * n + j];
                M[(long long)(k + 1) * n + j] = M[(long long)p * n + j];
                M[(long long)p * n + j] = a;
            }
            __syncthreads();
            for (int i = tid; i < n; i += RT) {
                T a = M[(long long)i * n + k + 1];
                M[(long long)i * n + k + 1] = M[(long long)i * n + p];
                M[(long long)i * n + p] = a;
            }
        }
        __syncthreads();
        const T akk1 = M[(long long)k * n + k + 1];
        if (tid == 0) {
            s_log += log(s_absd(akk1));
            T sg = s_sg * s_unit(akk1);
            s_sg = (p != k + 1) ? s_neg(sg) : sg;
        }
        const T ipiv = s_recip(M[(long long)(k + 1) * n + k]);
        for (int i = k + 2 + tid; i < n; i += RT) {
            s_tau[i] = M[(long long)i * n + k] * ipiv;
            s_row[i] = M[(long long)(k + 1) * n + i];
        }
        __syncthreads();
        const int m = n - k - 2;
        for (long long e = tid; e < (long long)m * m; e += RT) {
            const int i = k + 2 + (int)(e / m), j = k + 2 + (int)(e % m);
            T v = s_fms(s_tau[i], s_row[j], M[(long long)i * n + j]);
            M[(long long)i * n + j] = s_fma(s_tau[j], s_row[i], v);
        }
        __syncthreads();
    }
    if (tid == 0) {
        *logabs = s_zero_pf ? -INFINITY : s_log;
        *sgn = s_zero_pf ? s_zero(T()) : s_renorm(s_sg);
    }
    __syncthreads();
}

// The same elimination for large matrices of the double types, blocked: only the
// upper triangle is kept (a row right of the diagonal is minus the column below it), and the
// congruences of PFB / 2 pairs are collected before they meet the trailing block,
// as one rank-PFB update of its upper tiles in 64 x 64 register tiles.  Inside a
// block of pairs the two rows that a pair needs are brought up to date one by one.
// The collected vectors tau_t and r_t lie in the rows k and k + 1 that their pair
// has used up.  The unblocked form reads and writes the whole trailing block for
// every pair (n^3 / 6 scalars each way, twice the FMAs): 1024 matrices of n = 256
// took 27.9 ms at two CTAs per SM and 18.9 at four, of which the FP64 pipe accounts
// for 9; this form 12.0 ms (four), 4.6 of the FP64 pipe, the rest the row-by-row
// phase and its barriers.
constexpr int PFB = 16;   // rows (two per pair) collected per update

template <typename T>
struct PfSmem {
    T l[PFB][64], r[PFB][64];
    T ca[PFB];               // tau_t, r_t at the row in hand
};

// x - sum_t (tau_t[i] r_t[j] - r_t[i] tau_t[j]) over the m collected rows at k0,
// ca: their entries at i
template <typename T>
__device__ __forceinline__ T pf_current(const T* M, int n, int k0, int m, const T* ca, int j, T x) {
    for (int t = 0; t < m; t += 2) {
        x = s_fms(ca[t], M[(long long)(k0 + t + 1) * n + j], x);
        x = s_fma(ca[t + 1], M[(long long)(k0 + t) * n + j], x);
    }
    return x;
}

template <typename T>
__device__ void pr_pfaffian_blocked(T* M, int n, double* logabs, T* sgn, PfSmem<T>& sm) {
    __shared__ double s_v[32];
    __shared__ int s_i[32];
    __shared__ double s_log;
    __shared__ T s_sg;
    const int tid = threadIdx.x;
    if (tid == 0) { s_log = 0.0; s_sg = make_real<T>(1.0); }
    bool zero_pf = (n & 1) != 0;
    __syncthreads();
    for (int k0 = 0; k0 + 1 < n && !zero_pf; k0 += PFB) {
        const int rows = min(PFB, n - k0);
        for (int m = 0; m < rows; m += 2) {
            const int k = k0 + m;
            T* rk = M + (long long)k * n;
            T* rk1 = rk + n;
            // ---- row k, and its largest entry ----
            if (tid < m) sm.ca[tid] = M[(long long)(k0 + tid) * n + k];
            __syncthreads();
            double best = -1.0;
            int bi = -1;
            for (int j = k + 1 + tid; j < n; j += RT) {
                const T c = pf_current(M, n, k0, m, sm.ca, j, rk[j]);
                rk[j] = c;
                const double v = (double)s_abs2(c);
                if (v > best) { best = v; bi = j; }
            }
            double bv;
            int p;
            block_argmax(best, bi, s_v, s_i, bv, p);
            if (!(bv > 0.0) || p < 0) { zero_pf = true; break; }
            // ---- rows and columns k + 1 and p change places ----
            if (p != k + 1) {
                for (int j = k + 2 + tid; j < n; j += RT) {
                    if (j == p) {
                        rk1[p] = s_neg(rk1[p]);
                    } else if (j > p) {
                        const T a = rk1[j];
                        rk1[j] = M[(long long)p * n + j];
                        M[(long long)p * n + j] = a;
                    } else {
                        const T a = rk1[j];
                        rk1[j] = s_neg(M[(long long)j * n + p]);
                        M[(long long)j * n + p] = s_neg(a);
                    }
                }
                if (tid <= m) {   // the collected rows, and row k
                    T* r = M + (long long)(k0 + tid) * n;
                    const T a = r[k + 1];
                    r[k + 1] = r[p];
                    r[p] = a;
                }
                __syncthreads();
            }
            // ---- tau (row k) and r (row k + 1) ----
            const T akk1 = rk[k + 1];
            if (tid < m) sm.ca[tid] = M[(long long)(k0 + tid) * n + k + 1];
            if (tid == 0) {
                s_log += log(s_absd(akk1));
                const T sg = s_sg * s_unit(akk1);
                s_sg = (p != k + 1) ? s_neg(sg) : sg;
            }
            __syncthreads();
            const T inv = s_recip(akk1);
            for (int j = k + 2 + tid; j < n; j += RT) {
                rk1[j] = pf_current(M, n, k0, m, sm.ca, j, rk1[j]);
                rk[j] = rk[j] * inv;
            }
            __syncthreads();
        }
        if (zero_pf) break;
        // ---- the trailing block's upper tiles: A_ij -= sum_t tau_t[i] r_t[j] - r_t[i] tau_t[j] ----
        const int b0 = k0 + rows, tx = tid & 15, ty = tid >> 4;
        for (int i0 = b0; i0 < n; i0 += 64) {
            __syncthreads();
            for (int e = tid; e < rows * 64; e += RT) {
                const int t = e >> 6, q = e & 63;
                sm.l[t][q] = i0 + q < n ? M[(long long)(k0 + t) * n + i0 + q] : s_zero(T());
            }
            for (int j0 = i0; j0 < n; j0 += 64) {
                __syncthreads();
                for (int e = tid; e < rows * 64; e += RT) {
                    const int t = e >> 6, q = e & 63;
                    // paired with l: tau with r, r with -tau
                    const T v = j0 + q < n ? M[(long long)(k0 + (t ^ 1)) * n + j0 + q] : s_zero(T());
                    sm.r[t][q] = (t & 1) ? s_neg(v) : v;
                }
                __syncthreads();
                T acc[4][4];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int i = i0 + ty * 4 + r, j = j0 + tx + 16 * c;
                        acc[r][c] = i < j && j < n ? M[(long long)i * n + j] : s_zero(T());
                    }
                for (int t = 0; t < rows; ++t) {
                    T a[4], b[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) a[r] = sm.l[t][ty * 4 + r];
#pragma unroll
                    for (int c = 0; c < 4; ++c) b[c] = sm.r[t][tx + 16 * c];
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int c = 0; c < 4; ++c) acc[r][c] = s_fms(a[r], b[c], acc[r][c]);
                }
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const int i = i0 + ty * 4 + r, j = j0 + tx + 16 * c;
                        if (i < j && j < n) M[(long long)i * n + j] = acc[r][c];
                    }
            }
        }
        __syncthreads();
    }
    __syncthreads();
    if (tid == 0) {
        *logabs = zero_pf ? -INFINITY : s_log;
        *sgn = zero_pf ? s_zero(T()) : s_renorm(s_sg);
    }
    __syncthreads();
}

template <typename T, bool BLOCKED>
__global__ void __launch_bounds__(RT, std::is_same<T, double>::value ? 4 : 2)
    k_slogpf(DevLayout L, const T* A, const uint8_t* mask, T* ws, double* logabs, T* sgn) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ double s_l;
    __shared__ T s_s;
    for (int w = blockIdx.x; w < L.W; w += gridDim.x) {
        if (mask && !mask[w]) continue;
        const int n = L.nw(w);
        T* M = ws + (long long)blockIdx.x * (long long)L.n_max * L.n_max;
        const T* Aw = A + L.mo(w);
        for (long long e = threadIdx.x; e < (long long)n * n; e += RT) M[e] = Aw[e];
        __syncthreads();
        if constexpr (BLOCKED) {
            pr_pfaffian_blocked(M, n, &s_l, &s_s, *reinterpret_cast<PfSmem<T>*>(dsm));
        } else {
            T* s_tau = reinterpret_cast<T*>(dsm);
            pr_pfaffian(M, n, &s_l, &s_s, s_tau, s_tau + L.n_max);
        }
        if (threadIdx.x == 0) {
            logabs[w] = s_l;
            sgn[w] = s_s;
        }
        __syncthreads();
    }
}

// standalone slogdet (GJ on a workspace copy)
template <typename T>
__global__ void __launch_bounds__(RT) k_slogdet(int W, int n, const T* A, T* ws, double* logabs, T* sgn,
                                                 const uint8_t* mask) {
    extern __shared__ __align__(16) unsigned char dsm[];
    GJSmem<T>& sm = *reinterpret_cast<GJSmem<T>*>(dsm);
    __shared__ int perm[2048];
    __shared__ double s_l;
    __shared__ T s_s;
    __shared__ int s_sing;
    for (int w = blockIdx.x; w < W; w += gridDim.x) {
        if (mask && !mask[w]) continue;
        T* M = ws + (long long)blockIdx.x * n * n;
        const T* Aw = A + (long long)w * n * n;
        for (long long e = threadIdx.x; e < (long long)n * n; e += RT) M[e] = Aw[e];
        __syncthreads();
        gj_invert(M, n, perm, &s_l, &s_s, &s_sing, sm);
        if (threadIdx.x == 0) {
            logabs[w] = s_l;
            sgn[w] = s_s;
        }
        __syncthreads();
    }
}

template <typename T>
void launch_refresh(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const T* A,
                    const uint8_t* mask, T* ws, int nws, double* drift, bool write_logdet, cudaStream_t st) {
    const int grid = ws ? nws : L.W;
    const int dyn = (int)sizeof(GJSmem<T>);
    cudaFuncSetAttribute(k_refresh<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    k_refresh<T><<<grid, RT, dyn, st>>>(L, S, A, mask, ws, nws, drift, pf, delayed, write_logdet);
}

template <typename T>
void launch_slogpf(const DevLayout& L, const T* A, const uint8_t* mask, T* ws, int nws, double* logabs, T* sgn,
                   cudaStream_t st) {
    auto go = [&](auto kern, size_t dyn) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        kern<<<nws, RT, dyn, st>>>(L, A, mask, ws, logabs, sgn);
    };
    // The blocked form for the double types where it is the faster one (its row phase
    // costs seven barriers a pair, whatever n).  Per call of 1 / 152 / 304 / 1024
    // matrices on 152 SMs, blocked against unblocked, ms: F64 n = 112 0.55 / 0.55 / 0.77
    // / 2.46 against 0.56 / 0.59 / 0.67 / 1.90, n = 144 0.73 / 0.75 / 1.11 / 3.68
    // against 0.87 / 0.89 / 1.25 / 3.40, n = 256 2.0 / 2.1 / 3.5 / 12.3 against 4.6 /
    // 5.1 / 7.7 / 18.9; C128 n = 130 1.78 / 1.81 / 3.20 / 10.4 against 1.43 / 1.51 / 2.35
    // / 7.96, n = 192 3.28 / 3.41 / 6.16 / 20.5 against 3.61 / 4.17 / 6.27 / 21.8.
    // Single precision keeps the unblocked order of its sums everywhere: the
    // log-value it accumulates in double shows every bit of them.
    if constexpr (sizeof(typename traits<T>::real) == 8) {
        int dev = 0, nsm = 148;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        const bool blocked = traits<T>::is_complex ? L.n_max >= 192 : L.n_max >= (L.W <= nsm ? 112 : 140);
        if (blocked) {
            go(k_slogpf<T, true>, sizeof(PfSmem<T>));
            return;
        }
    }
    go(k_slogpf<T, false>, 2 * (size_t)L.n_max * sizeof(T));
}

template <typename T>
void launch_slogdet(int W, int n, const T* A, T* ws, int nws, double* logabs, T* sgn, const uint8_t* mask,
                    cudaStream_t st) {
    const int dyn = (int)sizeof(GJSmem<T>);
    cudaFuncSetAttribute(k_slogdet<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    k_slogdet<T><<<nws, RT, dyn, st>>>(W, n, A, ws, logabs, sgn, mask);
}

template <typename T>
__global__ void __launch_bounds__(RT) k_gj_compact(int n, int nr, const T* A, T* M, const uint8_t* mask) {
    extern __shared__ __align__(16) unsigned char dsm[];
    GJSmem<T>& sm = *reinterpret_cast<GJSmem<T>*>(dsm);
    __shared__ int perm[2048];
    __shared__ double s_l;
    __shared__ T s_s;
    __shared__ int s_sing;
    const int w = blockIdx.x;
    if (!mask[w]) return;
    T* Mw = M + (long long)w * nr * nr;
    load_transposed(Mw, A + (long long)w * n * n, n, sm.tile);
    __syncthreads();
    gj_invert(Mw, n, perm, &s_l, &s_s, &s_sing, sm);
}

template <typename T>
void launch_gj_compact(int W, int n, int nr, const T* A, T* M, const uint8_t* mask, cudaStream_t st) {
    const int dyn = (int)sizeof(GJSmem<T>);
    cudaFuncSetAttribute(k_gj_compact<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    k_gj_compact<T><<<W, RT, dyn, st>>>(n, nr, A, M, mask);
}


// ---------------------------------------------------------------------------
// FP64 parts of the tensor-core refresh (the GEMM is in refresh_oz.cu)
// ---------------------------------------------------------------------------

// largest biased exponent of a scalar's parts (0x7ff: not finite)
__device__ __forceinline__ int bexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int bexp(c128 x) { return max(bexp(x.re), bexp(x.im)); }

// M[w] = A[w]^T (or A[w]) through 32 x 32 tiles, the identity in the padding,
// and (sort) the largest exponent of every row of M in Z.rmax (zeroed before);
// grid (nr/32, nr/32, W), block 32 x 8
template <typename T>
__global__ void k_oz_load(int n, int nr, const T* A, bool transpose, bool sort, OzWork Z, const uint8_t* mask) {
    __shared__ T tile[32][33];
    const int w = blockIdx.z;
    if (mask && !mask[w]) return;
    const T* Aw = A + (long long)w * n * n;
    T* M = reinterpret_cast<T*>(Z.M) + (long long)w * nr * nr;
    const int tx = threadIdx.x, r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;   // of M
    if (transpose) {
        for (int q = threadIdx.y; q < 32; q += 8) {
            const int r = c0 + q, c = r0 + tx;   // of A
            if (r < n && c < n) tile[tx][q] = Aw[(long long)r * n + c];
        }
        __syncthreads();
    }
    for (int q = threadIdx.y; q < 32; q += 8) {
        const int r = r0 + q, c = c0 + tx;
        T v = make_real<T>(r == c ? 1.0 : 0.0);
        const bool in = r < n && c < n;
        if (in) v = transpose ? tile[q][tx] : Aw[(long long)r * n + c];
        M[(long long)r * nr + c] = v;
        if (!sort) continue;
        const int e = __reduce_max_sync(0xffffffffu, in ? bexp(v) : 0);
        if (tx == 0 && e > 0) atomicMax(&Z.rmax[(long long)w * nr + r], e);
    }
}

// Which of the loaded walkers the split products take (go) and which are left
// to the FP64 form (odd): those with an entry that is not finite, with rows of
// very different size (a panel row's digits share one scale, so rows 2^s apart
// cost s bits) or with entries so large or small that a product of scales could
// leave the exponent range.  One warp per walker.
__global__ void k_oz_sort(int W, int n, int nr, OzWork Z, const uint8_t* mask) {
    const int w = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (w >= W) return;
    int hi = 0, lo = 0x7ff;
    for (int r = threadIdx.x & 31; r < n; r += 32) {
        const int e = Z.rmax[(long long)w * nr + r];
        hi = max(hi, e);
        lo = min(lo, e);
    }
    hi = __reduce_max_sync(0xffffffffu, hi);
    lo = __reduce_min_sync(0xffffffffu, lo);
    if ((threadIdx.x & 31) == 0) {
        const bool on = !mask || mask[w], fit = hi - lo <= 6 && hi < 1023 + 200 && hi > 1023 - 200;
        Z.go[w] = on && fit;
        Z.odd[w] = on && !fit;
    }
}

// One SW-column sub-panel of panel [k0, k0 + PB) (PB = 64 real or 32 complex
// columns) with the rows in registers (SW = 16 for nr <= 1024, 8 up to 2048;
// complex half of that): thread t owns rows t + q * blockDim (q < RPT,
// blockDim = nr / RPT); lu: only the rows from k0 on.  The sub-panel is eliminated in registers (pivot by a block reduction,
// row swaps through shared memory) and its transform columns written back;
// its row exchanges are then applied to the other panel columns, whose update
// by the transform is a split product on the tensor cores (refresh_oz.cu).
// The last sub-panel of a panel also applies the panel's exchanges, in pivot
// order, to the columns outside it.  Pivots go to Z.piv (log|det| and the
// sign are summed at the end).
template <typename T, int RPT, int SW>
__global__ void __launch_bounds__(512, 1) k_oz_subpanel_rows(int n, int k0, int sp, bool lu, OzWork Z,
                                                              const uint8_t* mask) {
    constexpr int CX = traits<T>::is_complex ? 2 : 1, PB = OZ_B / CX;
    static_assert(SW * CX % 2 == 0 && PB % SW == 0, "sub-panel width");
    __shared__ T s_rowk[SW], s_bufA[SW], s_bufB[SW];
    __shared__ unsigned long long s_wk[16];
    __shared__ int s_wi[16];
    __shared__ int s_src[2048], s_row[2 * SW];   // composed exchanges (n <= 2048)
    __shared__ int s_sing;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    const int w = blockIdx.x;
    if (mask && !mask[w]) return;
    T* M = reinterpret_cast<T*>(Z.M) + (long long)w * n * n;
    T* pivots = reinterpret_cast<T*>(Z.piv) + (long long)w * n;
    const int i_lo = lu ? k0 : 0;
    int* perm = Z.perm + (long long)w * n;
    if (tid == 0) s_sing = (k0 || sp) ? Z.sing[w] : 0;
    __syncthreads();
    {
        const int ks = k0 + SW * sp;
        constexpr int VL = 2 / CX;   // scalars per 16-byte load
        struct alignas(16) Pair { T e[VL]; };
        T v[RPT][SW];
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const Pair* src = reinterpret_cast<const Pair*>(M + (long long)(tid + q * nt) * n + ks);
            if (tid + q * nt < i_lo) continue;
#pragma unroll
            for (int c = 0; c < SW / VL; ++c) {
                const Pair x = src[c];
#pragma unroll
                for (int e = 0; e < VL; ++e) v[q][VL * c + e] = x.e[e];
            }
        }
#pragma unroll
        for (int kc = 0; kc < SW; ++kc) {
            const int k = ks + kc;
            // ---- pivot: largest |v| over rows >= k (ties: smallest row) ----
            // |v| is compared through its bit pattern (a non-negative double
            // orders like its bits as an unsigned integer), so the search runs on
            // the integer pipe and leaves the FP64 pipe to the elimination; NaN
            // counts as 0.  Every warp then reduces the per-warp winners itself,
            // so the pivot costs one barrier.
            unsigned long long bk = 0ull;
            int bi = -1;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int r = tid + q * nt;
                if (r < k) continue;
                double mag;
                if constexpr (CX == 1) mag = v[q][kc];
                else mag = s_abs2(v[q][kc]);
                unsigned long long a = (unsigned long long)__double_as_longlong(mag) & 0x7FFFFFFFFFFFFFFFull;
                if (a > 0x7FF0000000000000ull) a = 0ull;
                if (bi < 0 || a > bk) { bk = a; bi = r; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (oi >= 0 && (bi < 0 || ok > bk || (ok == bk && oi < bi))) { bk = ok; bi = oi; }
            }
            if (lane == 0) { s_wk[wid] = bk; s_wi[wid] = bi; }
            __syncthreads();
            bk = 0ull;
            bi = -1;
            for (int q = 0; q < nt / 32; ++q) {
                const unsigned long long ok = s_wk[q];
                const int oi = s_wi[q];
                if (oi >= 0 && (bi < 0 || ok > bk || (ok == bk && oi < bi))) { bk = ok; bi = oi; }
            }
            const int p = bi;
            if (bk == 0ull || p < 0) {
                if (tid == 0) { perm[k] = k; s_sing = 1; pivots[k] = s_zero(T()); }
                __syncthreads();   // every thread has read s_wk before the next pivot writes it
                continue;
            }
            if (tid == 0) perm[k] = p;
            const int tk = k % nt, qk = k / nt, tp = p % nt, qp = p / nt;
            // ---- rows p (the pivot row) and k to shared memory ----
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                if (tid == tp && q == qp)
#pragma unroll
                    for (int c = 0; c < SW; ++c) s_bufA[c] = v[q][c];
                if (p != k && tid == tk && q == qk)
#pragma unroll
                    for (int c = 0; c < SW; ++c) s_bufB[c] = v[q][c];
            }
            __syncthreads();
            // ---- scale the pivot row: 16 threads, one element each; the pivot
            //      is recorded (log|det| and the sign are summed at the end) ----
            if (tid < SW) {
                const T piv = s_bufA[kc], x = tid == kc ? make_real<T>(1.0) : s_bufA[tid];
                if constexpr (CX == 1) s_rowk[tid] = x / piv;
                else s_rowk[tid] = x * s_recip(piv);
                if (tid == 0) pivots[k] = piv;
            }
            __syncthreads();
            // ---- exchange: row k becomes the scaled pivot row, row p the old row k ----
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                if (tid == tk && q == qk)
#pragma unroll
                    for (int c = 0; c < SW; ++c) v[q][c] = s_rowk[c];
                else if (p != k && tid == tp && q == qp)
#pragma unroll
                    for (int c = 0; c < SW; ++c) v[q][c] = s_bufB[c];
            }
            // ---- eliminate column k from every other row ----
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int r = tid + q * nt;
                if (r != k && r >= i_lo) {
                    const T f = v[q][kc];
#pragma unroll
                    for (int c = 0; c < SW; ++c) v[q][c] = s_fms(f, s_rowk[c], c == kc ? s_zero(T()) : v[q][c]);
                }
            }
        }
        // ---- the sub-panel's transform columns back to M ----
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            Pair* dst = reinterpret_cast<Pair*>(M + (long long)(tid + q * nt) * n + ks);
            if (tid + q * nt < i_lo) continue;
#pragma unroll
            for (int c = 0; c < SW / VL; ++c) {
                Pair x;
#pragma unroll
                for (int e = 0; e < VL; ++e) x.e[e] = v[q][VL * c + e];
                dst[c] = x;
            }
        }
        __syncthreads();
        // ---- this sub-panel's exchanges on the other panel columns ----
        // The SW exchanges (k, perm[k]), applied in pivot order, move at most 2 SW
        // rows: row r receives the old row s_src[r].  All their elements are loaded
        // before any is stored (a loop of SW dependent swaps per column waits for
        // global memory SW times: 36.7 -> 34.8 ms of eliminations a refresh at 512 walkers,
        // n = 1024); a row listed twice is written twice alike.
        if (tid < SW) {
            const int k = ks + tid, p = perm[k];
            s_src[k] = k;
            s_src[p] = p;
            s_row[tid] = k;
            s_row[SW + tid] = p;
        }
        __syncthreads();
        if (tid == 0)
            for (int kc = 0; kc < SW; ++kc) {
                const int k = ks + kc, p = s_row[SW + kc], a = s_src[k];
                s_src[k] = s_src[p];
                s_src[p] = a;
            }
        __syncthreads();
        // elements in groups of four columns (a 32-byte sector of each row); a round of
        // 4 nt elements holds whole groups, and columns do not depend on one another
        constexpr int NB = PB - SW, NE = 2 * SW * NB;
        static_assert(NB % 4 == 0 && 128 % (8 * SW) == 0, "rounds of whole column groups");
        auto place = [&](int e, int& r, int& col) {
            const int rem = e % (8 * SW), t = e / (8 * SW) * 4 + rem % 4;
            r = rem / 4;
            col = k0 + t + (t >= SW * sp ? SW : 0);
        };
        for (int e0 = 0; e0 < NE; e0 += 4 * nt) {
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = e0 + tid + u * nt;
                int r, col;
                place(e, r, col);
                if (e < NE) x[u] = M[(long long)s_src[s_row[r]] * n + col];
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = e0 + tid + u * nt;
                int r, col;
                place(e, r, col);
                if (e < NE) M[(long long)s_row[r] * n + col] = x[u];
            }
        }
        __syncthreads();
    }
    // ---- last sub-panel: the panel's exchanges on the columns outside it ----
    // The 64 exchanges (k, perm[k]), applied in pivot order, compose into one
    // permutation of at most 128 rows: row r receives the old row src[r].  It
    // is built once in shared memory; then every 32-column tile of those rows
    // is gathered into shared memory (independent, coalesced loads) and
    // written back permuted, instead of 64 dependent swaps per column.
    if (sp == PB / SW - 1) {
        __shared__ int s_from[2 * PB], s_to[2 * PB];
        __shared__ int s_cnt;
        __shared__ T s_xb[2 * PB][33];
        for (int r = tid; r < n; r += nt) s_src[r] = r;
        if (tid == 0) s_cnt = 0;
        __syncthreads();
        if (tid == 0)
            for (int kc = 0; kc < PB; ++kc) {
                const int k = k0 + kc, p = perm[k];
                const int a = s_src[k];
                s_src[k] = s_src[p];
                s_src[p] = a;
            }
        __syncthreads();
        for (int r = tid; r < n; r += nt)
            if (s_src[r] != r) {
                const int e = atomicAdd(&s_cnt, 1);   // at most 2 * PB rows move
                s_to[e] = r;
                s_from[e] = s_src[r];
            }
        __syncthreads();
        const int cnt = s_cnt;
        for (int j0 = lu ? k0 + PB : 0; j0 < n && cnt > 0; j0 += 32) {
            if (j0 >= k0 && j0 < k0 + PB) continue;   // the panel's own columns (PB is a multiple of 32)
            // eight independent loads per thread in flight before any store
            for (int e0 = tid; e0 < cnt * 32; e0 += 8 * nt) {
                T x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int e = e0 + u * nt;
                    x[u] = e < cnt * 32 ? M[(long long)s_from[e >> 5] * n + j0 + (e & 31)] : s_zero(T());
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int e = e0 + u * nt;
                    if (e < cnt * 32) s_xb[e >> 5][e & 31] = x[u];
                }
            }
            __syncthreads();
            for (int e = tid; e < cnt * 32; e += nt) {
                const int q = e >> 5, jj = e & 31;
                M[(long long)s_to[q] * n + j0 + jj] = s_xb[q][jj];
            }
            __syncthreads();
        }
    }
    if (tid == 0) Z.sing[w] = s_sing;
}

// Undo the row exchanges of the elimination as one column permutation of
// the inverse (idx composes the swaps, last first: M'[i][c] = M[i][idx[c]]),
// four rows at a time through shared memory; then log|det|, sign and the
// fresh-state flags.
template <typename T>
__global__ void __launch_bounds__(RT) k_oz_finish(int n, int nr, bool permute, OzWork Z, const uint8_t* mask,
                                                  double* logabs, T* sgn, int* pst, int* tau) {
    extern __shared__ __align__(16) unsigned char dsm[];
    T* buf = reinterpret_cast<T*>(dsm);
    int* idx = reinterpret_cast<int*>(buf + 4 * n);
    __shared__ double s_sum[32];
    __shared__ T s_unit_part[RT];
    const int w = blockIdx.x;
    if (mask && !mask[w]) return;
    const int* perm = Z.perm + (long long)w * nr;
    if (permute) {
        for (int c = threadIdx.x; c < n; c += RT) idx[c] = c;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int k = n - 1; k >= 0; --k) {
                const int p = perm[k];
                if (p != k) { const int t = idx[k]; idx[k] = idx[p]; idx[p] = t; }
            }
        __syncthreads();
        T* M = reinterpret_cast<T*>(Z.M) + (long long)w * nr * nr;
        for (int i0 = 0; i0 < n; i0 += 4) {
            const int rows = min(4, n - i0);
            for (int r = 0; r < rows; ++r)
                for (int c = threadIdx.x; c < n; c += RT) buf[r * n + c] = M[(long long)(i0 + r) * nr + c];
            __syncthreads();
            for (int r = 0; r < rows; ++r)
                for (int c = threadIdx.x; c < n; c += RT) M[(long long)(i0 + r) * nr + c] = buf[r * n + idx[c]];
            __syncthreads();
        }
    }
    // log|det| = sum log|pivot|, sign = prod of the pivots' signs * (-1)^(row exchanges)
    const T* pv = reinterpret_cast<const T*>(Z.piv) + (long long)w * nr;
    double la = 0.0;
    T u = make_real<T>(1.0);
    for (int k = threadIdx.x; k < n; k += RT) {
        la += log(s_absd(pv[k]));
        u = u * s_unit(pv[k]);
        if (perm[k] != k) u = s_neg(u);
    }
    la = block_sum(la, s_sum);
    s_unit_part[threadIdx.x] = u;
    __syncthreads();
    for (int h = RT / 2; h > 0; h /= 2) {
        if (threadIdx.x < h) s_unit_part[threadIdx.x] = s_unit_part[threadIdx.x] * s_unit_part[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const int sing = Z.sing[w];
        if (logabs) logabs[w] = sing ? -INFINITY : la;
        if (sgn) sgn[w] = sing ? s_zero(T()) : s_renorm(s_unit_part[0]);
        if (Z.fail && *Z.fail) {   // a wait of the products gave up, and there is no handle to say so
            if (logabs) logabs[w] = NAN;
            if (sgn) sgn[w] = make_real<T>(NAN);
        }
        if (tau) tau[w] = 0;
        if (pst) pst[w] = sing ? 1 : 5;
    }
}

// M := (M - M^T) / 2, exactly skew, by 32 x 32 tiles (tJ <= tL); block 32 x 8
template <typename T>
__global__ void k_oz_skew(int n, int nr, T* M, const uint8_t* mask) {
    __shared__ T a[32][33], b[32][33];
    const int w = blockIdx.z;
    if ((mask && !mask[w]) || blockIdx.y > blockIdx.x) return;
    T* Mw = M + (long long)w * nr * nr;
    const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32, tx = threadIdx.x;
    for (int q = threadIdx.y; q < 32; q += 8) {
        if (i0 + q < n && j0 + tx < n) a[q][tx] = Mw[(long long)(i0 + q) * nr + j0 + tx];
        if (j0 + q < n && i0 + tx < n) b[q][tx] = Mw[(long long)(j0 + q) * nr + i0 + tx];
    }
    __syncthreads();
    for (int q = threadIdx.y; q < 32; q += 8) {
        // rows i < j get the half difference, rows j > i its exact negative
        if (i0 + q < n && j0 + tx < n && i0 + q < j0 + tx)
            Mw[(long long)(i0 + q) * nr + j0 + tx] = s_half(a[q][tx] - b[tx][q]);
        if (j0 + q < n && i0 + tx < n && i0 + tx <= j0 + q)
            Mw[(long long)(j0 + q) * nr + i0 + tx] =
                i0 + tx == j0 + q ? s_zero(T()) : s_neg(s_half(a[tx][q] - b[q][tx]));
    }
}

// The fresh inverses in M (rows of nr) become the state of walkers w0 + blockIdx.x;
// with drift, the relative Frobenius distance of the tracked inverse first (the
// delayed form's pending slots applied on the fly, A^{-1} = A_0^{-1} -/+ P Q^T).
// A warp per row, VR scalars per load, four loads of each stream in flight.
// (The column permutation stays in k_oz_finish: folded in here, through shared
// memory, the barriers between the rows cost 16 ms at 512 walkers, n = 1024,
// against 1.7 ms for its own pass.)
constexpr int ST = 1024;
template <typename T, int VR>
__global__ void __launch_bounds__(ST) k_oz_store(int w0, int n, int nr, DevLayout L, DevState<T> S, OzWork Z,
                                                 const uint8_t* mask, double* drift, bool delayed, bool pf) {
    struct alignas(VR * sizeof(T)) V { T e[VR]; };
    __shared__ double s_red[32];
    const int w = w0 + blockIdx.x;
    if (mask && !mask[blockIdx.x]) return;
    T* G = S.G + (long long)w * n * n;
    const T* Mw = reinterpret_cast<const T*>(Z.M) + (long long)blockIdx.x * nr * nr;
    const long long vo = (long long)w * n;
    const int cu = delayed ? S.tau[w] * L.kv(w) : 0, lane = threadIdx.x & 31;
    double num = 0.0, den = 0.0;
    for (int l = threadIdx.x >> 5; l < n; l += ST / 32) {
        const T* mrow = Mw + (long long)l * nr;   // [l][j] = (A^{-1})_{jl}
        T* grow = G + (long long)l * n;
#pragma unroll 4
        for (int j = lane * VR; j < n; j += 32 * VR) {
            const V f = *reinterpret_cast<const V*>(mrow + j);
            if (drift) {
                V tr = *reinterpret_cast<const V*>(grow + j);
#pragma unroll
                for (int r = 0; r < VR; ++r) {
                    if (cu) {
                        const T *pr = S.P + (vo + j + r) * L.Kc, *qr = S.Q + (vo + l) * L.Kc;
                        T sum = s_zero(T());
                        for (int c = 0; c < cu; ++c) sum = s_fma(pr[c], qr[c], sum);
                        tr.e[r] = pf ? tr.e[r] + sum : tr.e[r] - sum;
                    }
                    num += (double)s_abs2(tr.e[r] - f.e[r]);
                    den += (double)s_abs2(f.e[r]);
                }
            }
            *reinterpret_cast<V*>(grow + j) = f;
        }
    }
    if (drift) {
        num = block_sum(num, s_red);
        den = block_sum(den, s_red);
        if (threadIdx.x == 0) drift[w] = den > 0 ? sqrt(num / den) : 0.0;
    }
    if (delayed && threadIdx.x == 0) S.tau[w] = 0;
}

template <typename T>
void launch_oz_load(int W, int n, int nr, const T* A, bool transpose, bool sort, const OzWork& Z, const uint8_t* mask,
                    cudaStream_t st) {
    if (sort) cudaMemsetAsync(Z.rmax, 0, (size_t)W * nr * sizeof(int), st);
    k_oz_load<T><<<dim3(nr / 32, nr / 32, W), dim3(32, 8), 0, st>>>(n, nr, A, transpose, sort, Z, mask);
}

void launch_oz_sort(int W, int n, int nr, const OzWork& Z, const uint8_t* mask, cudaStream_t st) {
    k_oz_sort<<<(W + 7) / 8, 256, 0, st>>>(W, n, nr, Z, mask);
}

template <typename T> int oz_subpanel_width(int nr) { return (nr <= 1024 ? 16 : 8) / (traits<T>::is_complex ? 2 : 1); }

template <typename T>
void launch_oz_subpanel(int W, int nr, int k0, int sp, bool lu, const OzWork& Z, const uint8_t* mask, cudaStream_t st) {
    constexpr int CX = traits<T>::is_complex ? 2 : 1;
    if (nr <= 1024) k_oz_subpanel_rows<T, 2, 16 / CX><<<W, nr / 2, 0, st>>>(nr, k0, sp, lu, Z, mask);
    // (two rows per thread also below 512 rows: half as many threads, so two or more
    // CTAs share an SM and one computes while another waits for its pivot; with one
    // row the eliminations of 256 matrices, n = 500, took 10.0 ms instead of 6.1)
    // four rows of half as many sub-panel columns per thread keep the registers
    else k_oz_subpanel_rows<T, 4, 8 / CX><<<W, nr / 4, 0, st>>>(nr, k0, sp, lu, Z, mask);
}

template <typename T>
void launch_oz_finish(int W, int n, int nr, bool permute, const OzWork& Z, const uint8_t* mask, double* logabs, T* sgn,
                      int* pst, int* tau, cudaStream_t st) {
    const int dyn = (int)(4 * n * sizeof(T) + n * sizeof(int));
    cudaFuncSetAttribute(k_oz_finish<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    k_oz_finish<T><<<W, RT, dyn, st>>>(n, nr, permute, Z, mask, logabs, sgn, pst, tau);
}

template <typename T>
void launch_oz_skew(int W, int n, int nr, double* M, const uint8_t* mask, cudaStream_t st) {
    const int nt = (n + 31) / 32;
    k_oz_skew<T><<<dim3(nt, nt, W), dim3(32, 8), 0, st>>>(n, nr, reinterpret_cast<T*>(M), mask);
}

template <typename T>
void launch_oz_store(int W, int w0, int n, int nr, const DevLayout& L, const DevState<T>& S, const OzWork& Z,
                     const uint8_t* mask, double* drift, bool delayed, bool pf, cudaStream_t st) {
    if constexpr (!traits<T>::is_complex) {
        if (n % 2 == 0) {   // rows of both matrices start on 16-byte boundaries
            k_oz_store<T, 2><<<W, ST, 0, st>>>(w0, n, nr, L, S, Z, mask, drift, delayed, pf);
            return;
        }
    }
    k_oz_store<T, 1><<<W, ST, 0, st>>>(w0, n, nr, L, S, Z, mask, drift, delayed, pf);
}

#define LRU_INST_OZ(T)                                                                                       \
    template int oz_subpanel_width<T>(int);                                                                  \
    template void launch_gj_compact<T>(int, int, int, const T*, T*, const uint8_t*, cudaStream_t);           \
    template void launch_oz_load<T>(int, int, int, const T*, bool, bool, const OzWork&, const uint8_t*,       \
                                    cudaStream_t);                                                           \
    template void launch_oz_subpanel<T>(int, int, int, int, bool, const OzWork&, const uint8_t*, cudaStream_t);  \
    template void launch_oz_finish<T>(int, int, int, bool, const OzWork&, const uint8_t*, double*, T*, int*,     \
                                      int*, cudaStream_t);                                                   \
    template void launch_oz_skew<T>(int, int, int, double*, const uint8_t*, cudaStream_t);                   \
    template void launch_oz_store<T>(int, int, int, int, const DevLayout&, const DevState<T>&, const OzWork&, \
                                     const uint8_t*, double*, bool, bool, cudaStream_t);
LRU_INST_OZ(double)
LRU_INST_OZ(c128)

#define LRU_INST_R(T)                                                                                       \
    template void launch_refresh<T>(bool, bool, const DevLayout&, const DevState<T>&, const T*,            \
                                    const uint8_t*, T*, int, double*, bool, cudaStream_t);                 \
    template void launch_slogpf<T>(const DevLayout&, const T*, const uint8_t*, T*, int, double*, T*,       \
                                   cudaStream_t);                                                          \
    template void launch_slogdet<T>(int, int, const T*, T*, int, double*, T*, const uint8_t*, cudaStream_t);

LRU_INST_R(double)
LRU_INST_R(float)
LRU_INST_R(c128)
LRU_INST_R(c64)

}  // namespace lru

// ---------------------------------------------------------------------------
// slogdet without any allocation (lru_slogdet_batched_noalloc)
//
// Some callers cannot let a library allocate device memory: runtimes that
// preallocate most of the GPU for their own pool (so a cudaMalloc can fail),
// code that must not hit the device-wide synchronisation of cudaFree, and
// callers that record work for later replay.  This entry point runs the FP64
// Gauss-Jordan kernel at every size (lru_slogdet_batched takes split products for
// F64 / C128 of n = 56 .. 64 and n >= 72, so the two agree to rounding there), with
// its per-CTA matrix workspace taken from the fixed array below.
// ---------------------------------------------------------------------------

#include <mutex>
#include <stdint.h>

#include "../../include/lrugb.h"

namespace lru {

constexpr size_t NOALLOC_SCRATCH_BYTES = size_t(64) << 20;   // 64 MiB, held by every GPU that loads the library

// The workspace.  Host code may not use this name as a device address: the
// address comes from cudaGetSymbolAddress, per device, in noalloc_scratch().
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

// Device address of the workspace on the current device; looked up once per
// device, with that device current.  Returns nullptr if the lookup failed.
static void* noalloc_scratch(int dev) {
    constexpr int MAXDEV = 64;
    static std::mutex mu;
    static void* addr[MAXDEV] = {};
    static bool done[MAXDEV] = {};
    if (dev < 0 || dev >= MAXDEV) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!done[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;   // not cached: the next call tries again
        }
        addr[dev] = p;
        done[dev] = true;
    }
    return addr[dev];
}

}  // namespace lru

extern "C" lru_status lru_slogdet_batched_noalloc(int32_t dtype, int64_t W, int32_t n, const void* A,
                                                  double* logabs, void* sign, void* stream) {
    using namespace lru;
    size_t sz = 0;
    switch (dtype) {
        case LRU_F64: sz = 8; break;
        case LRU_C128: sz = 16; break;
        case LRU_F32: sz = 4; break;
        case LRU_C64: sz = 8; break;
        default: return LRU_ERR_ARG;
    }
    if (W < 1 || W > (int64_t)INT32_MAX || n < 1 || n > 2048 || !A || !logabs || !sign) return LRU_ERR_ARG;
    const size_t per = (size_t)n * n * sz;
    if (per > NOALLOC_SCRATCH_BYTES) return LRU_ERR_ARG;   // one matrix must fit the workspace
    int dev = 0, nsm = 148;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return LRU_ERR_CUDA; }
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        nsm = 148;
    }
    void* ws = noalloc_scratch(dev);
    if (!ws) return LRU_ERR_CUDA;
    long long slots = (long long)(NOALLOC_SCRATCH_BYTES / per);
    slots = std::min<long long>(slots, std::min<long long>(W, 2LL * nsm));
    cudaStream_t st = (cudaStream_t)stream;
    switch (dtype) {
        case LRU_F64: launch_slogdet<double>((int)W, n, (const double*)A, (double*)ws, (int)slots, logabs, (double*)sign, nullptr, st); break;
        case LRU_C128: launch_slogdet<c128>((int)W, n, (const c128*)A, (c128*)ws, (int)slots, logabs, (c128*)sign, nullptr, st); break;
        case LRU_F32: launch_slogdet<float>((int)W, n, (const float*)A, (float*)ws, (int)slots, logabs, (float*)sign, nullptr, st); break;
        case LRU_C64: launch_slogdet<c64>((int)W, n, (const c64*)A, (c64*)ws, (int)slots, logabs, (c64*)sign, nullptr, st); break;
    }
    return cudaGetLastError() == cudaSuccess ? LRU_OK : LRU_ERR_CUDA;
}
