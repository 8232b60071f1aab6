// Adjoint (vector-Jacobian product) of the log ratio of the pending proposal
// and of log|value|, for reverse-mode differentiation.
//
// Determinant (Sec. 2.1, Eqs. det_R, det_ratio): log r = log det R,
// R = I + V A^{-1} U.  With X = A^{-1} U and Y = V A^{-1},
//   d log r = tr(R^{-1} dR) = tr(R^{-1} (dV X + Y dU - Y dA X)),
// so dlogr/dU = (R^{-1} Y)^T, dlogr/dV = (X R^{-1})^T, dlogr/dA = -(X R^{-1} Y)^T.
// Pfaffian (App. A.2 Eq. pf_low_rank, App. A.3 Eq. pf_grad): log r =
// log pf M - log pf C^{-1}, M = C^{-1} + B^T A^{-1} B, d log pf M = tr(M^{-1} dM)/2
// for skew dM; with X = A^{-1} B and A^{-1}, M^{-1} skew:
//   dlogr/dB = X M^{-1},  dlogr/dA_ij = (X M^{-1} X^T)_ji / 2,
//   dlogr/dC = skew part of -[C^{-1} (M^{-1} - C) C^{-1}]^T / 2,
// where A and C enter through their skew parts (A - A^T)/2 as in App. A.3.
// log|value|: dlog det A / dA = A^{-T}; dlog pf A / dA_ij = (A^{-1})_ji / 2.
// For complex dtypes every output is the conjugate-Wirtinger vector-Jacobian
// product  g * conj(J)  that PyTorch's autograd expects for holomorphic maps.
// The delayed state never materialises A^{-1}: Y is recomputed from A_0^{-1}
// and the stored slots, Y = V A_0^{-1} - (V P) Q^T.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "passes.cuh"

#include <type_traits>

namespace lru {

constexpr int AT = 256;
constexpr int AMAXKK = 16;

template <typename T> __device__ __forceinline__ T s_conj(T a) { return a; }
template <> __device__ __forceinline__ c128 s_conj<c128>(c128 a) { return {a.re, -a.im}; }
template <> __device__ __forceinline__ c64 s_conj<c64>(c64 a) { return {a.re, -a.im}; }

template <typename T>
__device__ __forceinline__ const T* opvec(const DevOperand& O, const DevLayout& L, int w, int a, int n) {
    return reinterpret_cast<const T*>(O.dense) + (L.vo(w) * O.slots + (long long)a * n);
}

// gC = skew part of -[C^{-1} (M^{-1} - C) C^{-1}]^T / 2 of walker w (C = -J when
// C is null), by one thread; sR: M^{-1}.
template <typename T>
__device__ void backward_core(const T* Cw, int m, const T* sR, T gw, T* gCw) {
    T Cm[AMAXKK * AMAXKK], Ci[AMAXKK * AMAXKK], T1[AMAXKK * AMAXKK];
    for (int a = 0; a < m; ++a)
        for (int b = 0; b < m; ++b) {
            double v = (b == a + m / 2) ? -1.0 : ((a == b + m / 2) ? 1.0 : 0.0);   // -J
            Cm[a * AMAXKK + b] = Cw ? Cw[a * m + b] : make_real<T>(v);
        }
    // C^{-1} by Gauss-Jordan on a copy (small, m <= 16)
    for (int a = 0; a < m; ++a)
        for (int b = 0; b < m; ++b) Ci[a * AMAXKK + b] = Cm[a * AMAXKK + b];
    {
        int swp[AMAXKK];
        for (int k = 0; k < m; ++k) {
            int p = k;
            double best = (double)s_abs2(Ci[k * AMAXKK + k]);
            for (int i = k + 1; i < m; ++i)
                if ((double)s_abs2(Ci[i * AMAXKK + k]) > best) { best = (double)s_abs2(Ci[i * AMAXKK + k]); p = i; }
            swp[k] = p;
            if (p != k)
                for (int j = 0; j < m; ++j) {
                    T t = Ci[k * AMAXKK + j]; Ci[k * AMAXKK + j] = Ci[p * AMAXKK + j]; Ci[p * AMAXKK + j] = t;
                }
            T ip = s_recip(Ci[k * AMAXKK + k]);
            Ci[k * AMAXKK + k] = make_real<T>(1.0);
            for (int j = 0; j < m; ++j) Ci[k * AMAXKK + j] = Ci[k * AMAXKK + j] * ip;
            for (int i = 0; i < m; ++i) {
                if (i == k) continue;
                T f = Ci[i * AMAXKK + k];
                Ci[i * AMAXKK + k] = s_zero(T());
                for (int j = 0; j < m; ++j) Ci[i * AMAXKK + j] = s_fms(f, Ci[k * AMAXKK + j], Ci[i * AMAXKK + j]);
            }
        }
        for (int k = m - 1; k >= 0; --k)
            if (swp[k] != k)
                for (int i = 0; i < m; ++i) {
                    T t = Ci[i * AMAXKK + k]; Ci[i * AMAXKK + k] = Ci[i * AMAXKK + swp[k]]; Ci[i * AMAXKK + swp[k]] = t;
                }
    }
    // T1 = (M^{-1} - C) C^{-1}; then G = C^{-1} T1
    for (int a = 0; a < m; ++a)
        for (int b = 0; b < m; ++b) {
            T s = s_zero(T());
            for (int c = 0; c < m; ++c) s = s_fma(sR[a * AMAXKK + c] - Cm[a * AMAXKK + c], Ci[c * AMAXKK + b], s);
            T1[a * AMAXKK + b] = s;
        }
    for (int a = 0; a < m; ++a)
        for (int b = 0; b < m; ++b) {
            // unconstrained gradient entry (a, b) = -[C^{-1} T1]_{b a} / 2
            T sba = s_zero(T()), sab = s_zero(T());
            for (int c = 0; c < m; ++c) {
                sba = s_fma(Ci[b * AMAXKK + c], T1[c * AMAXKK + a], sba);
                sab = s_fma(Ci[a * AMAXKK + c], T1[c * AMAXKK + b], sab);
            }
            // skew part: (G_ab - G_ba) / 2 with G_ab = -sba / 2, G_ba = -sab / 2
            T v = s_half(s_half(sab - sba));
            gCw[a * m + b] = gw * s_conj(v);
        }
}

// gC of every walker, a thread each: where there are more walkers than SMs, beside
// k_backward, whose CTAs would wait for one thread of theirs (1024 walkers, n = 34, F64
// two-particle moves: 160 us with the core inside, 67 beside; 64 walkers 38 and 43)
template <typename T>
__global__ void __launch_bounds__(32) k_backward_core(DevLayout L, DevState<T> S, const T* C, const T* g, T* gC) {
    const int w = blockIdx.x * 32 + threadIdx.x;
    if (w >= L.W) return;
    const int kk = L.kv(w);
    T* gCw = gC + (long long)w * L.kk * L.kk;
    if (S.pst[w] != 0) {
        for (int e = 0; e < kk * kk; ++e) gCw[e] = s_zero(T());
        return;
    }
    backward_core<T>(C ? C + (long long)w * L.kk * L.kk : nullptr, kk, S.Rinv + (long long)w * AMAXKK * AMAXKK, g[w], gCw);
}

// |g| |x| far inside the range (2^-900 .. 2^900, single precision 2^-100 .. 2^100), by
// the exponents of the larger parts, or x = 0
__device__ __forceinline__ int part_exponent(double x) { return (__double2hiint(x) >> 20 & 0x7ff) - 1023; }
__device__ __forceinline__ int part_exponent(float x) { return (__float_as_int(x) >> 23 & 0xff) - 127; }
template <typename R>
__device__ __forceinline__ int part_exponent(cplx<R> x) { return max(part_exponent(x.re), part_exponent(x.im)); }
template <typename R> __device__ __forceinline__ bool is_zero(R x) { return x == R(0); }
template <typename R> __device__ __forceinline__ bool is_zero(cplx<R> x) { return x.re == R(0) && x.im == R(0); }
template <typename T>
__device__ __forceinline__ bool product_in_range(T g, T x) {
    constexpr int lim = sizeof(typename traits<T>::real) == 8 ? 900 : 100;
    const int e = part_exponent(g) + part_exponent(x);
    return (e >= -lim && e <= lim) || is_zero(x);
}

template <typename T>
struct BackSmem {
    YSmem<T> y;                  // det: Y of the item's columns, then its rows of the outer product
    T R[AMAXKK * AMAXKK];
    T VP[AMAXKK * 64];
    T out[AMAXKK][YC];           // the item's rows, conjugated: R^{-1} Y (det) or X M^{-1} (pf)
    int iv[AMAXKK];
};

// One CTA per work item (walker, columns [l0, l1) of A^{-1}), in blocks of YC.
// The gradient of A is the outer product of two rank-kk factors, n^2 outputs
// that nothing but the store should bound: a thread keeps the kk values of its
// column j in registers and walks the block's rows, whose factors are in
// shared memory, so the stores are coalesced and every factor is read once per
// block.
//   det: T = R^{-1} Y;  gU = g conj(T), gV = g conj(X R^{-1}),
//        gA[i][j] = -g conj(sum_a X_a[j] T[a][i])
//   pf : Z = X M^{-1};  gB = g conj(Z), gA[i][j] = -g conj(sum_b Z[i][b] X_b[j]) / 2
template <typename T, bool PF, bool DELAYED, int KBM>
__global__ void __launch_bounds__(AT, 2) k_backward(DevLayout L, DevState<T> S, DevOperand Vop, const T* C, const T* g,
                                                     T* gU, T* gV, T* gA, T* gC, const int4* items) {
    extern __shared__ __align__(16) unsigned char dsm[];
    BackSmem<T>& sm = *reinterpret_cast<BackSmem<T>*>(dsm);
    const int4 it = items[blockIdx.x];
    const int w = it.x;
    if (!LRU_DEBUG_OK(w >= 0 && w < L.W, S.err)) return;
    const int n = L.nw(w), kk = L.kv(w);
    if (!LRU_DEBUG_OK(it.y >= 0 && it.y <= it.z && it.z <= n, S.err)) return;
    const long long vo = L.vo(w);
    const int slots = L.kk;
    T* gUw = gU ? gU + vo * slots : nullptr;
    T* gVw = gV ? gV + vo * slots : nullptr;
    T* gAw = gA ? gA + L.mo(w) : nullptr;
    const int rows = it.z - it.y;
    if (S.pst[w] != 0) {
        // no pending proposal with a valid core: zero gradient
        for (int e = threadIdx.x; e < kk * rows; e += AT) {
            const int a = e / rows, j = it.y + e - a * rows;
            if (gUw) gUw[(long long)a * n + j] = s_zero(T());
            if (gVw) gVw[(long long)a * n + j] = s_zero(T());
        }
        if (gAw)
            for (long long e = threadIdx.x; e < (long long)rows * n; e += AT) gAw[(long long)it.y * n + e] = s_zero(T());
        if (PF && gC && it.y == 0 && threadIdx.x < kk * kk)
            gC[(long long)w * L.kk * L.kk + threadIdx.x] = s_zero(T());
        return;
    }
    const T gw = g[w];
    const T* X = S.X + vo * L.kk;             // kk vectors of n: X[a*n + j] = (A^{-1} U)_{j a}
    for (int e = threadIdx.x; e < kk * kk; e += AT) {
        const int a = e / kk, b = e - a * kk;
        sm.R[a * AMAXKK + b] = S.Rinv[(long long)w * AMAXKK * AMAXKK + a * AMAXKK + b];
    }
    if (threadIdx.x < kk)
        sm.iv[threadIdx.x] = ((Vop.mask >> threadIdx.x) & 1u) ? Vop.idx[(long long)w * Vop.slots + threadIdx.x] : -1;
    const int cu = DELAYED ? S.tau[w] * kk : 0;
    if constexpr (DELAYED && !PF)
        for (int e = threadIdx.x; e < kk * cu; e += AT) {
            const int b = e / cu, c = e - b * cu;
            sm.VP[b * 64 + c] = S.VP[(long long)w * AMAXKK * L.Kc + b * L.Kc + c];
        }
    __syncthreads();
    if (PF && gC && it.y == 0 && threadIdx.x == 0)
        backward_core<T>(C ? C + (long long)w * L.kk * L.kk : nullptr, kk, sm.R, gw, gC + (long long)w * L.kk * L.kk);

    for (int l0 = it.y; l0 < it.z; l0 += YC) {
        const int nc = min(YC, it.z - l0);
        if constexpr (!PF) {
            if (gUw || gAw) {
                const T* Vw = Vop.dense ? opvec<T>(Vop, L, w, 0, n) : nullptr;
                dense_y_cols<T, KBM>(S.G + L.mo(w), n, l0, nc, Vw, sm.iv, kk, sm.y);
                if (cu > 0) slot_correct_y<T>(S.Q + vo * L.Kc, L.Kc, cu, l0, nc, sm.VP, kk, sm.y);
            }
        }
        // this block's rows of the left factor, and the operand gradients
        for (int e = threadIdx.x; e < kk * nc; e += AT) {
            const int a = e / nc, c = e - a * nc, j = l0 + c;
            T t = s_zero(T()), z = s_zero(T());
            for (int b = 0; b < kk; ++b) {
                if constexpr (!PF) {
                    if (gUw || gAw) t = s_fma(sm.R[a * AMAXKK + b], sm.y.y[b][c], t);
                }
                z = s_fma(X[(long long)b * n + j], sm.R[b * AMAXKK + a], z);
            }
            sm.out[a][c] = s_conj(PF ? z : t);
            if (PF) {
                if (gUw) gUw[(long long)a * n + j] = gw * s_conj(z);
            } else {
                if (gUw) gUw[(long long)a * n + j] = gw * s_conj(t);
                if (gVw) gVw[(long long)a * n + j] = gw * s_conj(z);
            }
        }
        __syncthreads();
        if (gAw) {
            const T gs = PF ? s_half(s_neg(gw)) : s_neg(gw);
            // fewer columns than threads: the rows go to several groups of n threads
            const int stride = min(n, AT), groups = AT / stride, grp = (int)threadIdx.x / stride;
            auto column = [&](int j, auto one_group) {
                T x[KBM];
                // Where g X stays far inside the range, g goes into the n kk factors and
                // not the n^2 outputs: 551 against 611 us for the orbital gradient of 512
                // walkers, n = 256, which the FP64 pipe bounds.  Otherwise it multiplies
                // the finished sum.
                bool late = kk > KBM;
#pragma unroll
                for (int b = 0; b < KBM; ++b) {
                    x[b] = b < kk ? s_conj(X[(long long)b * n + j]) : s_zero(T());
                    late = late || !product_in_range(gs, x[b]);
                }
                constexpr bool one = decltype(one_group)::value;
                auto rows = [&](auto after) {
#pragma unroll 4
                    for (int c = one ? 0 : grp; c < nc; c += one ? 1 : groups) {
                        T s = s_zero(T());
#pragma unroll
                        for (int b = 0; b < KBM; ++b)
                            if (b < kk) s = s_fma(x[b], sm.out[b][c], s);
                        if constexpr (decltype(after)::value) {
                            for (int b = KBM; b < kk; ++b) s = s_fma(s_conj(X[(long long)b * n + j]), sm.out[b][c], s);
                            s = gs * s;
                        }
                        gAw[(long long)(l0 + c) * n + j] = s;
                    }
                };
                if (late) {
                    rows(std::true_type());
                } else {
#pragma unroll
                    for (int b = 0; b < KBM; ++b) x[b] = gs * x[b];
                    rows(std::false_type());
                }
            };
            if (groups == 1)
                for (int j = threadIdx.x; j < n; j += AT) column(j, std::true_type());
            else if (grp < groups)
                column((int)threadIdx.x - grp * stride, std::false_type());
        }
        __syncthreads();
    }
}

// gA = g A^{-T} (det) or g A^{-T}/2 = -g A^{-1}/2 (pf), conjugated for complex;
// A^{-1} = A_0^{-1} -/+ P Q^T for the delayed state.  Row-major output.
template <typename T, bool PF, bool DELAYED>
__global__ void k_backward_logvalue(DevLayout L, DevState<T> S, const T* g, T* gA) {
    const int w = blockIdx.y;
    const int n = L.nw(w), kk = L.kv(w);
    const long long vo = L.vo(w);
    const T* Gw = S.G + L.mo(w);
    T* out = gA + L.mo(w);
    const T gw = g[w];
    const int cu = DELAYED ? S.tau[w] * kk : 0;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n * n;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e % n);
        // (A^{-T})_{ij} = (A^{-1})_{ji}, stored at column-major position [i*n + j] = e
        T v = Gw[e];
        if (DELAYED && cu) {
            const T* pr = S.P + (vo + j) * L.Kc;
            const T* qr = S.Q + (vo + i) * L.Kc;
            T s = s_zero(T());
            for (int c = 0; c < cu; ++c) s = s_fma(pr[c], qr[c], s);
            v = PF ? v + s : v - s;
        }
        v = gw * s_conj(v);
        out[e] = PF ? s_half(v) : v;
    }
}

// log of the stored ratios: real dtypes log|r|, complex the principal log r
template <typename T>
__global__ void k_log_ratio(int W, const T* ratio, T* out) {
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= W) return;
    const T r = ratio[w];
    if constexpr (traits<T>::is_complex) {
        using R = typename traits<T>::real;
        out[w] = T{(R)log(s_absd(r)), (R)atan2((double)r.im, (double)r.re)};
    } else {
        out[w] = (T)log(s_absd(r));
    }
}

// gPhi[rows[w][i]][:] += gA[w][i][:] (atomic; rows shared between walkers)
template <typename T>
__global__ void k_scatter_rows(DevLayout L, const T* gA, const int* rows, int m, T* gPhi, int* err) {
    const int w = blockIdx.y;
    const int n = L.n_uni;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < (long long)n * n;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e % n);
        const int r = rows[(long long)w * n + i];
        if (r < 0 || r >= m) { set_dev_error(err, DEV_ERR_INDEX); continue; }
        const T v = gA[(long long)w * n * n + e];
        if constexpr (traits<T>::is_complex) {
            atomicAdd(&gPhi[(long long)r * n + j].re, v.re);
            atomicAdd(&gPhi[(long long)r * n + j].im, v.im);
        } else {
            atomicAdd(&gPhi[(long long)r * n + j], v);
        }
    }
}

template <typename T, int KBM>
static void launch_backward_k(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const DevOperand& V,
                              const T* C, const T* g, T* gU, T* gV, T* gA, T* gC, const int4* items, int nitems,
                              cudaStream_t st) {
    auto kern = pf ? (delayed ? k_backward<T, true, true, KBM> : k_backward<T, true, false, KBM>)
                   : (delayed ? k_backward<T, false, true, KBM> : k_backward<T, false, false, KBM>);
    const int dyn = (int)sizeof(BackSmem<T>);
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);
    kern<<<nitems, AT, dyn, st>>>(L, S, V, C, g, gU, gV, gA, gC, items);
}

template <typename T>
void launch_backward(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const DevOperand& V,
                     const T* C, const T* g, T* gU, T* gV, T* gA, T* gC, const int* items, int nitems,
                     bool core_beside, cudaStream_t st) {
    const int4* it = reinterpret_cast<const int4*>(items);
    if (pf && gC && core_beside) {
        k_backward_core<T><<<(L.W + 31) / 32, 32, 0, st>>>(L, S, C, g, gC);
        gC = nullptr;
    }
    if (L.kk == 1) launch_backward_k<T, 1>(pf, delayed, L, S, V, C, g, gU, gV, gA, gC, it, nitems, st);
    else if (L.kk == 2) launch_backward_k<T, 2>(pf, delayed, L, S, V, C, g, gU, gV, gA, gC, it, nitems, st);
    else if (L.kk <= 4) launch_backward_k<T, 4>(pf, delayed, L, S, V, C, g, gU, gV, gA, gC, it, nitems, st);
    else launch_backward_k<T, kb_max<T>()>(pf, delayed, L, S, V, C, g, gU, gV, gA, gC, it, nitems, st);
}

template <typename T>
void launch_backward_logvalue(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const T* g, T* gA,
                              cudaStream_t st) {
    dim3 grid(64, L.W);
    if (!pf && !delayed) k_backward_logvalue<T, false, false><<<grid, 256, 0, st>>>(L, S, g, gA);
    if (!pf && delayed) k_backward_logvalue<T, false, true><<<grid, 256, 0, st>>>(L, S, g, gA);
    if (pf && !delayed) k_backward_logvalue<T, true, false><<<grid, 256, 0, st>>>(L, S, g, gA);
    if (pf && delayed) k_backward_logvalue<T, true, true><<<grid, 256, 0, st>>>(L, S, g, gA);
}

template <typename T>
void launch_log_ratio(int W, const T* ratio, T* out, cudaStream_t st) {
    k_log_ratio<T><<<(W + 255) / 256, 256, 0, st>>>(W, ratio, out);
}

template <typename T>
void launch_scatter_rows(const DevLayout& L, const T* gA, const int* rows, int m, T* gPhi, int* err, cudaStream_t st) {
    dim3 grid(64, L.W);
    k_scatter_rows<T><<<grid, 256, 0, st>>>(L, gA, rows, m, gPhi, err);
}

// Gradient of the outputs (sign or phase s, log|value|) of the batched
// slogdet / slogpf: with t = tr(A^{-1} dA), d log|det A| = Re t and
// d s = i s Im t, so for a loss L with dL/dlog|.| = g_l and dL/ds = g_s (torch's
// convention for complex) dL = Re(conj(c) t), c = g_l + i beta,
// beta = -Im(conj(g_s) s), and grad_A = c A^{-H} (real: g_l A^{-T}).  The
// Pfaffian has log pf = (1/2) log det of the skew part (App. A.3, Eq.
// pf_grad): grad_A = (c / 2) (skew part of A^{-1})^H.  Ginv: the column-major
// inverses, Ginv[w][l n + j] = (A_w^{-1})_{jl}, so (A^{-H})_{ij} is
// conj(Ginv[w][i n + j]).
template <typename T>
__global__ void k_slog_grad(int W, int n, int nr, bool pf, const T* Ginv, const uint8_t* compact, const int* fail,
                            const double* g_l, const T* g_s, const T* sign, T* gA) {
    const bool failed = fail && *fail;
    const long long nn = (long long)n * n, total = nn * W;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int w = (int)(e / nn);
        const long long r = e - (long long)w * nn;
        const int i = (int)(r / n), j = (int)(r - (long long)i * n);
        const T* G = Ginv + (long long)w * nr * nr;
        const bool own = compact && compact[w];   // inverted by the FP64 form
        const int ld = own ? n : nr;
        T c = make_real<T>(g_l ? g_l[w] : 0.0);
        if constexpr (traits<T>::is_complex) {
            if (g_s) {
                const T q = s_conj(g_s[w]) * sign[w];
                c.im = -q.im;
            }
        }
        T v = G[(long long)i * ld + j];
        if (pf) v = s_half(s_half(v - G[(long long)j * ld + i]));   // (1/2) of the skew part
        gA[e] = failed && !own ? make_real<T>(NAN) : c * s_conj(v);
    }
}

template <typename T>
void launch_slog_grad(int W, int n, int nr, bool pf, const T* Ginv, const uint8_t* compact, const int* fail,
                      const double* g_l, const T* g_s, const T* sign, T* gA, cudaStream_t st) {
    const long long total = (long long)n * n * W;
    const int grid = (int)std::min<long long>((total + 255) / 256, 152 * 16);
    k_slog_grad<T><<<grid, 256, 0, st>>>(W, n, nr, pf, Ginv, compact, fail, g_l, g_s, sign, gA);
}

#define LRU_INST_A(T)                                                                                        \
    template void launch_slog_grad<T>(int, int, int, bool, const T*, const uint8_t*, const int*, const double*, const T*,     \
                                      const T*, T*, cudaStream_t);                                            \
    template void launch_backward<T>(bool, bool, const DevLayout&, const DevState<T>&, const DevOperand&,     \
                                     const T*, const T*, T*, T*, T*, T*, const int*, int, bool, cudaStream_t); \
    template void launch_backward_logvalue<T>(bool, bool, const DevLayout&, const DevState<T>&, const T*, T*, \
                                              cudaStream_t);                                                  \
    template void launch_log_ratio<T>(int, const T*, T*, cudaStream_t);                                       \
    template void launch_scatter_rows<T>(const DevLayout&, const T*, const int*, int, T*, int*, cudaStream_t);

LRU_INST_A(double)
LRU_INST_A(float)
LRU_INST_A(c128)
LRU_INST_A(c64)

}  // namespace lru
