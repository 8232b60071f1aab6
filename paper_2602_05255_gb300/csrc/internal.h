// Internal interface between the C-ABI (lrugb_api.cu) and the kernel
// translation units.  Not part of the public ABI.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lru {

// Per-walker geometry, as seen by kernels.  Walker w has an n_w x n_w
// inverse starting at element moff(w) (sum of n_v^2 before it) and length-n_w
// vectors starting at voff(w) (sum of n_v before it) times the slot count.
struct DevLayout {
    int W;
    int n_uni;                 // > 0: every walker has this n (moff, voff computed)
    int n_max;                 // largest n (workspace slot size n_max^2)
    const int* n;              // per-walker n (ragged)
    const long long* moff;
    const long long* voff;
    int kk;                    // vector slots per update (det: k, pf: 2k), max over walkers
    const int* kvec;           // per-walker vector count, or nullptr (= kk)
    int Kc;                    // delay columns per walker row of P, Q (K * kk), 0 if plain
    int K;                     // delay length (>= 2 for the delayed form)
    int Kc32;                  // row stride (elements) of the split copies: Kc rounded up to 32 (TF32) or 64 (BF16)
    long long rows;            // sum of n over walkers (rows of P, Q)
    __device__ __forceinline__ int nw(int w) const { return n_uni > 0 ? n_uni : n[w]; }
    __device__ __forceinline__ long long mo(int w) const {
        return n_uni > 0 ? (long long)w * n_uni * n_uni : moff[w];
    }
    __device__ __forceinline__ long long vo(int w) const {
        return n_uni > 0 ? (long long)w * n_uni : voff[w];
    }
    __device__ __forceinline__ int kv(int w) const { return kvec ? kvec[w] : kk; }
};

// Per-walker state and proposal scratch (one device allocation).
template <typename T>
struct DevState {
    T* G;          // A^{-1} (plain) or A_0^{-1} (delayed), column-major per walker
    T* P;          // delayed: n_w x Kc per walker, row j contiguous
    T* Q;
    int split_bf16;  // 0: the split copies are TF32 in fp32 words; 1: bf16
    float* P32h;   // delayed, tensor-core flush: split copies of P and Q (K-major rows of Kc32)
    float* P32l;
    float* Q32h;
    float* Q32l;
    int* tau;      // filled delay slots per walker
    double* logabs;
    T* sgn;        // sign (real) or unit phase (complex)
    // scratch of the last proposal
    T* X;          // A^{-1} U (det) or A^{-1} B (pf): kk vectors of n_w
    T* Rinv;       // kk x kk per walker: R^{-1} (det) or M^{-1} (pf)
    T* ratio;      // W
    int* pst;      // W proposal status
    T* VP;         // det delayed: V P (MAXKK x Kc per walker)
    int* err;      // sticky device error word
};

struct DevOperand {
    const void* dense;
    const int* idx;
    unsigned mask;   // bit a: slot a is one-hot
    int slots;       // vector slots per walker in the buffers (kmax)
};

// rows of X per work item of the persistent step (XT in passes.cuh)
constexpr int STEP_X_ROWS = 64;

// Dense columns of U for small matrices: the propose's own CTA sums X = A^{-1} U, a
// thread per row, instead of a pass that spreads it over the chip.  Up to
// x_inline_rows for every proposal (that pass is a launch of its own: one F32 walker,
// n = 4, k = 4, 14.7 us a propose with it, 11.4 without; complex128 pays for a longer
// chain per row: 1024 walkers of n = 16 42 and 48 us).
constexpr int x_inline_rows(size_t scalar) { return scalar == 16 ? 8 : 32; }
// In the persistent step also, in single precision, for one dense column of up to a
// row per thread while every walker's CTA has an SM to itself: handing the tiles
// around costs more than it spreads (64 walkers, delayed, rank 1, complex64: n = 64
// 37 / 32 us a step with tiles / in the CTA, n = 256 63 / 54).
inline bool step_x_inline(int n_max, size_t scalar, int dense, int W, int n_sm, bool single) {
    return n_max <= x_inline_rows(scalar) || (single && dense == 1 && W <= n_sm && n_max <= 256);
}

// Control block of the persistent fused step (see k_step).
struct StepCtl {
    int* counter;             // work-queue head, zeroed before each launch
    int* x_done;              // W counters of finished X tiles (zeroed)
    const int2* x_items;      // X tiles (walker, row block), largest walkers first
    int n_x_items;            // 0: every column of U is one-hot, or the propose sums them itself
    int* prop_done;           // W flags, zeroed before each launch
    int* items_done;          // W counters, zeroed before each launch
    int* fin;                 // W flags: the walker's propose, accept and commit are done (zeroed)
    int* flush_done;          // W counters of finished flush strips (zeroed)
    uint8_t* acc;             // W accept decisions (output)
    const int* order;         // W walkers in propose order
    const int4* acc_items;    // accept items (walker, l0, l1, use_smem), largest walkers first
    const int* nacc_w;        // accept items per walker
    int nacc;
    const int2* flush_items;  // delayed form: flush strips (walker, 32-column block), largest walkers first
    const int* nflush_w;      // flush strips per walker
    int nflush;
    int do_accept;            // 0: propose only
    const uint8_t* mask;      // optional acceptance mask
    const double* u;          // optional Metropolis uniforms: accept if |r|^2 >= u
};

// ---- launchers (defined in lru_kernels.cu, instantiated for every dtype) ----
// df: the pass over A^{-1} for a single dense column in double-float arithmetic (F64 only)
template <typename T>
void launch_propose(bool pf, bool delayed, bool df, const DevLayout& L, const DevState<T>& S, const DevOperand& U,
                    const DevOperand& V, const T* C, T* ratio_out, int* st_out, cudaStream_t st);
template <typename T>
// df: the delayed rank-1 determinant GEMV in double-float arithmetic (F64 only)
void launch_accept(bool pf, bool delayed, bool df, const DevLayout& L, const DevState<T>& S, const DevOperand& V,
                   const uint8_t* mask, const int* items, int nitems, cudaStream_t st);
template <typename T>
void launch_flush_native(bool pf, const DevLayout& L, const DevState<T>& S, const uint8_t* force_mask,
                         int nwalkers_tiles, cudaStream_t st);
void launch_flush_df(bool pf, const DevLayout& L, const DevState<double>& S, const uint8_t* force_mask,
                     cudaStream_t st);
template <typename T>
void launch_flush_finish(const DevLayout& L, const DevState<T>& S, const uint8_t* force_mask, cudaStream_t st);
template <typename T>
void launch_get_inverse(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, T* out, cudaStream_t st);
template <typename T>
void launch_form_row_moves(const DevLayout& L, const T* Phi, int m, const int* occ, const int* slot,
                           const int* newrow, T* Vout, int* idx, cudaStream_t st);
template <typename T>
void launch_form_pf_moves(const DevLayout& L, const T* F, int m, const int* pos, const int* slot,
                          const int* newsite, T* Bout, int* idx, cudaStream_t st);
template <typename T>
void launch_gather(bool pairs, const DevLayout& L, const T* src, int m, const int* occ, T* A, int* err,
                   cudaStream_t st);
template <typename T>
void launch_step(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const DevOperand& U,
                 const DevOperand& V, const T* C, T* ratio_out, int* st_out, const StepCtl& ctl, int grid,
                 cudaStream_t st);
template <typename T>
void launch_zero_split_tail(const DevLayout& L, const DevState<T>& S, const uint8_t* force, cudaStream_t st);
// ---- refresh with the trailing updates on the tensor cores (refresh_oz.cu) ----
constexpr int OZ_B = 64;   // panel width = inner dimension of each trailing update
constexpr int OZ_S = 7;    // BF16 slices per operand (8 bits each: 56 bits)
struct OzWork {
    double* M;        // W x nr x nc row-major working matrix (M = A^T, inverted in place)
    int* perm;        // W x nr pivot rows
    int* sing;        // W zero-pivot flags
    uint16_t* Sb;     // W x OZ_S x nc x OZ_B  BF16 slices of the columns of S (panel rows of M)
    uint16_t* Pb;     // W x OZ_S x nr x OZ_B  BF16 slices of the rows of (panel - E)
    int* eS;          // W x nc power-of-two exponents of the S columns
    int* eP;          // W x nr power-of-two exponents of the panel rows
    uint8_t* go;      // W      walkers that flush now (split-product flush), or that this form inverts
    uint8_t* odd;     // W      walkers whose matrix is left to the FP64 form (see k_oz_sort)
    double* piv;      // W x nr scalars: pivots (log|det| and sign at the end)
    int* rmax;        // W x nr largest biased exponent of each row of M
    int* fail;        // the error word of a call without a handle (its results become NaN), or NULL
};
// columns a split-product update writes: [c_lo, c_hi) minus [s_lo, s_hi), in
// the 128-column tiles jt_lo .. jt_hi - 1 (doubles), rows from tile it_lo on; a
// walker's M is rows x ld (the padded sizes of the slices, or the state's own);
// the row tiles are cut into rsplit parts
struct OzCols {
    int c_lo, c_hi, s_lo, s_hi, jt_lo, jt_hi, it_lo, rows, ld, rsplit;
};
// rows of the working matrix of an n x n inverse: n padded by the identity
int oz_rows(int n);
// The sizes eliminated on padded copies (rows in steps of 64): below 56 a padded
// panel, and between 64 and 72 the padding, costs more than the products gain.
constexpr bool oz_padded(int n) { return n >= 72 || (n >= 56 && n <= 64); }
// For the determinant alone (LU form) and complex scalars that is the whole rule:
// 1 / 1024 matrices, FP64 form (one CTA per matrix) against padded, ms: F64 LU n = 60
// 0.54 / 2.3 against 0.45 / 1.2, n = 72 0.85 / 4.0 against 0.78 / 2.7; C128 inverse n = 56
// 0.81 / 4.4 against 0.68 / 2.1, n = 72 2.0 / 11.9 against 1.4 / 6.1.  The inverse of F64
// matrices is as fast in the FP64 form while its CTAs still fill one wave: n = 56 ..
// 62 up to one per SM (n = 60, 1 / 152 / 228 walkers: 0.38 / 0.39 / 0.51 against 0.39 /
// 0.41 / 0.46), n = 72 .. 79, padded to 128, up to two (n = 76, 1 / 304 / 456: 0.73 / 1.16
// / 2.27 against 0.80 / 1.26 / 1.53; n = 80 0.89 / 1.33 / 2.64 against 0.79 / 1.26 / 1.54).
inline bool oz_padded_inverse(int n, int cx, long long W, int n_sm) {
    return oz_padded(n) && (cx == 2 || n >= 80 || n == 63 || n == 64 || W > (n < 64 ? 1 : 2) * (long long)n_sm);
}
// bytes of the workspace of W walkers of nr rows (cx = 2: complex), and its parts when Z is given
size_t oz_work_layout(OzWork* Z, void* base, int W, int nr, int cx, bool with_M);
// M[w] = A[w]^T (or A[w]) with an identity in rows and columns n .. nr - 1
template <typename T>
void launch_oz_load(int W, int n, int nr, const T* A, bool transpose, bool sort, const OzWork& Z, const uint8_t* mask,
                    cudaStream_t st);
// sorts the loaded walkers with mask[w] into Z.go and Z.odd
void launch_oz_sort(int W, int n, int nr, const OzWork& Z, const uint8_t* mask, cudaStream_t st);
// one sub-panel of the panel at column k0: elimination and its row exchanges on the
// other panel columns; the last one of a panel also exchanges the outside columns
template <typename T> int oz_subpanel_width(int nr);
template <typename T>
void launch_oz_subpanel(int W, int nr, int k0, int sp, bool lu, const OzWork& Z, const uint8_t* mask, cudaStream_t st);
template <typename T>
bool oz_eliminate(int W, int nr, const OzWork& Z, const uint8_t* mask, bool lu, int* err, cudaStream_t st,
                  void (*hook)(void*, int, int), void* hctx);
// permute: the row exchanges undone as a column permutation of M's rows 0 .. n - 1;
// then log|det|, sign (and status, tau := 0, where given)
template <typename T>
void launch_oz_finish(int W, int n, int nr, bool permute, const OzWork& Z, const uint8_t* mask, double* logabs, T* sgn,
                      int* pst, int* tau, cudaStream_t st);
// M := (M - M^T) / 2 exactly skew, n x n of rows of nr
template <typename T>
void launch_oz_skew(int W, int n, int nr, double* M, const uint8_t* mask, cudaStream_t st);
// the state of walkers w0 .. := the inverses in M (rows of nr), with the drift of the tracked ones when asked for
template <typename T>
void launch_oz_store(int W, int w0, int n, int nr, const DevLayout& L, const DevState<T>& S, const OzWork& Z,
                     const uint8_t* mask, double* drift, bool delayed, bool pf, cudaStream_t st);
// delayed flush A_0^{-1} += sgnQ * P Q^T (determinant: -1, Pfaffian: +1) as the
// same exact split product (uniform n, K kk <= 64 doubles a row, kv: ranks of the
// walkers, NULL: kk each; Z of oz_flush_rows(n)
// rows, Z.M the state); walkers with tau >= K, or force && tau > 0
constexpr int oz_flush_rows(int n) { return (n + 63) / 64 * 64; }
template <typename T>
bool launch_flush_split(int W, int n, int K, int kk, const int* kv, const T* P, const T* Q, double sgnQ, const int* tau,
                        const uint8_t* force, const OzWork& Z, int* err, cudaStream_t st);
// A_0^{-1} of the same walkers: the lower triangle := the exact negative of the
// upper, diagonal 0 (after the Pfaffian split-product flush)
template <typename T>
void launch_skew_project(int W, int n, int K, T* G, const int* tau, const uint8_t* force, cudaStream_t st);
// hook(ctx, class, begin) brackets the panel (class 4) and update (class 5) launches
bool launch_refresh_oz(int W, int n, const double* A, const OzWork& Z, const DevState<double>& S,
                       const uint8_t* mask, bool delayed, bool in_state, int* err, cudaStream_t st,
                       void (*hook)(void*, int, int), void* hctx);
void launch_wait_selftest(const int* flag, long long iters, int* err, cudaStream_t st);
void launch_commit_moves(int W, int n, int k, int* occ, const int* slot, const int* newrow, const uint8_t* mask,
                         const int* pst, cudaStream_t st);
template <typename T>
void launch_set_delay_zero(const DevLayout& L, const DevState<T>& S, cudaStream_t st);

// ---- refresh / dense (refresh.cu) ----
// For each selected walker: G := A^{-1} (column-major) by Gauss-Jordan on A^T,
// log|det| and sign into S (write_logdet), tau := 0.  With ws (nws slots of
// n_uni^2 scalars) the inverse is formed in the CTA's slot first and the drift
// of the tracked inverse against it is written before it replaces G.
template <typename T>
void launch_refresh(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const T* A,
                    const uint8_t* mask, T* ws, int nws, double* drift, bool write_logdet, cudaStream_t st);
// Pfaffian (Parlett-Reid) of the selected walkers' A into logabs / sgn; ws: nws slots.
template <typename T>
void launch_slogpf(const DevLayout& L, const T* A, const uint8_t* mask, T* ws, int nws, double* logabs, T* sgn,
                   cudaStream_t st);
template <typename T>
void launch_slogdet(int W, int n, const T* A, T* ws, int nws, double* logabs, T* sgn, const uint8_t* mask,
                    cudaStream_t st);
// M (slots of nr^2 scalars) of the masked walkers := the Gauss-Jordan inverse of A^T as n rows of n
template <typename T>
void launch_gj_compact(int W, int n, int nr, const T* A, T* M, const uint8_t* mask, cudaStream_t st);

// ---- adjoint (adjoint.cu) ----
template <typename T>
void launch_backward(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const DevOperand& V,
                     const T* C, const T* g, T* gU, T* gV, T* gA, T* gC, const int* items, int nitems,
                     bool core_beside, cudaStream_t st);
template <typename T>
void launch_backward_logvalue(bool pf, bool delayed, const DevLayout& L, const DevState<T>& S, const T* g, T* gA,
                              cudaStream_t st);
template <typename T>
void launch_log_ratio(int W, const T* ratio, T* out, cudaStream_t st);
// gradient of (sign, log|det|) or (phase, log|pf|) from the column-major inverses
// (slots of nr^2 scalars, rows of nr; of n where compact[w]); NaN, except where
// compact[w], if the word fail (NULL: none) is set
template <typename T>
void launch_slog_grad(int W, int n, int nr, bool pf, const T* Ginv, const uint8_t* compact, const int* fail,
                      const double* g_l, const T* g_s, const T* sign, T* gA, cudaStream_t st);
template <typename T>
void launch_scatter_rows(const DevLayout& L, const T* gA, const int* rows, int m, T* gPhi, int* err, cudaStream_t st);

// ---- tensor-core flush (flush_tc.cu) ----
// Returns false when the combination is not built.
bool launch_flush_tc(int mode, bool pf, const DevLayout& L, double* G, const void* Ph, const void* Pl,
                     const void* Qh, const void* Ql, const int* tau, const uint8_t* force_mask,
                     int* err, cudaStream_t st);

}  // namespace lru
