// Relaxation and test-vector kernels: omega-Jacobi SpMM over row-interleaved blocks of
// test vectors (Section 3, Eq. (3.1)), the shifted sweeps of Algorithm 3, the LS
// weights of Section 3.2, Rayleigh-quotient updates, injection and prolongation of
// vector blocks, and the construction of B = I - A.
#include <cfloat>

#include <algorithm>
#include <array>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <vector>

#include "kernels.cuh"

namespace bamg {

// ---------------------------------------------------------------- initial vectors
template <typename T>
__global__ void k_tv_init(int n, int ncols, int ld, int col0, uint64_t seed, double lo, double hi, T* X) {
    pdl_begin();
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * ncols) return;
    int i = (int)(t / ncols);
    int k = (int)(t - (int64_t)i * ncols);
    double u = counter_uniform(seed, STREAM_TV + (uint64_t)k, (uint64_t)i);
    double v = __dadd_rn(lo, __dmul_rn(hi - lo, u));
    X[(int64_t)i * ld + col0 + k] = (T)v;
}

template <typename T>
void launch_tv_init(int n, int ncols, int ld, int col0, uint64_t seed, double lo, double hi, T* X, cudaStream_t s) {
    int64_t work = (int64_t)n * ncols;
    if (work == 0) return;
    BAMG_LAUNCH(k_tv_init<T>, blocks_for(work, 256), 256, 0, s, n, ncols, ld, col0, seed, lo, hi, X);
}

// ---------------------------------------------------------------- diagonals
template <typename T>
__global__ void k_diag(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const T* __restrict__ v,
                       T* __restrict__ d) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T x = T(0);
    for (int p = rp[i]; p < rp[i + 1]; ++p)
        if (ci[p] == i) {
            x = v[p];
            break;
        }
    d[i] = x;
}
template <typename T>
void launch_diag_vals(int n, const int32_t* rp, const int32_t* ci, const T* vals, T* d, cudaStream_t s) {
    if (n) BAMG_LAUNCH(k_diag<T>, blocks_for(n, 256), 256, 0, s, n, rp, ci, vals, d);
}
template <typename T>
void launch_diag(const MatView<T>& M, T* d, cudaStream_t s) {
    launch_diag_vals<T>(M.n, M.rp, M.ci, M.v, d, s);
}

// diag(B), diag(T) (when tv != null) and 1 / diag(B) in one pass
template <typename T>
__global__ void k_diagonals(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                            const T* __restrict__ bv, const T* __restrict__ tv, T* __restrict__ dB, T* __restrict__ dT,
                            T* __restrict__ dinv) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T b = T(0), t = T(0);
    for (int p = rp[i]; p < rp[i + 1]; ++p)
        if (ci[p] == i) {
            b = bv[p];
            if (tv) t = tv[p];
            break;
        }
    dB[i] = b;
    if (tv) dT[i] = t;
    dinv[i] = T(1) / b;
}
template <typename T>
void launch_diagonals(int n, const int32_t* rp, const int32_t* ci, const T* bv, const T* tv, T* dB, T* dT, T* dinv,
                      cudaStream_t s) {
    if (n) BAMG_LAUNCH(k_diagonals<T>, blocks_for(n, 256), 256, 0, s, n, rp, ci, bv, tv, dB, dT, dinv);
}

template <typename T>
__global__ void k_reciprocal(int n, const T* d, T* dinv) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dinv[i] = T(1) / d[i];
}
template <typename T>
void launch_reciprocal(int n, const T* d, T* dinv, cudaStream_t s) {
    if (n) BAMG_LAUNCH(k_reciprocal<T>, blocks_for(n, 256), 256, 0, s, n, d, dinv);
}

template <typename T>
__global__ void k_identity_on_pattern(int n, const int32_t* rp, const int32_t* ci, T* tv) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int p = rp[i]; p < rp[i + 1]; ++p) tv[p] = (ci[p] == i) ? T(1) : T(0);
}
template <typename T>
void launch_identity_on_pattern(int n, const int32_t* rp, const int32_t* ci, T* tv, cudaStream_t s) {
    if (n) BAMG_LAUNCH(k_identity_on_pattern<T>, blocks_for(n, 256), 256, 0, s, n, rp, ci, tv);
}

// ---------------------------------------------------------------- omega-Jacobi SpMM
// One thread owns one 16-byte chunk (W columns) of a row: it walks the row of B once,
// gathering the matching chunk of each neighbour's test-vector row (contiguous in the
// row-interleaved layout), so the W columns share every matrix load.  The grid is a
// fixed number of blocks per SM that strides over the rows; while a row's gathers are in
// flight the thread loads the next row's first JB column indices and values and the row
// pointers of the row after it, so the three dependent loads of a row (row pointers,
// entries, gathers) overlap with earlier rows' work.  Entries beyond the first JB of a
// row are read in predicated batches of JB; JB is 5 for matrices with at most five
// entries per row on average (grid walks, tandem queues), else 6.
//
// DIAG: the diagonal arrays are not there yet.  The sweep finds the row's diagonal among the entries
// it reads anyway, and stores it (1 / b_ii, or b_ii and t_ii for the shifted sweep) for the sweeps
// after it.  A pass of its own over the matrix and one over the diagonal took 61 us of a four-sweep
// call of 650 us on 2048 x 2048 states.  FP32 only: every thread of a row divides, which the FP64
// pipe does not repeat for nothing.
constexpr int JAC_BLOCKS_PER_SM = 2;

template <typename T, bool SHIFT, int JB, int CPT, bool DIAG>
__global__ void __launch_bounds__(256, JAC_BLOCKS_PER_SM)
    k_jacobi(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const T* __restrict__ bv,
             const T* __restrict__ tv, T* __restrict__ dB, T* __restrict__ dinvB, T* __restrict__ dT,
             const double* __restrict__ lam, int ncols, const T* __restrict__ X, T* __restrict__ Y, int ld, int col0,
             int nvec, T omega) {
    pdl_begin();
    constexpr int W = V16<T>::W;
    constexpr int CW = CPT * W;         // columns per thread
    constexpr int NT = SHIFT ? JB : 1;  // T values are carried only by the shifted sweep
    const int tpr = nvec / CPT;         // threads per row
    const int64_t stride = (int64_t)gridDim.x * blockDim.x / tpr;  // rows per pass of the grid
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= stride * tpr) return;
    int64_t row = t / tpr;
    if (row >= n) return;
    const int ch = (int)(t - row * tpr);
    const int off = col0 + ch * CW;
    const bool has_t = SHIFT && tv != nullptr;
    int p0 = __ldg(rp + row), p1 = __ldg(rp + row + 1);
    int cnt = min(JB, p1 - p0);
    int jj[JB];
    T bb[JB], tt[NT];
#pragma unroll
    for (int u = 0; u < JB; ++u)
        if (u < cnt) {
            jj[u] = __ldg(ci + p0 + u);
            bb[u] = __ldg(bv + p0 + u);
            if (has_t) tt[u < NT ? u : 0] = __ldg(tv + p0 + u);
        }
    int64_t nrow = row + stride;
    int np0 = 0, np1 = 0;
    if (nrow < n) {
        np0 = __ldg(rp + nrow);
        np1 = __ldg(rp + nrow + 1);
    }
    for (;;) {
        // this row's gathers, its own values and diagonal terms ...
        T xv[JB][CW];
#pragma unroll
        for (int u = 0; u < JB; ++u)
            if (u < cnt)
#pragma unroll
                for (int q = 0; q < CPT; ++q) V16<T>::load(X + (int64_t)jj[u] * ld + off + q * W, xv[u] + q * W);
        T xs[CW];
#pragma unroll
        for (int q = 0; q < CPT; ++q) V16<T>::load(X + row * ld + off + q * W, xs + q * W);
        T d0 = DIAG ? T(0) : SHIFT ? __ldg(dB + row) : __ldg(dinvB + row);
        T d1 = DIAG && has_t ? T(0) : has_t ? __ldg(dT + row) : T(1);
        // ... while the next row's first entries and the row pointers after it arrive
        const int ncnt = nrow < n ? min(JB, np1 - np0) : 0;
        int njj[JB];
        T nbb[JB], ntt[NT];
#pragma unroll
        for (int u = 0; u < JB; ++u)
            if (u < ncnt) {
                njj[u] = __ldg(ci + np0 + u);
                nbb[u] = __ldg(bv + np0 + u);
                if (has_t) ntt[u < NT ? u : 0] = __ldg(tv + np0 + u);
            }
        const int64_t nnrow = nrow + stride;
        int nnp0 = 0, nnp1 = 0;
        if (nnrow < n) {
            nnp0 = __ldg(rp + nnrow);
            nnp1 = __ldg(rp + nnrow + 1);
        }
        T acc[CW], accT[CW];
#pragma unroll
        for (int e = 0; e < CW; ++e) acc[e] = accT[e] = T(0);
        if constexpr (CPT > 1) {  // the rest of a long row, one entry at a time (registers)
            for (int p = p0 + JB; p < p1; ++p) {
                const int j = __ldg(ci + p);
                const T b = __ldg(bv + p);
                const T tq = has_t ? __ldg(tv + p) : T(0);
                if (DIAG && j == row) {
                    d0 = b;
                    if (has_t) d1 = tq;
                }
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    T xq[W];
                    V16<T>::load(X + (int64_t)j * ld + off + q * W, xq);
#pragma unroll
                    for (int e = 0; e < W; ++e) {
                        acc[q * W + e] += b * xq[e];
                        if (has_t) accT[q * W + e] += tq * xq[e];
                    }
                }
            }
        }
        for (int base = p0 + JB; CPT == 1 && base < p1; base += JB) {  // the rest of a long row, JB at a time
            const int c2 = min(JB, p1 - base);
            int kj[JB];
            T kb[JB], kt[NT], kx[JB][CW];
#pragma unroll
            for (int u = 0; u < JB; ++u)
                if (u < c2) {
                    kj[u] = __ldg(ci + base + u);
                    kb[u] = __ldg(bv + base + u);
                    if (has_t) kt[u < NT ? u : 0] = __ldg(tv + base + u);
                }
#pragma unroll
            for (int u = 0; u < JB; ++u)
                if (u < c2)
#pragma unroll
                    for (int q = 0; q < CPT; ++q) V16<T>::load(X + (int64_t)kj[u] * ld + off + q * W, kx[u] + q * W);
#pragma unroll
            for (int u = 0; u < JB; ++u)
                if (u < c2) {
                    if (DIAG && kj[u] == row) {
                        d0 = kb[u];
                        if (has_t) d1 = kt[u < NT ? u : 0];
                    }
#pragma unroll
                    for (int e = 0; e < CW; ++e) acc[e] += kb[u] * kx[u][e];
                    if (has_t)
#pragma unroll
                        for (int e = 0; e < CW; ++e) accT[e] += kt[u < NT ? u : 0] * kx[u][e];
                }
        }
#pragma unroll
        for (int u = 0; u < JB; ++u)
            if (u < cnt) {
                if (DIAG && jj[u] == row) {
                    d0 = bb[u];
                    if (has_t) d1 = tt[u < NT ? u : 0];
                }
#pragma unroll
                for (int e = 0; e < CW; ++e) acc[e] += bb[u] * xv[u][e];
                if (has_t)
#pragma unroll
                    for (int e = 0; e < CW; ++e) accT[e] += tt[u < NT ? u : 0] * xv[u][e];
            }
        if (DIAG) {
            if (!SHIFT) d0 = T(1) / d0;
            if (ch == 0) {
                (SHIFT ? dB : dinvB)[row] = d0;
                if (has_t) dT[row] = d1;
            }
        }
        T y[CW];
        if (SHIFT) {
#pragma unroll
            for (int e = 0; e < CW; ++e) {
                const int c = ch * CW + e;
                const T l = c < ncols ? (T)lam[c] : T(0);
                const T tx = has_t ? accT[e] : xs[e];
                const T r = acc[e] - l * tx;
                const T d = d0 - l * d1;
                y[e] = xs[e] - omega * r / d;
            }
        } else {
#pragma unroll
            for (int e = 0; e < CW; ++e) y[e] = xs[e] - omega * (d0 * acc[e]);
        }
#pragma unroll
        for (int q = 0; q < CPT; ++q) V16<T>::store(Y + row * ld + off + q * W, y + q * W);
        if (nrow >= n) break;
        row = nrow;
        p0 = np0;
        p1 = np1;
        cnt = ncnt;
#pragma unroll
        for (int u = 0; u < JB; ++u) {
            jj[u] = njj[u];
            bb[u] = nbb[u];
        }
#pragma unroll
        for (int u = 0; u < NT; ++u) tt[u] = ntt[u];
        nrow = nnrow;
        np0 = nnp0;
        np1 = nnp1;
    }
}

static int sm_count() {
    static int nsm = 0;
    if (nsm == 0) {
        int dev = 0, v = 0;
        BAMG_CK(cudaGetDevice(&dev));
        BAMG_CK(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
        nsm = v > 0 ? v : 1;
    }
    return nsm;
}

template <typename T>
__global__ void k_copy_cols(int n, const T* __restrict__ src, T* __restrict__ dst, int ld, int col0, int nvec) {
    pdl_begin();
    constexpr int W = V16<T>::W;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int row = (int)(t / nvec);
    if (row >= n) return;
    int ch = (int)(t - (int64_t)row * nvec);
    T v[W];
    V16<T>::load(src + (int64_t)row * ld + col0 + ch * W, v);
    V16<T>::store(dst + (int64_t)row * ld + col0 + ch * W, v);
}

// One sweep of the launch shape (chunks per thread, blocks per SM of the grid): Y from X.
template <typename T>
static void jacobi_sweep(const MatView<T>& B, const T* T_val, T* dB, T* dinvB, T* dT, const double* d_lambda, int ncols,
                         int ld, int col0, T omega, int nvec, bool short_rows, int cpt, int bps, bool diag, const T* X,
                         T* Y, cudaStream_t s) {
    const unsigned grid = (unsigned)std::min<int64_t>(blocks_for((int64_t)B.n * (nvec / cpt), 256),
                                                      (int64_t)sm_count() * bps);
    auto go = [&](auto kern) {
        BAMG_LAUNCH(kern, grid, 256, 0, s, B.n, B.rp, B.ci, B.v, T_val, dB, dinvB, dT, d_lambda, ncols, X, Y, ld, col0, nvec,
                    omega);
    };
#define BAMG_JAC(SH, JBV, CP)                          \
    do {                                              \
        if constexpr (sizeof(T) == 4)                 \
            if (diag) {                               \
                go(k_jacobi<T, SH, JBV, CP, true>);   \
                break;                                \
            }                                         \
        go(k_jacobi<T, SH, JBV, CP, false>);          \
    } while (0)
    const int variant = (d_lambda ? 4 : 0) + (cpt == 2 ? 2 : 0) + (short_rows ? 0 : 1);
    switch (variant) {
        case 0: BAMG_JAC(false, 5, 1); break;
        case 1: BAMG_JAC(false, 6, 1); break;
        case 2: BAMG_JAC(false, 5, 2); break;
        case 3: BAMG_JAC(false, 6, 2); break;
        case 4: BAMG_JAC(true, 5, 1); break;
        case 5: BAMG_JAC(true, 6, 1); break;
        case 6: BAMG_JAC(true, 5, 2); break;
        default: BAMG_JAC(true, 6, 2); break;
    }
#undef BAMG_JAC
}

// ---------------------------------------------------------------- launch-shape autotuner
// The sweep's launch shape (one or two 16-byte chunks per thread; one, two or four blocks
// per SM in the grid) changes how the rows are spread over the GPU, never the arithmetic:
// every shape writes the same bits.  On levels large enough for the shape to matter (more
// than four rows per thread of the one-chunk grid), the first sweep of each (precision,
// shift, entry batch, chunks per row, size class log2 n) times the shapes on the caller's
// own data with CUDA events (X -> work, X untouched) and keeps the fastest for the
// process.  BAMG_AUTOTUNE=0 keeps the fixed rule (two chunks when they pair up, two blocks
// per SM).
struct JacShape {
    int cpt, bps;
};
static bool autotune_enabled() {
    static const bool on = [] {
        const char* e = std::getenv("BAMG_AUTOTUNE");
        return !(e && std::strcmp(e, "0") == 0);
    }();
    return on;
}
static std::mutex& tune_mutex() {
    static std::mutex m;
    return m;
}
static std::map<std::array<int, 5>, JacShape>& tune_cache() {
    static std::map<std::array<int, 5>, JacShape> c;
    return c;
}
// the cached choices as (key..., cpt, bps) rows, for reports and tests
int jacobi_tuned_shapes(int* out, int max_rows) {
    std::lock_guard<std::mutex> lock(tune_mutex());
    int k = 0;
    for (const auto& kv : tune_cache()) {
        if (k >= max_rows) break;
        for (int q = 0; q < 5; ++q) out[7 * k + q] = kv.first[q];
        out[7 * k + 5] = kv.second.cpt;
        out[7 * k + 6] = kv.second.bps;
        ++k;
    }
    return k;
}

template <typename T>
void relax(const MatView<T>& B, const T* T_val, T* dB, T* dinvB, T* dT, const double* d_lambda, int ncols, int ld,
           int col0, T omega, int nu, T* X, T* work, cudaStream_t s, bool tune, bool diag) {
    constexpr int W = V16<T>::W;
    const int nvec = (ncols + W - 1) / W;
    if (B.n == 0 || nvec == 0 || nu <= 0) return;
    const int64_t work_items = (int64_t)B.n * nvec;
    const bool short_rows = (int64_t)B.nnz <= 5 * (int64_t)B.n;
    // small levels: one chunk per thread, two blocks per SM (the shorter per-thread work is
    // faster there); large levels: the fixed rule or the tuned shape
    const int64_t grid_threads = (int64_t)sm_count() * JAC_BLOCKS_PER_SM * 256;
    const bool large = work_items > 4 * grid_threads;
    JacShape shape{(large && nvec % 2 == 0) ? 2 : 1, JAC_BLOCKS_PER_SM};
    if (large && tune && autotune_enabled()) {
        int lg = 0;
        while ((int64_t(1) << (lg + 1)) <= B.n) ++lg;
        const std::array<int, 5> key{(int)sizeof(T), d_lambda ? 1 : 0, short_rows ? 5 : 6, nvec, lg};
        std::lock_guard<std::mutex> lock(tune_mutex());
        auto it = tune_cache().find(key);
        if (it != tune_cache().end()) {
            shape = it->second;
        } else {
            std::vector<JacShape> cand{{1, 2}, {1, 4}};
            if (nvec % 2 == 0) cand.insert(cand.end(), {{2, 1}, {2, 2}, {2, 4}});
            cudaEvent_t e0, e1;
            BAMG_CK(cudaEventCreate(&e0));
            BAMG_CK(cudaEventCreate(&e1));
            float best = 0.f;
            for (const JacShape& c : cand) {
                jacobi_sweep<T>(B, T_val, dB, dinvB, dT, d_lambda, ncols, ld, col0, omega, nvec, short_rows, c.cpt,
                                c.bps, diag, X, work, s);  // warm-up
                BAMG_CK(cudaEventRecord(e0, s));
                for (int r = 0; r < 3; ++r)
                    jacobi_sweep<T>(B, T_val, dB, dinvB, dT, d_lambda, ncols, ld, col0, omega, nvec, short_rows, c.cpt,
                                    c.bps, false, X, work, s);
                BAMG_CK(cudaEventRecord(e1, s));
                BAMG_CK(cudaEventSynchronize(e1));
                float ms = 0.f;
                BAMG_CK(cudaEventElapsedTime(&ms, e0, e1));
                if (&c == &cand[0] || ms < best) {
                    best = ms;
                    shape = c;
                }
            }
            cudaEventDestroy(e0);
            cudaEventDestroy(e1);
            tune_cache()[key] = shape;
        }
    }
    T* src = X;
    T* dst = work;
    for (int k = 0; k < nu; ++k) {
        jacobi_sweep<T>(B, T_val, dB, dinvB, dT, d_lambda, ncols, ld, col0, omega, nvec, short_rows, shape.cpt,
                        shape.bps, diag && k == 0, src, dst, s);
        T* t = src;
        src = dst;
        dst = t;
    }
    if (src != X) BAMG_LAUNCH(k_copy_cols<T>, blocks_for(work_items, 256), 256, 0, s, B.n, src, X, ld, col0, nvec);
}

// ---------------------------------------------------------------- column statistics
// MODE 0: (sum x^2, sum (Bx)^2) per column; MODE 1: (sum x (Bx), sum x (Tx)).
// Block (nvec x ny): threads own chunks of rows in a grid-stride loop; per-thread sums
// in T, then a fixed-order tree in FP64 per block, then a fixed-order sum over blocks.
template <typename T, int MODE>
__global__ void k_colstats(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                           const T* __restrict__ bv, const T* __restrict__ tv, const T* __restrict__ X, int ld,
                           int col0, int nvec, double* __restrict__ partial, unsigned* __restrict__ ticket) {
    pdl_begin();
    constexpr int W = V16<T>::W;
    extern __shared__ double sh[];
    const int ch = threadIdx.x, ry = threadIdx.y, ny = blockDim.y;
    if (blockIdx.x == 0 && ch == 0 && ry == 0) *ticket = 0u;  // for the kernel that adds up the partials
    const int off = col0 + ch * W;
    T s0[W], s1[W];
#pragma unroll
    for (int e = 0; e < W; ++e) s0[e] = s1[e] = T(0);
    for (int row = blockIdx.x * ny + ry; row < n; row += gridDim.x * ny) {
        T acc[W], accT[W];
#pragma unroll
        for (int e = 0; e < W; ++e) acc[e] = accT[e] = T(0);
        for (int p = rp[row]; p < rp[row + 1]; ++p) {
            const int j = ci[p];
            T xv[W];
            V16<T>::load(X + (int64_t)j * ld + off, xv);
            const T b = bv[p];
#pragma unroll
            for (int e = 0; e < W; ++e) acc[e] += b * xv[e];
            if (MODE == 1 && tv != nullptr) {
                const T tt = tv[p];
#pragma unroll
                for (int e = 0; e < W; ++e) accT[e] += tt * xv[e];
            }
        }
        T xs[W];
        V16<T>::load(X + (int64_t)row * ld + off, xs);
#pragma unroll
        for (int e = 0; e < W; ++e) {
            if (MODE == 0) {
                s0[e] += xs[e] * xs[e];
                s1[e] += acc[e] * acc[e];
            } else {
                s0[e] += xs[e] * acc[e];
                s1[e] += xs[e] * (tv ? accT[e] : xs[e]);
            }
        }
    }
    const int base = (ry * nvec + ch) * 2 * W;
#pragma unroll
    for (int e = 0; e < W; ++e) {
        sh[base + e] = (double)s0[e];
        sh[base + W + e] = (double)s1[e];
    }
    __syncthreads();
    for (int stride = ny >> 1; stride > 0; stride >>= 1) {
        if (ry < stride) {
            const int o = ((ry + stride) * nvec + ch) * 2 * W;
            for (int q = 0; q < 2 * W; ++q) sh[base + q] += sh[o + q];
        }
        __syncthreads();
    }
    if (ry == 0)
        for (int q = 0; q < 2 * W; ++q) partial[(int64_t)blockIdx.x * (nvec * 2 * W) + ch * 2 * W + q] = sh[base + q];
}


// Workspace of one column-statistics pair of kernels: the partials, the sums and a ticket.
struct ColWork {
    double *partial, *sums;
    unsigned* ticket;
    static size_t doubles(int nb, int width) { return (size_t)nb * width + width + 1; }
    ColWork(double* p, int nb, int width)
        : partial(p), sums(p + (size_t)nb * width), ticket(reinterpret_cast<unsigned*>(p + (size_t)nb * width + width)) {}
};
// Column statistics of Eq. (3.4) / the Rayleigh quotients as per-block partial sums
// (nb rows of `width` values in `partial`); the consumer forms the sums with
// colsum_partials.  Returns nb.
template <typename T>
static int colstats_blocks(int n, int ncols, int* width) {
    constexpr int W = V16<T>::W;
    const int nvec = (ncols + W - 1) / W;
    int ny = 1;
    while (ny * 2 * nvec <= 256) ny *= 2;
    int nb = (int)blocks_for(n, ny);
    // the consumers sum the partials in FP64 on one SM, where GB300's FP64 rate makes every
    // partial count: 128 blocks cover levels up to 2^18 rows; larger ones stream enough
    // test-vector bytes to need up to 512
    const int cap = n <= (1 << 18) ? 128 : (n >= (1 << 20) ? 512 : n >> 11);
    if (nb > cap) nb = cap;
    *width = nvec * 2 * W;
    return nb;
}
template <typename T, int MODE>
static void colstats(const MatView<T>& B, const T* T_val, const T* X, int ld, int col0, int ncols, const ColWork& cw,
                     cudaStream_t s) {
    constexpr int W = V16<T>::W;
    const int nvec = (ncols + W - 1) / W;
    int ny = 1;
    while (ny * 2 * nvec <= 256) ny *= 2;
    int width = 0;
    const int nb = colstats_blocks<T>(B.n, ncols, &width);
    size_t smem = (size_t)ny * nvec * 2 * W * sizeof(double);
    BAMG_LAUNCH((k_colstats<T, MODE>), nb, dim3(nvec, ny), smem, s, B.n, B.rp, B.ci, B.v, T_val, X, ld, col0, nvec,
                cw.partial, cw.ticket);
}
// sums[q] for q < width from the partials, one warp per output (lanes stride the blocks, then a
// fixed butterfly), COLSUM_T / 32 outputs a block of the grid.  True in every thread of the block that
// finishes last, which sees all sums.  One block for all outputs took 16 us for 128 partials of 40
// outputs and 32 for 512 of 48: some 900 FP64 additions of a warp, 16 cycles each on one SM's pipe.
constexpr int COLSUM_T = 128;
static int colsum_blocks(int width) { return (width + COLSUM_T / 32 - 1) / (COLSUM_T / 32); }
__device__ bool colsum_partials(int nblocks, int width, const double* __restrict__ partial, double* sums,
                                unsigned* ticket) {
    __shared__ int s_last;
    const int lane = threadIdx.x & 31;
    const int q = blockIdx.x * (COLSUM_T / 32) + (threadIdx.x >> 5);
    if (q < width) {
        double s = 0.0;
#pragma unroll 4
        for (int b = lane; b < nblocks; b += 32) s += partial[(int64_t)b * width + q];
        s = warp_sum(s);
        if (lane == 0) {
            sums[q] = s;
            __threadfence();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    return true;
}

// ---------------------------------------------------------------- LS weights
// nrm[k] = ||x_k||_2 and nrm[32 + k] = 1 / nrm[k] (used by FP32 test vectors)
__global__ void __launch_bounds__(COLSUM_T) k_weights(int ncols, int W, int nblocks, const ColWork cw,
                                                        const uint8_t* __restrict__ active, double floor,
                                                        double* __restrict__ w, double* __restrict__ nrm) {
    pdl_begin();
    if (!colsum_partials(nblocks, 2 * ((ncols + W - 1) / W) * W, cw.partial, cw.sums, cw.ticket)) return;
    if (threadIdx.x >= 32) return;
    const int k = threadIdx.x;  // one warp, ncols <= 32
    double m = 0.0, nk = 1.0;
    if (k < ncols) {
        const int ch = k / W, e = k - ch * W;
        const double xx = __ldcg(cw.sums + ch * 2 * W + e), bb = __ldcg(cw.sums + ch * 2 * W + W + e);
        const bool act = active ? active[k] != 0 : true;
        if (act && xx > 0.0) {
            nk = sqrt(xx);
            m = 1.0 / fmax(bb / xx, floor);
        }
    }
    double mx = m;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (k < ncols) {
        w[k] = mx > 0.0 ? m / mx : 0.0;
        nrm[k] = nk;
        nrm[32 + k] = 1.0 / nk;
    }
}

template <typename T>
__global__ void k_scale_cols(int n, T* __restrict__ X, int ld, int col0, int ncols, const double* __restrict__ nrm) {
    pdl_begin();
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int row = (int)(t / ncols);
    if (row >= n) return;
    int k = (int)(t - (int64_t)row * ncols);
    const double d = nrm[k];
    if (d != 1.0) {
        T* p = X + (int64_t)row * ld + col0 + k;
        if constexpr (sizeof(T) == 4)  // the FP64 product rounds to the same FP32 value as the quotient
            *p = (T)((double)*p * nrm[32 + k]);  // (but for double rounding); an FP64 division per element is slow
        else
            *p = (T)((double)*p / d);
    }
}

template <typename T>
void tv_weights(const MatView<T>& B, int ncols, int ld, int col0, const uint8_t* d_active, double floor, T* X,
                double* d_w, cudaStream_t s) {
    constexpr int W = V16<T>::W;
    BAMG_REQUIRE(ncols >= 1 && ncols <= 32, BAMG_EINVAL, "tv_weights: 1 <= ncols <= 32");
    int width = 0;
    const int nb = colstats_blocks<T>(B.n, ncols, &width);
    TmpBuf<double> work(64 + ColWork::doubles(nb, width), s);
    double* nrm = work.get();
    const ColWork cw(nrm + 64, nb, width);
    colstats<T, 0>(B, nullptr, X, ld, col0, ncols, cw, s);
    BAMG_LAUNCH(k_weights, colsum_blocks(width), COLSUM_T, 0, s, ncols, W, nb, cw, d_active, floor, d_w, nrm);
    BAMG_LAUNCH(k_scale_cols<T>, blocks_for((int64_t)B.n * ncols, 256), 256, 0, s, B.n, X, ld, col0, ncols,
                (const double*)nrm);
}

// ---------------------------------------------------------------- Rayleigh update
__global__ void __launch_bounds__(COLSUM_T) k_rayleigh(int ncols, int W, int nblocks, const ColWork cw, double tol,
                                                         double* __restrict__ lam, uint8_t* __restrict__ sel) {
    pdl_begin();
    if (!colsum_partials(nblocks, 2 * ((ncols + W - 1) / W) * W, cw.partial, cw.sums, cw.ticket)) return;
    const int k = threadIdx.x;
    if (k >= ncols) return;
    const int ch = k / W, e = k - ch * W;
    const double num = __ldcg(cw.sums + ch * 2 * W + e), den = __ldcg(cw.sums + ch * 2 * W + W + e);
    const double old = lam[k];
    const double nw = (k == 0) ? 0.0 : num / den;
    const double change = fabs(nw - old) / fmax(fabs(old), 1e-300);
    sel[k] = (k == 0 || change > tol) ? 1 : 0;
    lam[k] = nw;
}

template <typename T>
void rayleigh_update(const MatView<T>& B, const T* T_val, const T* X, int ncols, int ld, int col0, double tol,
                     double* d_lam, uint8_t* d_sel, cudaStream_t s) {
    constexpr int W = V16<T>::W;
    int width = 0;
    const int nb = colstats_blocks<T>(B.n, ncols, &width);
    TmpBuf<double> work(ColWork::doubles(nb, width), s);
    const ColWork cw(work.get(), nb, width);
    colstats<T, 1>(B, T_val, X, ld, col0, ncols, cw, s);
    BAMG_LAUNCH(k_rayleigh, colsum_blocks(width), COLSUM_T, 0, s, ncols, W, nb, cw, tol, d_lam, d_sel);
}

// ---------------------------------------------------------------- injection / prolongation
template <typename T>
__global__ void k_inject(int nc, const int32_t* __restrict__ c2f, const T* __restrict__ X, T* __restrict__ Xc, int ld,
                         int col0, int nvec) {
    pdl_begin();
    constexpr int W = V16<T>::W;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int I = (int)(t / nvec);
    if (I >= nc) return;
    int ch = (int)(t - (int64_t)I * nvec);
    T v[W];
    V16<T>::load(X + (int64_t)c2f[I] * ld + col0 + ch * W, v);
    V16<T>::store(Xc + (int64_t)I * ld + col0 + ch * W, v);
}
template <typename T>
void inject_cols(int nc, const int32_t* c2f, const T* X, T* Xc, int ld, int col0, int ncols, cudaStream_t s) {
    constexpr int W = V16<T>::W;
    const int nvec = (ncols + W - 1) / W;
    if (nc && nvec) BAMG_LAUNCH(k_inject<T>, blocks_for((int64_t)nc * nvec, 256), 256, 0, s, nc, c2f, X, Xc, ld, col0, nvec);
}

template <typename T>
__global__ void k_prolong_cols(int n, int c, const int32_t* __restrict__ pcol, const T* __restrict__ pval,
                               const int32_t* __restrict__ pcnt, const T* __restrict__ Xc, T* __restrict__ X, int ld,
                               int col0, int nvec) {
    pdl_begin();
    constexpr int W = V16<T>::W;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int i = (int)(t / nvec);
    if (i >= n) return;
    int ch = (int)(t - (int64_t)i * nvec);
    T acc[W];
#pragma unroll
    for (int e = 0; e < W; ++e) acc[e] = T(0);
    const int cnt = pcnt[i];
    for (int q = 0; q < cnt; ++q) {
        const int J = pcol[(int64_t)i * c + q];
        const T pv = pval[(int64_t)i * c + q];
        T xv[W];
        V16<T>::load(Xc + (int64_t)J * ld + col0 + ch * W, xv);
#pragma unroll
        for (int e = 0; e < W; ++e) acc[e] += pv * xv[e];
    }
    V16<T>::store(X + (int64_t)i * ld + col0 + ch * W, acc);
}
template <typename T>
void prolong_cols(const EllView<T>& P, const T* Xc, T* X, int ld, int col0, int ncols, cudaStream_t s) {
    constexpr int W = V16<T>::W;
    const int nvec = (ncols + W - 1) / W;
    if (P.n && nvec)
        BAMG_LAUNCH(k_prolong_cols<T>, blocks_for((int64_t)P.n * nvec, 256), 256, 0, s, P.n, P.c, P.pcol, P.pval,
                    P.pcnt, Xc, X, ld, col0, nvec);
}

// ---------------------------------------------------------------- conversions
template <typename Tin, typename Tout>
__global__ void k_convert(int64_t n, const Tin* a, Tout* b) {
    pdl_begin();
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (Tout)a[i];
}
template <typename Tin, typename Tout>
void launch_convert(int64_t n, const Tin* a, Tout* b, cudaStream_t s) {
    if (n > 0) BAMG_LAUNCH((k_convert<Tin, Tout>), blocks_for(n, 256), 256, 0, s, n, a, b);
}
template <typename Tin, typename Tout>
__global__ void k_strided_to_vec(int n, const Tin* X, int ld, int col, Tout* y) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = (Tout)X[(int64_t)i * ld + col];
}
template <typename Tin, typename Tout>
void launch_strided_to_vec(int n, const Tin* X, int ld, int col, Tout* y, cudaStream_t s) {
    if (n) BAMG_LAUNCH((k_strided_to_vec<Tin, Tout>), blocks_for(n, 256), 256, 0, s, n, X, ld, col, y);
}
// nv vectors y[q * n + i] to the columns col0 + q
template <typename Tin, typename Tout>
__global__ void k_vecs_to_strided(int n, int nv, const Tin* y, Tout* X, int ld, int col0) {
    pdl_begin();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)n * nv) return;
    const int q = (int)(t / n), i = (int)(t - (int64_t)q * n);
    X[(int64_t)i * ld + col0 + q] = (Tout)y[t];
}
template <typename Tin, typename Tout>
void launch_vecs_to_strided(int n, int nv, const Tin* y, Tout* X, int ld, int col0, cudaStream_t s) {
    if (n && nv)
        BAMG_LAUNCH((k_vecs_to_strided<Tin, Tout>), blocks_for((int64_t)n * nv, 256), 256, 0, s, n, nv, y, X, ld, col0);
}

// ---------------------------------------------------------------- B = I - A
__global__ void k_count_B(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const double* __restrict__ v, int32_t* __restrict__ cnt, int* __restrict__ flags,
                          double* __restrict__ colsum) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int f = 0;
    bool has_diag = false;
    const int p0 = rp[i], p1 = rp[i + 1];
    if (p1 < p0) f |= 8;
    for (int p = p0; p < p1; ++p) {
        const int j = ci[p];
        if (j < 0 || j >= n || (p > p0 && j <= ci[p - 1])) {
            f |= 8;
            continue;
        }
        const double a = v[p];
        if (!(a >= 0.0)) f |= 1;
        if (j == i) {
            has_diag = true;
            if (a >= 1.0) f |= 4;
        }
        atomicAdd(colsum + j, a);
    }
    cnt[i] = (p1 - p0) + (has_diag ? 0 : 1);
    if (f) atomicOr(flags, f);
}

__global__ void k_fill_B(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                         const double* __restrict__ v, const int32_t* __restrict__ rpB, int32_t* __restrict__ ciB,
                         double* __restrict__ vB) {
    pdl_begin();
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int q = rpB[i];
    bool done = false;
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
        const int j = ci[p];
        if (!done && j > i) {
            ciB[q] = i;
            vB[q] = 1.0;
            ++q;
            done = true;
        }
        if (j == i) {
            ciB[q] = i;
            vB[q] = 1.0 - v[p];
            done = true;
        } else {
            ciB[q] = j;
            vB[q] = -v[p];
        }
        ++q;
    }
    if (!done) {
        ciB[q] = i;
        vB[q] = 1.0;
    }
}

__global__ void k_check_colsum(int n, const double* __restrict__ colsum, int* __restrict__ flags) {
    pdl_begin();
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < n && !(fabs(colsum[j] - 1.0) <= 1e-12)) atomicOr(flags, 2);
}

int build_system_matrix(int n, int nnzA, const int32_t* rpA, const int32_t* ciA, const double* vA,
                        DevBuf<int32_t>& rpB, DevBuf<int32_t>& ciB, DevBuf<double>& vB, cudaStream_t s) {
    TmpBuf<int32_t> cnt(n, s);
    TmpBuf<double> colsum(n, s);
    TmpBuf<int> flags(1, s);
    BAMG_CK(cudaMemsetAsync(colsum.get(), 0, sizeof(double) * n, s));
    BAMG_CK(cudaMemsetAsync(flags.get(), 0, sizeof(int), s));
    BAMG_LAUNCH(k_count_B, blocks_for(n, 256), 256, 0, s, n, rpA, ciA, vA, cnt.get(), flags.get(), colsum.get());
    BAMG_LAUNCH(k_check_colsum, blocks_for(n, 256), 256, 0, s, n, colsum.get(), flags.get());
    const int h_flags = read_int(flags.get(), s);
    if (h_flags) return h_flags;
    rpB.alloc(n + 1);
    const int nnzB = exclusive_scan_total(cnt.get(), rpB.get(), n, s);
    ciB.alloc(nnzB);
    vB.alloc(nnzB);
    BAMG_LAUNCH(k_fill_B, blocks_for(n, 256), 256, 0, s, n, rpA, ciA, vA, rpB.get(), ciB.get(), vB.get());
    (void)nnzA;
    return 0;
}

// ---------------------------------------------------------------- instantiations
#define INST(T)                                                                                                    \
    template void launch_tv_init<T>(int, int, int, int, uint64_t, double, double, T*, cudaStream_t);               \
    template void launch_diag<T>(const MatView<T>&, T*, cudaStream_t);                                             \
    template void launch_diag_vals<T>(int, const int32_t*, const int32_t*, const T*, T*, cudaStream_t);            \
    template void launch_reciprocal<T>(int, const T*, T*, cudaStream_t);                                           \
    template void launch_diagonals<T>(int, const int32_t*, const int32_t*, const T*, const T*, T*, T*, T*,         \
                                      cudaStream_t);                                                                \
    template void launch_identity_on_pattern<T>(int, const int32_t*, const int32_t*, T*, cudaStream_t);            \
    template void relax<T>(const MatView<T>&, const T*, T*, T*, T*, const double*, int, int, int, T, int, T*, T*,  \
                           cudaStream_t, bool, bool);                                                    \
    template void tv_weights<T>(const MatView<T>&, int, int, int, const uint8_t*, double, T*, double*, cudaStream_t); \
    template void rayleigh_update<T>(const MatView<T>&, const T*, const T*, int, int, int, double, double*,         \
                                     uint8_t*, cudaStream_t);                                                      \
    template void inject_cols<T>(int, const int32_t*, const T*, T*, int, int, int, cudaStream_t);                  \
    template void prolong_cols<T>(const EllView<T>&, const T*, T*, int, int, int, cudaStream_t);
INST(float)
INST(double)
#undef INST
template void launch_convert<double, float>(int64_t, const double*, float*, cudaStream_t);
template void launch_convert<float, double>(int64_t, const float*, double*, cudaStream_t);
template void launch_convert<double, double>(int64_t, const double*, double*, cudaStream_t);
template void launch_strided_to_vec<float, double>(int, const float*, int, int, double*, cudaStream_t);
template void launch_strided_to_vec<double, double>(int, const double*, int, int, double*, cudaStream_t);
template void launch_vecs_to_strided<double, float>(int, int, const double*, float*, int, int, cudaStream_t);
template void launch_vecs_to_strided<double, double>(int, int, const double*, double*, int, int, cudaStream_t);

}  // namespace bamg
