// Interpolation and coarse operators: full coarsening (Section 5.1), the coarse
// neighbourhoods of Eq. (3.5), the greedy least-squares fit of Algorithm 2 / Eq. (3.6),
// the averaging restriction Q of Section 4, and the Petrov-Galerkin products
// B_{l+1} = Q B P, T_{l+1} = Q T P (Section 1 step 3, Algorithm 3).
#include <cfloat>

#include <algorithm>
#include <atomic>
#include <chrono>

#include "kernels.cuh"

namespace bamg {

// ================================================================ scan
constexpr int SCAN_T = 256, SCAN_I = 8, SCAN_B = SCAN_T * SCAN_I;

__global__ void k_scan_local(const int32_t* __restrict__ in, int32_t* __restrict__ out, int n,
                             int32_t* __restrict__ bsum) {
    pdl_begin();
    __shared__ int32_t wsum[SCAN_T / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t base = (int64_t)blockIdx.x * SCAN_B + (int64_t)threadIdx.x * SCAN_I;
    int32_t v[SCAN_I];
    int32_t tsum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_I; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0;
        tsum += v[k];
    }
    int32_t x = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int32_t w = lane < SCAN_T / 32 ? wsum[lane] : 0;
        int32_t incl = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane < SCAN_T / 32) wsum[lane] = incl - w;
        if (lane == SCAN_T / 32 - 1) bsum[blockIdx.x] = incl;
    }
    __syncthreads();
    int32_t run = x - tsum + wsum[warp];
#pragma unroll
    for (int k = 0; k < SCAN_I; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
}

__global__ void k_scan_sums(int32_t* __restrict__ bsum, int nb, int32_t* __restrict__ total,
                            int32_t* __restrict__ h_total) {
    pdl_begin();
    __shared__ int32_t wsum[32];
    __shared__ int32_t carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int c0 = 0; c0 < nb; c0 += blockDim.x) {
        const int i = c0 + threadIdx.x;
        const int32_t v = i < nb ? bsum[i] : 0;
        int32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            int32_t w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
            int32_t incl = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            wsum[lane] = incl - w;
        }
        __syncthreads();
        const int32_t excl = carry + wsum[warp] + x - v;
        __syncthreads();
        if (i < nb) bsum[i] = excl;
        if (threadIdx.x == blockDim.x - 1) carry = excl + v;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        *total = carry;
        if (h_total) {
            *(volatile int32_t*)h_total = carry;
            __threadfence_system();
        }
    }
}

__global__ void k_scan_add(int32_t* __restrict__ out, int n, const int32_t* __restrict__ bsum) {
    pdl_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += bsum[i / SCAN_B];
}

// Arrays of up to SCAN_ONE_MAX entries: one block walks the tiles in order with a running
// carry (one launch instead of three).  out[n] = total; out may alias in.
constexpr int SCAN_ONE_T = 1024, SCAN_ONE_MAX = 32768;
__global__ void __launch_bounds__(SCAN_ONE_T) k_scan_one(const int32_t* in, int32_t* out, int n,
                                                         int32_t* __restrict__ h_total) {
    pdl_begin();
    __shared__ int32_t wsum[SCAN_ONE_T / 32];
    __shared__ int32_t carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) carry = 0;
    for (int64_t t0 = 0; t0 < n; t0 += (int64_t)SCAN_ONE_T * SCAN_I) {
        const int64_t base = t0 + (int64_t)threadIdx.x * SCAN_I;
        int32_t v[SCAN_I];
        int32_t tsum = 0;
#pragma unroll
        for (int k = 0; k < SCAN_I; ++k) {
            v[k] = (base + k < n) ? in[base + k] : 0;
            tsum += v[k];
        }
        int32_t x = tsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        if (warp == 0) {
            const int32_t w = wsum[lane];
            int32_t incl = w;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            wsum[lane] = incl - w;
        }
        __syncthreads();
        int32_t run = carry + wsum[warp] + x - tsum;
#pragma unroll
        for (int k = 0; k < SCAN_I; ++k) {
            if (base + k < n) out[base + k] = run;
            run += v[k];
        }
        __syncthreads();  // every thread has read carry and wsum
        if (threadIdx.x == SCAN_ONE_T - 1) carry = run;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[n] = carry;
        if (h_total) {
            *(volatile int32_t*)h_total = carry;
            __threadfence_system();
        }
    }
}

// ---------------------------------------------------------------- counts read by the host
// A word of mapped pinned host memory per host thread and device: a kernel stores a count
// there and the host polls it, instead of a device-to-host copy and a stream synchronisation
// (whose completion path left the GPU idle for about 20 us per read in the setup).
struct HostWord {
    int32_t* h = nullptr;
    int32_t* d = nullptr;
    ~HostWord() {  // at the thread's end
        if (h) pinned_release(h);
    }
};
static HostWord& host_word() {
    thread_local HostWord w[64];
    int dev = 0;
    BAMG_CK(cudaGetDevice(&dev));
    BAMG_REQUIRE(dev >= 0 && dev < 64, BAMG_EINVAL, "device ordinal out of range");
    HostWord& hw = w[dev];
    if (!hw.h) {
        hw.h = static_cast<int32_t*>(pinned_acquire());
        BAMG_CK(cudaHostGetDevicePointer((void**)&hw.d, hw.h, 0));
    }
    return hw;
}
constexpr int32_t HOST_WORD_EMPTY = INT32_MIN;
// The count a kernel queued on s stores in the word: polled, with the stream's state checked
// now and then so that an error or a stream that finished without storing is reported; a
// bounded wait (BAMG_ETIMEOUT after 60 s).
static int32_t host_word_wait(const HostWord& hw, cudaStream_t s) {
    const auto t0 = std::chrono::steady_clock::now();
    for (uint64_t k = 0;; ++k) {
        const int32_t v = *(volatile int32_t*)hw.h;
        if (v != HOST_WORD_EMPTY) return v;
        if ((k & 1023) == 1023) {
            const cudaError_t e = cudaStreamQuery(s);
            if (e != cudaSuccess && e != cudaErrorNotReady) BAMG_CK(e);
            if (e == cudaSuccess && *(volatile int32_t*)hw.h == HOST_WORD_EMPTY)
                throw Error(BAMG_ECUDA, "a count the host waits for was not stored");
            if (std::chrono::steady_clock::now() - t0 > std::chrono::seconds(60))
                throw Error(BAMG_ETIMEOUT, "waiting for a count from the device");
        }
    }
}
__global__ void k_word_copy(const int32_t* __restrict__ d_p, int32_t* __restrict__ h) {
    pdl_begin();
    *(volatile int32_t*)h = *d_p;
    __threadfence_system();
}

void exclusive_scan(const int32_t* d_in, int32_t* d_out, int n, cudaStream_t s, int32_t* h_total) {
    if (n <= 0) {
        BAMG_CK(cudaMemsetAsync(d_out, 0, sizeof(int32_t), s));
        if (h_total) BAMG_LAUNCH(k_word_copy, 1, 1, 0, s, (const int32_t*)d_out, h_total);
        return;
    }
    if (n <= SCAN_ONE_MAX) {
        BAMG_LAUNCH(k_scan_one, 1, SCAN_ONE_T, 0, s, d_in, d_out, n, h_total);
        return;
    }
    const int nb = (int)blocks_for(n, SCAN_B);
    TmpBuf<int32_t> bsum(nb, s);
    BAMG_LAUNCH(k_scan_local, nb, SCAN_T, 0, s, d_in, d_out, n, bsum.get());
    BAMG_LAUNCH(k_scan_sums, 1, 1024, 0, s, bsum.get(), nb, d_out + n, h_total);
    BAMG_LAUNCH(k_scan_add, blocks_for(n, 256), 256, 0, s, d_out, n, bsum.get());
}

// exclusive scan of n counts into d_out (n + 1 entries), returning the total to the host
int32_t exclusive_scan_total(const int32_t* d_in, int32_t* d_out, int n, cudaStream_t s) {
    HostWord& hw = host_word();
    *(volatile int32_t*)hw.h = HOST_WORD_EMPTY;
    exclusive_scan(d_in, d_out, n, s, hw.d);
    return host_word_wait(hw, s);
}
// the same scan with the total left on its way to the host word (scan_total_wait collects it)
static void exclusive_scan_total_begin(const int32_t* d_in, int32_t* d_out, int n, cudaStream_t s) {
    HostWord& hw = host_word();
    *(volatile int32_t*)hw.h = HOST_WORD_EMPTY;
    exclusive_scan(d_in, d_out, n, s, hw.d);
}
static int32_t scan_total_wait(cudaStream_t s) { return host_word_wait(host_word(), s); }

HostPost host_post_begin() {
    HostWord& hw = host_word();
    *(volatile int32_t*)hw.h = HOST_WORD_EMPTY;
    return HostPost{hw.d, reinterpret_cast<double*>(hw.d + 16)};
}
void host_post_wait(double* out, int k, cudaStream_t s) {
    const HostWord& hw = host_word();
    host_word_wait(hw, s);
    std::atomic_thread_fence(std::memory_order_acquire);
    for (int q = 0; q < k; ++q) out[q] = ((volatile double*)(hw.h + 16))[q];
}

int32_t read_int(const int32_t* d_p, cudaStream_t s) {
    HostWord& hw = host_word();
    *(volatile int32_t*)hw.h = HOST_WORD_EMPTY;
    BAMG_LAUNCH(k_word_copy, 1, 1, 0, s, d_p, hw.d);
    return host_word_wait(hw, s);
}

// ================================================================ coarsening
__global__ void k_coarsen_grid(int nx, int ny, uint8_t* __restrict__ cf, int32_t* __restrict__ cidx) {
    pdl_begin();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nx * ny) return;
    const int ix = (int)(i % nx), iy = (int)(i / nx);
    const bool c = (ix % 2 == 0) && (iy % 2 == 0);
    cf[i] = c ? 1 : 0;
    cidx[i] = c ? (ix / 2) + (iy / 2) * ((nx + 1) / 2) : -1;
}
void coarsen_grid(int nx, int ny, uint8_t* cf, int32_t* cidx, cudaStream_t s) {
    BAMG_LAUNCH(k_coarsen_grid, blocks_for((int64_t)nx * ny, 256), 256, 0, s, nx, ny, cf, cidx);
}

__global__ void k_coarse_to_fine(int n, const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx,
                                 int32_t* __restrict__ c2f) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n && cf[i]) c2f[cidx[i]] = i;
}
void coarse_to_fine(int n, const uint8_t* cf, const int32_t* cidx, int32_t* c2f, cudaStream_t s) {
    if (n) BAMG_LAUNCH(k_coarse_to_fine, blocks_for(n, 256), 256, 0, s, n, cf, cidx, c2f);
}

// ================================================================ least-squares interpolation
constexpr int LS_WARPS = 4;
constexpr int VIS_CAP = 256;    // nodes recorded by one neighbourhood search (first pass)
constexpr int VIS_CAP2 = 2048;  // second pass, for the points whose search overflowed
constexpr int LS2_BLOCKS = 608;
constexpr int MMAX = 16;
constexpr int CMAX = 4;
constexpr int KMAX = 32;

// Solves the SPD system A x = b of order m <= CM by Cholesky; false if not SPD.
template <typename T, int CM>
__device__ __forceinline__ bool chol_solve(T (&A)[CM][CM], const T (&b)[CM], int m, T (&x)[CM]) {
    T L[CM][CM];
    T y[CM];
#pragma unroll
    for (int j = 0; j < CM; ++j) {
        if (j < m) {
            T s = A[j][j];
#pragma unroll
            for (int k = 0; k < CM; ++k)
                if (k < j) s -= L[j][k] * L[j][k];
            if (!(s > T(0))) return false;
            const T d = sqrt(s);
            L[j][j] = d;
#pragma unroll
            for (int i = 0; i < CM; ++i) {
                if (i > j && i < m) {
                    T t = A[i][j];
#pragma unroll
                    for (int k = 0; k < CM; ++k)
                        if (k < j) t -= L[i][k] * L[j][k];
                    L[i][j] = t / d;
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < CM; ++j) {
        if (j < m) {
            T t = b[j];
#pragma unroll
            for (int k = 0; k < CM; ++k)
                if (k < j) t -= L[j][k] * y[k];
            y[j] = t / L[j][j];
        }
    }
#pragma unroll
    for (int j = CM - 1; j >= 0; --j) {
        if (j < m) {
            T t = y[j];
#pragma unroll
            for (int k = 0; k < CM; ++k)
                if (k > j && k < m) t -= L[k][j] * x[k];
            x[j] = t / L[j][j];
        }
    }
    return true;
}

template <typename T>
__device__ __forceinline__ T warp_sum_t(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// b_rc, or 0 when column c is not in row r
template <typename T>
__device__ __forceinline__ T entry_of(int r, int c, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                      const T* __restrict__ bv) {
    for (int p = rp[r]; p < rp[r + 1]; ++p)
        if (ci[p] == c) return bv[p];
    return T(0);
}

// Features of fine point i for the learned interpolation (one warp; lane s < ncand holds
// candidate `node` with path length `depth`, g_jj = gss and g_ij = bs): per slot
// [1, d / 3, g_ij / g_jj, g_ij / sqrt(g_ii g_jj), -b_ij / b_ii, -b_ji / b_jj] (ratios with a
// zero denominator are 0), zeros for empty slots, then [m / 16, sum_{j != i} |b_ij| / b_ii],
// zero-padded to MLP_F.
template <typename T>
__device__ void learned_features(int i, int lane, int node, int ncand, int depth, T gss, T bs, const T* xi,
                                 const T* s_w, int ncols, const int32_t* __restrict__ rp,
                                 const int32_t* __restrict__ ci, const T* __restrict__ bv, float* f) {
    T gii = T(0);
    for (int k = 0; k < ncols; ++k) gii += s_w[k] * xi[k] * xi[k];
    T bii_l = T(0), off_l = T(0);
    for (int p = rp[i] + lane; p < rp[i + 1]; p += 32) {
        const T v = bv[p];
        if (ci[p] == i)
            bii_l += v;
        else
            off_l += v < T(0) ? -v : v;
    }
    const T bii = warp_sum_t(bii_l), off = warp_sum_t(off_l);
    if (lane < MLP_S) {
        float o[MLP_NF_SLOT] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (lane < ncand && node >= 0) {
            const T bij = entry_of<T>(i, node, rp, ci, bv);
            const T bji = entry_of<T>(node, i, rp, ci, bv);
            const T bjj = entry_of<T>(node, node, rp, ci, bv);
            o[0] = 1.f;
            o[1] = (float)((double)depth / 3.0);
            o[2] = gss != T(0) ? (float)(bs / gss) : 0.f;
            o[3] = gii * gss != T(0) ? (float)(bs / sqrt(gii * gss)) : 0.f;
            o[4] = (float)(-bij / bii);
            o[5] = (float)(-bji / bjj);
        }
#pragma unroll
        for (int e = 0; e < MLP_NF_SLOT; ++e) f[MLP_NF_SLOT * lane + e] = o[e];
    }
    for (int k = MLP_NF_SLOT * MLP_S + lane; k < MLP_F; k += 32) {
        float v = 0.f;
        if (k == MLP_NF_SLOT * MLP_S) v = (float)((double)ncand / (double)MLP_S);
        if (k == MLP_NF_SLOT * MLP_S + 1) v = (float)(off / bii);
        f[k] = v;
    }
}

// One warp per point.  Fine points: breadth-first search to depth z over the row
// pattern of B (edges i -> j for b_ij != 0, i != j), continued up to depth 3 while no
// coarse point has been found, and stopped early once mmax coarse points are known at
// the depths already completed; candidates = coarse points found, ranked by (depth,
// coarse index) and cut to mmax; then the greedy steps of
// Algorithm 2 with one lane per candidate: each lane forms its (|J|+1)-square weighted
// normal equations (plus the Tikhonov term), solves them by Cholesky and evaluates the
// functional of Eq. (3.6) directly; the lane with the smallest value (lowest slot on
// ties) joins J.
// Visited set of a neighbourhood search: open addressing over 2 CAP slots (load <= 1/2),
// keys are node indices, -1 = empty.
// (the product's top bits: its low bits repeat for states whose indices differ by a multiple of
// nslots, as neighbours in adjacent rows of a grid 512 wide do)
__device__ __forceinline__ unsigned vis_hash(int v, int nslots) {
    return ((unsigned)v * 2654435761u) >> (__clz(nslots) + 1);
}
__device__ __forceinline__ bool vis_contains(const int* hs, int nslots, int v) {
    for (unsigned h = vis_hash(v, nslots);; h = (h + 1) & (nslots - 1)) {
        const int k = hs[h];
        if (k == v) return true;
        if (k == -1) return false;
    }
}
__device__ __forceinline__ void vis_insert(int* hs, int nslots, int v) {
    for (unsigned h = vis_hash(v, nslots);; h = (h + 1) & (nslots - 1)) {
        const int prev = atomicCAS(&hs[h], -1, v);
        if (prev == -1 || prev == v) return;
    }
}

template <typename T, int CAP, bool EXTRA>
__device__ bool ls_point(int i, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                         const T* __restrict__ bv, const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx, const T* __restrict__ X,
                         int ncols, int ld, const T* s_w, int z, int mmax, int c, double ridge,
                         int32_t* __restrict__ pcol, T* __restrict__ pval, int32_t* __restrict__ pcnt, int* vis,
                         unsigned long long* key, uint8_t* dist, int* cand, uint8_t* cdep, T* xi, T (*xj)[KMAX],
                         int* hs, bool defer, const LsOut& ex) {
    constexpr int HS = 2 * CAP;  // visited-set slots
    const int lane = threadIdx.x & 31;
    const int64_t prow = (int64_t)i * c;
    if (cf[i]) {
        if (lane < c) {
            pcol[prow + lane] = lane == 0 ? cidx[i] : -1;
            pval[prow + lane] = lane == 0 ? T(1) : T(0);
        }
        if (lane == 0) pcnt[i] = 1;
        if (EXTRA) {
            if (ex.feat)
                for (int k = lane; k < MLP_F; k += 32) ex.feat[(int64_t)i * MLP_F + k] = 0.f;
            if (ex.target && lane < MLP_S) ex.target[(int64_t)i * MLP_S + lane] = 0.f;
            if (ex.cand && lane < MLP_S) ex.cand[(int64_t)i * MLP_S + lane] = -1;
        }
        return false;
    }
    // ---- neighbourhood search (Eq. (3.5))
    __syncwarp();
    for (int e = lane; e < HS; e += 32) hs[e] = -1;
    __syncwarp();
    if (lane == 0) {
        vis[0] = i;
        dist[0] = 0;
        vis_insert(hs, HS, i);
    }
    __syncwarp();
    int nvis = 1, fs = 0, fe = 1, ncvis = 0;
    bool ovf = false;
    for (int d = 1; d <= 3; ++d) {
        // beyond z only while no coarse point has been reached (the extension of R30);
        // and no deeper once mmax coarse points are known: deeper ones would rank after them
        if ((d > z && ncvis > 0) || ncvis >= mmax) break;
        bool fonly = false;  // visited list full: record only coarse nodes for the rest of this depth
        // the frontier's rows, 32 frontier nodes at a time: the lanes load the row pointers
        // together, lay the rows end to end (warp prefix sum), and take 32 entries of the
        // concatenation per batch (the same entries in the same order as row by row)
        for (int f0 = fs; f0 < fe; f0 += 32) {
            const int fu = f0 + lane;
            const int u = fu < fe ? vis[fu] : -1;
            const int ra = u >= 0 ? rp[u] : 0;
            const int rlen = u >= 0 ? rp[u + 1] - ra : 0;
            int incl = rlen;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            __syncwarp();
            for (int e0 = 0; e0 < total; e0 += 32) {
                const int e = e0 + lane;
                int k = 0;  // the lane whose row holds entry e: the first with incl > e
#pragma unroll
                for (int st = 16; st >= 1; st >>= 1) {
                    const int ic = __shfl_sync(0xffffffffu, incl, k + st - 1);
                    if (ic <= e) k += st;
                }
                const int ka = __shfl_sync(0xffffffffu, ra, k);
                const int kx = __shfl_sync(0xffffffffu, incl - rlen, k);
                const int v = e < total ? ci[ka + e - kx] : -1;
                const bool vc = v >= 0 && cf[v] != 0;  // loaded with v: the count below reads it from dist
                const bool isnew = v >= 0 && !vis_contains(hs, HS, v);
                const int key = isnew ? v : -1 - lane;
                const unsigned grp = __match_any_sync(0xffffffffu, key);
                const unsigned lt = (1u << lane) - 1u;
                const bool leader = isnew && (grp & lt) == 0u;
                unsigned bal = __ballot_sync(0xffffffffu, leader);
                if (fonly || nvis + __popc(bal) > CAP) {  // list full: keep the coarse nodes only
                    fonly = true;
                    bal = __ballot_sync(0xffffffffu, leader && vc);
                }
                const bool rec = (bal >> lane) & 1u;
                const int pos = nvis + __popc(bal & lt);
                if (rec && pos < CAP) {
                    vis[pos] = v;
                    dist[pos] = (uint8_t)(d | (vc ? 0x80 : 0));  // depth, and the C flag in bit 7
                    vis_insert(hs, HS, v);
                }
                int added = __popc(bal);
                if (nvis + added > CAP) {
                    ovf = true;
                    added = CAP - nvis;
                }
                nvis += added;
                __syncwarp();
            }
        }
        for (int q0 = fe; q0 < nvis; q0 += 32) {  // coarse points recorded at this depth
            const int q = q0 + lane;
            ncvis += __popc(__ballot_sync(0xffffffffu, q < nvis && (dist[q] & 0x80) != 0));
        }
        // a truncated depth (fine nodes not recorded) is exact only if the search ends here
        if (fonly) {
            if (d < 3 && ncvis < mmax && !(d >= z && ncvis > 0)) ovf = true;
            break;
        }
        fs = fe;
        fe = nvis;
    }
    if (ovf && defer) return true;  // the second pass redoes this point with a larger list
    // ---- candidates: coarse points ranked by (depth, coarse index).  The coarse entries
    // are compacted to the front of key (and their nodes to the front of vis; the point
    // itself at vis[0] is no longer needed), then ranked among themselves.
    int ntot = 0;
    for (int q0 = 1; q0 < nvis; q0 += 32) {
        const int q = q0 + lane;
        int v = -1;
        bool isc = false;
        unsigned long long kq = 0;
        if (q < nvis) {
            v = vis[q];
            isc = (dist[q] & 0x80) != 0;
            if (isc) kq = ((unsigned long long)(dist[q] & 0x7f) << 32) | (unsigned)cidx[v];
        }
        const unsigned bal = __ballot_sync(0xffffffffu, isc);
        __syncwarp();  // every lane has read vis[q] before the compacted writes below
        if (isc) {
            const int pos = ntot + __popc(bal & ((1u << lane) - 1u));
            key[pos] = kq;
            vis[pos] = v;
        }
        ntot += __popc(bal);
        __syncwarp();
    }
    for (int q0 = 0; q0 < ntot; q0 += 32) {
        const int q = q0 + lane;
        if (q < ntot) {
            const unsigned long long kq = key[q];
            int rank = 0;
            for (int q2 = 0; q2 < ntot; ++q2) rank += key[q2] < kq;
            if (rank < mmax) {
                cand[rank] = vis[q];
                cdep[rank] = (uint8_t)(kq >> 32);
            }
        }
    }
    const int ncand = ntot < mmax ? ntot : mmax;
    for (int k = lane; k < KMAX; k += 32) xi[k] = k < ncols ? X[(int64_t)i * ld + k] : T(0);
    __syncwarp();
    // ---- greedy least squares (Algorithm 2)
    const int node = lane < ncand ? cand[lane] : -1;
    const T* xs = node >= 0 ? X + (int64_t)node * ld : nullptr;
    T gss = T(0), bs = T(0);
    if (node >= 0)
        for (int k = 0; k < ncols; ++k) {
            const T wk = s_w[k], v = xs[k];
            gss += wk * v * v;
            bs += wk * v * xi[k];
        }
    if (EXTRA && ex.cand && lane < MLP_S) ex.cand[(int64_t)i * MLP_S + lane] = node;
    if (EXTRA && ex.feat) learned_features<T>(i, lane, node, ncand, lane < ncand ? cdep[lane] : 0, gss, bs, xi, s_w, ncols, rp,
                                     ci, bv, ex.feat + (int64_t)i * MLP_F);
    if (EXTRA && !ex.greedy) return false;
    T gsj[CMAX], GJJ[CMAX][CMAX], bJ[CMAX], pbest[CMAX];
    int J[CMAX];
#pragma unroll
    for (int a = 0; a < CMAX; ++a) {
        gsj[a] = bJ[a] = pbest[a] = T(0);
        J[a] = -1;
#pragma unroll
        for (int b = 0; b < CMAX; ++b) GJJ[a][b] = T(0);
    }
    bool used = false;
    int nJ = 0;
    const T INF = (T)INFINITY;
#pragma unroll
    for (int t = 0; t < CMAX; ++t) {
        if (t >= c) break;
        T L = INF;
        T pl[CMAX];
#pragma unroll
        for (int a = 0; a < CMAX; ++a) pl[a] = T(0);
        if (node >= 0 && !used) {
            T A[CMAX][CMAX], rhs[CMAX];
            T tr = gss;
#pragma unroll
            for (int a = 0; a < CMAX; ++a) {
#pragma unroll
                for (int b = 0; b < CMAX; ++b) A[a][b] = (a < t && b < t) ? GJJ[a][b] : T(0);
                rhs[a] = a < t ? bJ[a] : T(0);
                if (a < t) tr += GJJ[a][a];
            }
#pragma unroll
            for (int a = 0; a < CMAX; ++a) {
                if (a < t) {
                    A[a][t] = gsj[a];
                    A[t][a] = gsj[a];
                }
            }
            A[t][t] = gss;
            rhs[t] = bs;
            const T delta = (T)ridge * tr / (T)(t + 1);
#pragma unroll
            for (int a = 0; a < CMAX; ++a)
                if (a <= t) A[a][a] += delta;
            if (chol_solve<T, CMAX>(A, rhs, t + 1, pl)) {
                T acc = T(0);
                for (int k = 0; k < ncols; ++k) {
                    T r = xi[k] - pl[t] * xs[k];
#pragma unroll
                    for (int a = 0; a < CMAX; ++a)
                        if (a < t) r -= pl[a] * xj[a][k];
                    acc += s_w[k] * r * r;
                }
                L = (acc == acc) ? acc : INF;
            }
        }
        T bestL = L;
        int bestLane = lane;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const T oL = __shfl_xor_sync(0xffffffffu, bestL, o);
            const int oLane = __shfl_xor_sync(0xffffffffu, bestLane, o);
            if (oL < bestL || (oL == bestL && oLane < bestLane)) {
                bestL = oL;
                bestLane = oLane;
            }
        }
        if (!(bestL < INF)) break;
        const T w_gss = __shfl_sync(0xffffffffu, gss, bestLane);
        const T w_bs = __shfl_sync(0xffffffffu, bs, bestLane);
        const int w_node = __shfl_sync(0xffffffffu, node, bestLane);
#pragma unroll
        for (int a = 0; a < CMAX; ++a) {
            const T g = __shfl_sync(0xffffffffu, gsj[a], bestLane);
            const T pv = __shfl_sync(0xffffffffu, pl[a], bestLane);
            if (a < t) {
                GJJ[t][a] = g;
                GJJ[a][t] = g;
            }
            pbest[a] = a <= t ? pv : T(0);
        }
        GJJ[t][t] = w_gss;
        bJ[t] = w_bs;
        J[t] = w_node;
        nJ = t + 1;
        if (lane == bestLane) used = true;
        for (int k = lane; k < KMAX; k += 32) xj[t][k] = k < ncols ? X[(int64_t)w_node * ld + k] : T(0);
        __syncwarp();
        if (node >= 0) {
            T g = T(0);
            for (int k = 0; k < ncols; ++k) g += s_w[k] * xs[k] * xj[t][k];
            gsj[t] = g;
        }
    }
    if (lane == 0) {
        int cols[CMAX];
        T vals[CMAX];
#pragma unroll
        for (int a = 0; a < CMAX; ++a) {
            cols[a] = a < nJ ? cidx[J[a]] : 0x7fffffff;
            vals[a] = pbest[a];
        }
        for (int a = 1; a < nJ; ++a)
            for (int b = a; b > 0 && cols[b - 1] > cols[b]; --b) {
                int tc = cols[b];
                cols[b] = cols[b - 1];
                cols[b - 1] = tc;
                T tv = vals[b];
                vals[b] = vals[b - 1];
                vals[b - 1] = tv;
            }
        for (int a = 0; a < c; ++a) {
            pcol[prow + a] = a < nJ ? cols[a] : -1;
            pval[prow + a] = a < nJ ? vals[a] : T(0);
        }
        pcnt[i] = nJ;
    }
    if (EXTRA && ex.target && lane < MLP_S) {  // the LS row on the slots (Algorithm 2's choice)
        float tv = 0.f;
#pragma unroll
        for (int a = 0; a < CMAX; ++a)
            if (a < nJ && node >= 0 && J[a] == node) tv = (float)pbest[a];
        ex.target[(int64_t)i * MLP_S + lane] = tv;
    }
    return ovf;
}

// First pass (list == nullptr): warp per point i; a point whose search overflows the
// CAP-entry list is appended to ovf_list (or flags err when ovf_list is null).  Second
// pass (list != nullptr): persistent warps over the *list_count points of list.
template <typename T, int CAP, int WARPS, bool EXTRA>
__global__ void __launch_bounds__(WARPS * 32, (WARPS > 1 && sizeof(T) == 4) ? 8 : 1)  // FP32: 8 blocks/SM
    k_ls_fit(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const T* __restrict__ bv,
             const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx, const T* __restrict__ X, int ncols,
             int ld, const double* __restrict__ w, int z, int mmax, int c, double ridge, int32_t* __restrict__ pcol,
             T* __restrict__ pval, int32_t* __restrict__ pcnt, const int* __restrict__ list,
             const int* __restrict__ list_count, int* __restrict__ ovf_list, int* __restrict__ ovf_count,
             int* __restrict__ err, LsOut ex) {
    pdl_begin();
    __shared__ int s_vis[WARPS][CAP];
    __shared__ unsigned long long s_key[WARPS][CAP];
    __shared__ uint8_t s_dist[WARPS][CAP];
    __shared__ int s_cand[WARPS][MMAX];
    __shared__ uint8_t s_cdep[WARPS][MMAX];
    __shared__ int s_hash[WARPS][2 * CAP];
    __shared__ T s_xi[WARPS][KMAX];
    __shared__ T s_xj[WARPS][CMAX][KMAX];
    __shared__ T s_w[KMAX];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < KMAX) s_w[threadIdx.x] = threadIdx.x < ncols ? (T)w[threadIdx.x] : T(0);
    __syncthreads();
    if (list == nullptr) {
        const int i = blockIdx.x * WARPS + wid;
        if (i >= n) return;
        const bool ovf = ls_point<T, CAP, EXTRA>(i, rp, ci, bv, cf, cidx, X, ncols, ld, s_w, z, mmax, c, ridge, pcol, pval,
                                          pcnt, s_vis[wid], s_key[wid], s_dist[wid], s_cand[wid], s_cdep[wid],
                                          s_xi[wid], s_xj[wid], s_hash[wid], ovf_list != nullptr, ex);
        if (ovf && lane == 0) {
            if (ovf_list)
                ovf_list[atomicAdd(ovf_count, 1)] = i;
            else
                atomicOr(err, 1);
        }
        return;
    }
    const int cnt = *list_count;
    for (int k = blockIdx.x * WARPS + wid; k < cnt; k += gridDim.x * WARPS) {
        const bool ovf = ls_point<T, CAP, EXTRA>(list[k], rp, ci, bv, cf, cidx, X, ncols, ld, s_w, z, mmax, c, ridge, pcol,
                                          pval, pcnt, s_vis[wid], s_key[wid], s_dist[wid], s_cand[wid], s_cdep[wid],
                                          s_xi[wid], s_xj[wid], s_hash[wid], false, ex);
        if (ovf && lane == 0) atomicOr(err, 1);
    }
}

// ---------------------------------------------------------------- several points a warp
// The fit without optional outputs, in two kernels: the neighbourhood searches (half a warp a point, on
// long rows a whole one), then the greedy fits (four points a warp with eight lanes each, or two with 16, a
// candidate a lane).  Same candidates and the same arithmetic per candidate as ls_point, so the same rows
// bit for bit.
//
// What bounds them: instruction issue and the chain of dependent loads (every operand sits in L1 or
// L2).  One warp a point with half its lanes idle in the fit took 2240 warp instructions a fine point
// (631 us for 2^18 points of a triangulation, 16 columns).  Here
//  - the search's batches need no order within a depth (candidates are ranked by depth and coarse
//    index, and a search cut short by the list's capacity goes to the second pass), so an entry is
//    new if it wins its slot of the visited table: one compare-and-swap instead of a lookup, a match
//    over the warp and an insertion, and 4, 8 or 16 lanes walk a row instead of a search for the row
//    of each entry;
//  - at the last depth only coarse entries are taken down (the old list, filled by fine ones, sent
//    points of long-row levels to the second pass);
//  - coarse entries are listed as they are found, so a rank is a count within its depth;
//  - a lane keeps its candidate's test-vector row in registers (NC columns, 16-byte loads where X
//    allows them) instead of reading it again in each of the fit's five passes;
//  - the search, which waits for loads, runs with few registers and many warps, apart from the fit.
// Measured on those 2^18 points: one kernel 576 us; apart, search 307 and fit 172; with the visited
// table hashed by the product's top bits search 154 (ncu); the call 725 -> 370 us.  FP64, 16 columns,
// 93,300 points: 1591 -> 923 us.
constexpr int LSP_WARPS = 4;
// One search by GL lanes: CAP nodes recorded (beyond, the second pass) for the frontiers, and as
// many coarse nodes with their coarse indices, depth by depth.
template <int GL>
struct LsSearch {
    static constexpr int CAP = 8 * GL;
    int vis[CAP], hash[2 * CAP];
    int cnode[CAP], ccol[CAP];
};

// whether v is new: it wins (or finds) its slot of the visited table
template <int HS>
__device__ __forceinline__ bool lsp_claim(int* hs, int v) {
    for (unsigned h = vis_hash(v, HS);; h = (h + 1) & (HS - 1)) {
        int k = *(volatile int*)&hs[h];
        if (k == -1) {
            k = atomicCAS(&hs[h], -1, v);
            if (k == -1) return true;
        }
        if (k == v) return false;
    }
}

// Neighbourhood search (Eq. (3.5), with the extension to depth 3) of point i (i < 0: none) by GL lanes
// (half a warp or a whole one): candidates (nodes, in rank order) into cand; their count, or -1 when
// the list overflowed.  1 << gs lanes walk a row, U entries each at a time.  Every lane of the warp
// calls it.
template <int GL, int U>
__device__ __forceinline__ int lsp_search(int i, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                          const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx, int z,
                                          int mmax, int gs, LsSearch<GL>& sh, int32_t* __restrict__ cand) {
    constexpr int CAP = LsSearch<GL>::CAP;
    const int lane = threadIdx.x & 31, sub = lane & (GL - 1), hb = lane & ~(GL - 1);
    const unsigned lt = ((1u << sub) - 1u) << hb, half = (GL == 32 ? 0xffffffffu : 0xffffu) << hb;
    {
        int4* h4 = reinterpret_cast<int4*>(sh.hash);
#pragma unroll
        for (int e = 0; e < 2 * CAP / 4 / GL; ++e) h4[GL * e + sub] = make_int4(-1, -1, -1, -1);
    }
    __syncwarp();
    if (sub == 0 && i >= 0) {
        sh.vis[0] = i;
        sh.hash[vis_hash(i, 2 * CAP)] = i;
    }
    __syncwarp();
    int nvis = 1, nclaim = 1, fs = 0, fe = 1;
    int nc = 0, c1 = 0, c2 = 0;  // nc coarse nodes, c1 at depth 1, c2 up to depth 2
    bool run = i >= 0, ovf = false;
    const int rows = GL >> gs, width = 1 << gs;
#pragma unroll 1
    for (int d = 1; d <= 3; ++d) {
        // beyond z only while no coarse point has been reached; no deeper once mmax are known
        run = run && !((d > z && nc > 0) || nc >= mmax);
        if (!__any_sync(0xffffffffu, run)) break;
        // the last depth, or the list is full: only coarse nodes count from here on
        bool fonly = d == 3 || (d >= z && nc > 0);
#pragma unroll 1
        for (int f0 = fs; __any_sync(0xffffffffu, run && f0 < fe); f0 += rows) {
            const int f = f0 + (sub >> gs);
            int p = 0, pe = 0;
            if (run && f < fe) {
                const int u = sh.vis[f];
                p = rp[u] + (sub & (width - 1));
                pe = rp[u + 1];
            }
#pragma unroll 1
            for (; __any_sync(0xffffffffu, p < pe); p += U * width) {
                int v[U];
                bool c[U];
#pragma unroll
                for (int u = 0; u < U; ++u) v[u] = p + u * width < pe ? ci[p + u * width] : -1;
#pragma unroll
                for (int u = 0; u < U; ++u) c[u] = v[u] >= 0 && cf[v[u]] != 0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const bool want = run && v[u] >= 0 && (!fonly || c[u]);
                    if (U > 1 && !__any_sync(0xffffffffu, want)) continue;
                    const bool isnew = want && lsp_claim<2 * CAP>(sh.hash, v[u]);
                    const bool vc = isnew && c[u];
                    const unsigned bal = __ballot_sync(0xffffffffu, isnew) & half;
                    const unsigned balc = __ballot_sync(0xffffffffu, vc) & half;
                    fonly = fonly || nvis + __popc(bal) > CAP;
                    nclaim += __popc(bal);
                    // the coarse list is full, or the table would be with the next batch
                    if (nc + __popc(balc) > CAP || nclaim > 2 * CAP - 1 - GL) {
                        ovf = true;
                        run = false;
                        pe = 0;
                    } else {
                        if (isnew && !fonly) sh.vis[nvis + __popc(bal & lt)] = v[u];
                        if (vc) {
                            const int q = nc + __popc(balc & lt);
                            sh.cnode[q] = v[u];
                            sh.ccol[q] = cidx[v[u]];
                        }
                        if (!fonly) nvis += __popc(bal);
                        nc += __popc(balc);
                    }
                    __syncwarp();
                }
            }
        }
        if (fonly && run) {  // a truncated depth is exact only if the search ends here
            if (d < 3 && nc < mmax && !(d >= z && nc > 0)) ovf = true;
            run = false;
        }
        if (d == 1) c1 = nc;
        if (d <= 2) c2 = nc;
        fs = fe;
        fe = nvis;
    }
    if (i < 0 || ovf) nc = 0;
    // rank by (depth, coarse index): the list holds depth 1, then 2, then 3
#pragma unroll 1
    for (int q = sub; __any_sync(0xffffffffu, q < nc); q += GL) {
        if (q < nc) {
            const int a = q < c1 ? 0 : q < c2 ? c1 : c2, b = q < c1 ? c1 : q < c2 ? c2 : nc;
            const int kq = sh.ccol[q];
            int rank = a;
            for (int e = a; e < b && rank < mmax; ++e) rank += sh.ccol[e] < kq;
            if (rank < mmax) cand[rank] = sh.cnode[q];
        }
    }
    return ovf ? -1 : (nc < mmax ? nc : mmax);
}

// cand: mmax nodes a point; ncand: their count, -1 for a coarse point or one left to the second pass.
template <int GL, int U>
__global__ void __launch_bounds__(LSP_WARPS * 32, 10)
    k_ls_search(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const uint8_t* __restrict__ cf,
                const int32_t* __restrict__ cidx, int z, int mmax, int gs, int32_t* __restrict__ cand,
                int32_t* __restrict__ ncand, int* __restrict__ ovf_list, int* __restrict__ ovf_count) {
    pdl_begin();
    constexpr int PW = 32 / GL;  // points a warp
    __shared__ alignas(16) LsSearch<GL> s_point[LSP_WARPS][PW];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane & (GL - 1), h = lane / GL;
    LsSearch<GL>& sh = s_point[wid][h];
    const int64_t work = ((int64_t)n + PW - 1) / PW, stride = (int64_t)gridDim.x * LSP_WARPS;
#pragma unroll 1
    for (int64_t q = (int64_t)blockIdx.x * LSP_WARPS + wid; q < work; q += stride) {
        const int64_t i = PW * q + h;
        const bool fine = i < n && cf[i] == 0;
        int m = -1;
        if (__any_sync(0xffffffffu, fine)) {
            m = lsp_search<GL, U>(fine ? (int)i : -1, rp, ci, cf, cidx, z, mmax, gs, sh, cand + i * mmax);
            if (m < 0 && sub == 0) ovf_list[atomicAdd(ovf_count, 1)] = (int)i;  // the second pass redoes it
        }
        if (sub == 0 && i < n) ncand[i] = fine ? m : -1;
        __syncwarp();  // the shared memory takes the next points
    }
}

template <typename T, int CM>
struct LsFit {
    alignas(16) T xi[KMAX];
    alignas(16) T xj[CM][KMAX];
    T pad[32 / sizeof(T)];  // the four points of a warp read the same column on distinct banks
};
// blocks an SM: as many as leave the registers a candidate's row needs
constexpr int lsp_blocks(int size, int nc) {
    return size == 4 ? (nc <= 8 ? 6 : nc <= 16 ? 5 : 4) : (nc <= 8 ? 4 : nc <= 16 ? 3 : 2);
}
// The greedy fit (Algorithm 2) of one point by GL lanes, a candidate each (ncand <= GL): i64 the
// point, fine whether it is one to fit (ncand its candidates).  Every lane of the warp calls it.
template <typename T, int NC, int CM, int GL>
__device__ __forceinline__ void lsp_fit(int64_t i64, bool fine, int ncand, const int32_t* __restrict__ cidx,
                                        const int32_t* __restrict__ cand, const T* __restrict__ X, int ncols, int ld,
                                        const T* s_w, int mmax, int c, double ridge, bool vec, LsFit<T, CM>& sh,
                                        int32_t* __restrict__ pcol, T* __restrict__ pval, int32_t* __restrict__ pcnt) {
    constexpr int W = V16<T>::W;
    const T INF = (T)INFINITY;
    const int lane = threadIdx.x & 31, sub = lane & (GL - 1);
    const int node = sub < ncand ? cand[i64 * mmax + sub] : -1;
    const int ccol = node >= 0 ? cidx[node] : 0;
    T xs[NC];
    if (node >= 0) {
        const T* x = X + (int64_t)node * ld;
        if (vec) {
#pragma unroll
            for (int k = 0; k < NC; k += W)
                if (k < ncols) {
                    V16<T>::load(x + k, xs + k);
#pragma unroll
                    for (int e = 1; e < W; ++e)
                        if (k + e >= ncols) xs[k + e] = T(0);
                } else {
#pragma unroll
                    for (int e = 0; e < W; ++e) xs[k + e] = T(0);
                }
        } else {
#pragma unroll
            for (int k = 0; k < NC; ++k) xs[k] = k < ncols ? x[k] : T(0);
        }
    } else {
#pragma unroll
        for (int k = 0; k < NC; ++k) xs[k] = T(0);
    }
    for (int k = sub; k < NC; k += GL) sh.xi[k] = fine && k < ncols ? X[i64 * ld + k] : T(0);
    __syncwarp();
    T gss = T(0), bs = T(0);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
        const T wk = s_w[k], v = xs[k];
        gss += wk * v * v;
        bs += wk * v * sh.xi[k];
    }
    // greedy least squares (Algorithm 2)
    T gsj[CM], GJJ[CM][CM], bJ[CM], pbest[CM];
    int J[CM];
#pragma unroll
    for (int a = 0; a < CM; ++a) {
        gsj[a] = bJ[a] = pbest[a] = T(0);
        J[a] = 0x7fffffff;
#pragma unroll
        for (int b = 0; b < CM; ++b) GJJ[a][b] = T(0);
    }
    bool used = false, go = fine;
    int nJ = 0;
#pragma unroll
    for (int t = 0; t < CM; ++t) {
        if (t >= c) break;
        T L = INF;
        T pl[CM];
#pragma unroll
        for (int a = 0; a < CM; ++a) pl[a] = T(0);
        if (go && node >= 0 && !used) {
            T A[CM][CM], rhs[CM];
            T tr = gss;
#pragma unroll
            for (int a = 0; a < CM; ++a) {
#pragma unroll
                for (int b = 0; b < CM; ++b) A[a][b] = (a < t && b < t) ? GJJ[a][b] : T(0);
                rhs[a] = a < t ? bJ[a] : T(0);
                if (a < t) tr += GJJ[a][a];
            }
#pragma unroll
            for (int a = 0; a < CM; ++a) {
                if (a < t) {
                    A[a][t] = gsj[a];
                    A[t][a] = gsj[a];
                }
            }
            A[t][t] = gss;
            rhs[t] = bs;
            const T delta = (T)ridge * tr / (T)(t + 1);
#pragma unroll
            for (int a = 0; a < CM; ++a)
                if (a <= t) A[a][a] += delta;
            if (chol_solve<T, CM>(A, rhs, t + 1, pl)) {
                T acc = T(0);
#pragma unroll
                for (int k = 0; k < NC; ++k) {
                    T r = sh.xi[k] - pl[t] * xs[k];
#pragma unroll
                    for (int a = 0; a < CM; ++a)
                        if (a < t) r -= pl[a] * sh.xj[a][k];
                    acc += s_w[k] * r * r;
                }
                L = (acc == acc) ? acc : INF;
            }
        }
        T bestL = L;
        int bestLane = lane;
#pragma unroll
        for (int o = GL / 2; o > 0; o >>= 1) {
            const T oL = __shfl_xor_sync(0xffffffffu, bestL, o);
            const int oLane = __shfl_xor_sync(0xffffffffu, bestLane, o);
            if (oL < bestL || (oL == bestL && oLane < bestLane)) {
                bestL = oL;
                bestLane = oLane;
            }
        }
        go = go && bestL < INF;
        if (!__any_sync(0xffffffffu, go)) break;
        const T w_gss = __shfl_sync(0xffffffffu, gss, bestLane);
        const T w_bs = __shfl_sync(0xffffffffu, bs, bestLane);
        const int w_c = __shfl_sync(0xffffffffu, ccol, bestLane);
        T w_g[CM], w_p[CM];
#pragma unroll
        for (int a = 0; a < CM; ++a) {
            w_g[a] = __shfl_sync(0xffffffffu, gsj[a], bestLane);
            w_p[a] = __shfl_sync(0xffffffffu, pl[a], bestLane);
        }
        if (go) {
#pragma unroll
            for (int a = 0; a < CM; ++a) {
                if (a < t) {
                    GJJ[t][a] = w_g[a];
                    GJJ[a][t] = w_g[a];
                }
                pbest[a] = a <= t ? w_p[a] : T(0);
            }
            GJJ[t][t] = w_gss;
            bJ[t] = w_bs;
            J[t] = w_c;
            nJ = t + 1;
            if (lane == bestLane) {  // the winner's row, from its registers
                used = true;
#pragma unroll
                for (int k = 0; k < NC; k += W) V16<T>::store(&sh.xj[t][k], xs + k);
            }
        }
        __syncwarp();
        if (t + 1 < CM && t + 1 < c) {
            T g = T(0);
#pragma unroll
            for (int k = 0; k < NC; ++k) g += s_w[k] * xs[k] * sh.xj[t][k];
            gsj[t] = g;
        }
    }
    if (fine && sub == 0) {
        T vals[CM];
#pragma unroll
        for (int a = 0; a < CM; ++a) vals[a] = pbest[a];
#pragma unroll
        for (int a = 1; a < CM; ++a)  // by coarse index; empty slots (index 0x7fffffff) last
#pragma unroll
            for (int b = a; b > 0; --b)
                if (J[b - 1] > J[b]) {
                    const int tc = J[b];
                    J[b] = J[b - 1];
                    J[b - 1] = tc;
                    const T tv = vals[b];
                    vals[b] = vals[b - 1];
                    vals[b - 1] = tv;
                }
#pragma unroll
        for (int a = 0; a < CM; ++a)
            if (a < c) {
                pcol[i64 * c + a] = a < nJ ? J[a] : -1;
                pval[i64 * c + a] = a < nJ ? vals[a] : T(0);
            }
        pcnt[i64] = nJ;
    }
    __syncwarp();  // the shared memory takes the next points
}

// Four points a warp at a time: eight lanes each where none has more than eight candidates (full
// coarsening of a grid gives two or four, an independent set of a triangulation five to eight), else two
// by two with 16 lanes.
template <typename T, int NC, int CM>
__global__ void __launch_bounds__(LSP_WARPS * 32, lsp_blocks(sizeof(T), NC))
    k_ls_pair(int n, const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx, const int32_t* __restrict__ cand,
              const int32_t* __restrict__ ncands, const T* __restrict__ X, int ncols, int ld,
              const double* __restrict__ w, int mmax, int c, double ridge, bool vec, int32_t* __restrict__ pcol,
              T* __restrict__ pval, int32_t* __restrict__ pcnt) {
    pdl_begin();
    __shared__ LsFit<T, CM> s_fit[LSP_WARPS][4];
    __shared__ alignas(16) T s_w[KMAX];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x < KMAX) s_w[threadIdx.x] = threadIdx.x < ncols ? (T)w[threadIdx.x] : T(0);
    __syncthreads();
    const int64_t quads = ((int64_t)n + 3) / 4, stride = (int64_t)gridDim.x * LSP_WARPS;
#pragma unroll 1
    for (int64_t q = (int64_t)blockIdx.x * LSP_WARPS + wid; q < quads; q += stride) {
        const int64_t i = 4 * q + (lane >> 3);
        const int m = i < n ? ncands[i] : -1;
        if (i < n && m < 0 && cf[i]) {  // a coarse point's unit row
            const int sub = lane & 7;
            if (sub < c) {
                pcol[i * c + sub] = sub == 0 ? cidx[i] : -1;
                pval[i * c + sub] = sub == 0 ? T(1) : T(0);
            }
            if (sub == 0) pcnt[i] = 1;
        }
        const unsigned any = __ballot_sync(0xffffffffu, m >= 0);
        if (!any) continue;
        if (!__any_sync(0xffffffffu, m > 8)) {
            lsp_fit<T, NC, CM, 8>(i, m >= 0, m, cidx, cand, X, ncols, ld, s_w, mmax, c, ridge, vec, s_fit[wid][lane >> 3],
                                  pcol, pval, pcnt);
            continue;
        }
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            if (!((any >> (16 * h)) & 0xffffu)) continue;
            const int g = 2 * h + (lane >> 4);
            const int mg = __shfl_sync(0xffffffffu, m, 8 * g);
            lsp_fit<T, NC, CM, 16>(4 * q + g, mg >= 0, mg, cidx, cand, X, ncols, ld, s_w, mmax, c, ridge, vec,
                                   s_fit[wid][g], pcol, pval, pcnt);
        }
    }
}

template <typename T>
int interp_ls(int n, int nnz, const int32_t* rp, const int32_t* ci, const T* bv, const uint8_t* cf, const int32_t* cidx,
              const T* X, int ncols, int ld, const double* d_w, int z, int mmax, int c, double ridge, int32_t* pcol,
              T* pval, int32_t* pcnt, cudaStream_t s, int* d_err, const LsOut& ex) {
    BAMG_REQUIRE(ncols >= 1 && ncols <= KMAX, BAMG_EINVAL, "interp_ls: 1 <= ncols <= 32");
    BAMG_REQUIRE(c >= 1 && c <= CMAX, BAMG_EINVAL, "interp_ls: 1 <= caliber <= 4");
    BAMG_REQUIRE(mmax >= 1 && mmax <= MMAX, BAMG_EINVAL, "interp_ls: 1 <= mmax <= 16");
    BAMG_REQUIRE(z >= 1 && z <= 3, BAMG_EINVAL, "interp_ls: 1 <= z <= 3");
    if (n == 0) return 0;
    // two passes: the common case with a small visited list and 4 warps per block, then the
    // (rare) points whose search overflowed it, with a large list and one warp per block
    const bool extra = ex.feat || ex.target || ex.cand || !ex.greedy;
    // one allocation: the overflow count and flag, the listed points, and the searches' results
    TmpBuf<int32_t> work(2 + (size_t)n * (extra ? 1 : 2 + mmax), s);
    int *ocount = work.get(), *err = work.get() + 1, *olist = work.get() + 2;
    int32_t *ncand = work.get() + 2 + n, *cand = ncand + n;
    BAMG_CK(cudaMemsetAsync(ocount, 0, 2 * sizeof(int), s));
    int* e = d_err ? d_err : err;  // with d_err the caller reads the overflow flag later
    // the optional outputs are compiled into a separate instance (they cost registers)
    if (extra) {
        BAMG_LAUNCH((k_ls_fit<T, VIS_CAP, LS_WARPS, true>), blocks_for(n, LS_WARPS), LS_WARPS * 32, 0, s, n, rp, ci, bv,
                    cf, cidx, X, ncols, ld, d_w, z, mmax, c, ridge, pcol, pval, pcnt, (const int*)nullptr,
                    (const int*)nullptr, olist, ocount, e, ex);
        BAMG_LAUNCH((k_ls_fit<T, VIS_CAP2, 1, true>), LS2_BLOCKS, 32, 0, s, n, rp, ci, bv, cf, cidx, X, ncols, ld, d_w,
                    z, mmax, c, ridge, pcol, pval, pcnt, (const int*)olist, (const int*)ocount,
                    (int*)nullptr, (int*)nullptr, e, ex);
    } else {
        int dev = 0, nsm = 0;
        BAMG_CK(cudaGetDevice(&dev));
        BAMG_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        // enough blocks for two rounds of the resident ones; beyond, the warps walk the pairs
        auto search = [&](auto kern, int per_block, int gs) {
            const unsigned g = (unsigned)std::min<int64_t>(((int64_t)n + per_block - 1) / per_block, (int64_t)nsm * 20);
            BAMG_LAUNCH(kern, g, LSP_WARPS * 32, 0, s, n, rp, ci, cf, cidx, z, mmax, gs, cand, ncand,
                        olist, ocount);
        };
        // short rows: half a warp a point, the lanes that take an average row in one step; long rows (or
        // too few points to fill the chip with halves): a warp a point, four rows of up to 32 entries at
        // a time.  On a triangulation's coarse levels (rows of 19 to 36 entries, 6015 to 464 points) the
        // fit of a rebuild took 119 to 247 us with halves, 70 to 110 with warps, 64 to 86 before.
        if ((int64_t)nnz > 10 * (int64_t)n || n <= nsm * 32)
            search(k_ls_search<32, 4>, LSP_WARPS, 3);
        else
            search(k_ls_search<16, 1>, 2 * LSP_WARPS, (int64_t)nnz <= 4 * (int64_t)n ? 2 : 3);
        const unsigned grid =
            (unsigned)std::min<int64_t>(((int64_t)n + 4 * LSP_WARPS - 1) / (4 * LSP_WARPS), (int64_t)nsm * 12);
        constexpr int W = V16<T>::W;
        const bool vec = ld % W == 0 && ((uintptr_t)X & 15) == 0;
        auto go = [&](auto kern) {
            BAMG_LAUNCH(kern, grid, LSP_WARPS * 32, 0, s, n, cf, cidx, (const int32_t*)cand,
                        (const int32_t*)ncand, X, ncols, ld, d_w, mmax, c, ridge, vec, pcol, pval, pcnt);
        };
        // A fit of NC columns and CM slots: up to two slots (the default) by the columns there are, because a
        // lane's row in registers sets the blocks an SM (2^18 points, FP32: 263 us with 8 columns, 363 with
        // 32).  Three or four slots take one form: its systems, not its columns, take the time in FP32 (404 us
        // with 8 columns, 423 with 32; 462 and 489 with four), and in FP64 8 columns cost what 32 do
        // (3.3 and 4.8 ms), which is still less than a point a warp took (5.3 and 7.4 ms; FP32 0.85 and 0.97).
        if (c <= 2) {
            if (ncols <= 8) go(k_ls_pair<T, 8, 2>);
            else if (ncols <= 16) go(k_ls_pair<T, 16, 2>);
            else if (ncols <= 24) go(k_ls_pair<T, 24, 2>);
            else go(k_ls_pair<T, 32, 2>);
        } else {
            go(k_ls_pair<T, 32, 4>);
        }
        BAMG_LAUNCH((k_ls_fit<T, VIS_CAP2, 1, false>), LS2_BLOCKS, 32, 0, s, n, rp, ci, bv, cf, cidx, X, ncols, ld,
                    d_w, z, mmax, c, ridge, pcol, pval, pcnt, (const int*)olist, (const int*)ocount,
                    (int*)nullptr, (int*)nullptr, e, ex);
    }
    if (d_err) return 0;
    int h = 0;
    BAMG_CK(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    BAMG_CK(cudaStreamSynchronize(s));
    return h ? BAMG_EOVERFLOW : 0;
}

// ================================================================ learned interpolation
// One thread per fine point: the c valid slots of largest |y| (lower slot on ties) form J;
// weights y, or with refit the minimiser of Eq. (3.6) over J with the Tikhonov term
// delta = ridge tr(G_JJ) / |J| (R25); the row is stored sorted by coarse index.
template <typename T>
__global__ void k_learned_select(int n, const uint8_t* __restrict__ cf, const int32_t* __restrict__ cidx,
                                 const int32_t* __restrict__ cand, const float* __restrict__ Y, const T* __restrict__ X,
                                 int ncols, int ld, const double* __restrict__ w, int c, int refit, double ridge,
                                 int32_t* __restrict__ pcol, T* __restrict__ pval, int32_t* __restrict__ pcnt) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || cf[i]) return;
    const int32_t* cd = cand + (int64_t)i * MLP_S;
    const float* y = Y + (int64_t)i * MLP_S;
    int m = 0;
    while (m < MLP_S && cd[m] >= 0) ++m;
    int slot[CMAX];
    int nJ = 0;
    unsigned used = 0u;
    for (int t = 0; t < c && t < m; ++t) {
        int best = -1;
        float bv = -1.f;
        for (int q = 0; q < m; ++q) {
            const float a = fabsf(y[q]);
            if (!((used >> q) & 1u) && a > bv) {
                bv = a;
                best = q;
            }
        }
        if (best < 0) break;
        used |= 1u << best;
        slot[nJ++] = best;
    }
    T p[CMAX];
#pragma unroll
    for (int a = 0; a < CMAX; ++a) p[a] = (a < nJ) ? (T)y[slot[a < nJ ? a : 0]] : T(0);
    if (refit && nJ > 0) {
        T A[CMAX][CMAX], rhs[CMAX], sol[CMAX];
        T tr = T(0);
#pragma unroll
        for (int a = 0; a < CMAX; ++a) {
            rhs[a] = T(0);
#pragma unroll
            for (int b = 0; b < CMAX; ++b) A[a][b] = T(0);
        }
        const T* xi = X + (int64_t)i * ld;
        for (int a = 0; a < nJ; ++a) {
            const T* xa = X + (int64_t)cd[slot[a]] * ld;
            for (int b = 0; b <= a; ++b) {
                const T* xb = X + (int64_t)cd[slot[b]] * ld;
                T g = T(0);
                for (int k = 0; k < ncols; ++k) g += (T)w[k] * xa[k] * xb[k];
                A[a][b] = g;
                A[b][a] = g;
            }
            T r = T(0);
            for (int k = 0; k < ncols; ++k) r += (T)w[k] * xa[k] * xi[k];
            rhs[a] = r;
            tr += A[a][a];
        }
        const T delta = (T)ridge * tr / (T)nJ;
        for (int a = 0; a < nJ; ++a) A[a][a] += delta;
        if (chol_solve<T, CMAX>(A, rhs, nJ, sol))
#pragma unroll
            for (int a = 0; a < CMAX; ++a) p[a] = a < nJ ? sol[a] : T(0);
    }
    int cols[CMAX];
#pragma unroll
    for (int a = 0; a < CMAX; ++a) cols[a] = a < nJ ? cidx[cd[slot[a < nJ ? a : 0]]] : 0x7fffffff;
    for (int a = 1; a < nJ; ++a)
        for (int b = a; b > 0 && cols[b - 1] > cols[b]; --b) {
            const int tc = cols[b];
            cols[b] = cols[b - 1];
            cols[b - 1] = tc;
            const T tv = p[b];
            p[b] = p[b - 1];
            p[b - 1] = tv;
        }
    const int64_t prow = (int64_t)i * c;
    for (int a = 0; a < c; ++a) {
        pcol[prow + a] = a < nJ ? cols[a] : -1;
        pval[prow + a] = a < nJ ? p[a] : T(0);
    }
    pcnt[i] = nJ;
}

template <typename T>
int interp_learned(int n, int nnz, const int32_t* rp, const int32_t* ci, const T* bv, const uint8_t* cf, const int32_t* cidx,
                   const T* X, int ncols, int ld, const double* d_w, int z, int mmax, int c, double ridge,
                   const Model* model, bool refit, int32_t* pcol, T* pval, int32_t* pcnt, cudaStream_t s, int* d_err) {
    BAMG_REQUIRE(model != nullptr, BAMG_EINVAL, "learned interpolation without a model");
    BAMG_REQUIRE(mmax <= MLP_S, BAMG_EINVAL, "learned interpolation: mmax must be <= 16");
    if (n == 0) return 0;
    TmpBuf<float> feat((size_t)n * MLP_F, s), Y((size_t)n * MLP_S, s);
    TmpBuf<int32_t> cand((size_t)n * MLP_S, s);
    LsOut ex;
    ex.feat = feat.get();
    ex.cand = cand.get();
    ex.greedy = false;
    const int e = interp_ls<T>(n, nnz, rp, ci, bv, cf, cidx, X, ncols, ld, d_w, z, mmax, c, ridge, pcol, pval, pcnt, s,
                               d_err, ex);
    if (e) return e;
    mlp_forward(model, n, feat.get(), Y.get(), s);
    BAMG_LAUNCH(k_learned_select<T>, blocks_for(n, 128), 128, 0, s, n, cf, cidx, (const int32_t*)cand.get(),
                (const float*)Y.get(), X, ncols, ld, d_w, c, refit ? 1 : 0, ridge, pcol, pval, pcnt);
    return 0;
}

// ================================================================ restriction Q
__global__ void k_q_count(int n, int c, const int32_t* __restrict__ pcol, const int32_t* __restrict__ pcnt,
                          int32_t* __restrict__ qcnt) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int t = 0; t < pcnt[i]; ++t) atomicAdd(qcnt + pcol[(int64_t)i * c + t], 1);
}
__global__ void k_q_fill(int n, int c, const int32_t* __restrict__ pcol, const int32_t* __restrict__ pcnt,
                         const int32_t* __restrict__ qrp, int32_t* __restrict__ cursor, int32_t* __restrict__ qci) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int t = 0; t < pcnt[i]; ++t) {
        const int I = pcol[(int64_t)i * c + t];
        const int pos = atomicAdd(cursor + I, 1);
        qci[qrp[I] + pos] = i;
    }
}
// Sort each row by fine index (the fill order above is arbitrary) and set the
// averaging weights 1/|J_i| (Section 4: identical entries per column, 1^T Q = 1^T).
// Rows of up to Q_SORT_REG entries are sorted in registers (one load and one store per
// entry), longer ones in place; 1 / |J_i| comes from constants where |J_i| <= 4 (every
// caliber the setup allows), the same values as the division.
constexpr int Q_SORT_REG = 16;
template <typename T>
__global__ void k_q_sort(int nc, const int32_t* __restrict__ qrp, int32_t* __restrict__ qci, T* __restrict__ qv,
                         const int32_t* __restrict__ pcnt) {
    pdl_begin();
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= nc) return;
    auto inv = [](int p) {  // 1 / p, from constants for the common p <= 4
        switch (p) {
            case 1: return (T)(1.0 / 1.0);
            case 2: return (T)(1.0 / 2.0);
            case 3: return (T)(1.0 / 3.0);
            case 4: return (T)(1.0 / 4.0);
            default: return (T)(1.0 / (double)p);
        }
    };
    const int a = qrp[I], b = qrp[I + 1];
    if (b - a <= Q_SORT_REG) {
        int v[Q_SORT_REG];
#pragma unroll
        for (int k = 0; k < Q_SORT_REG; ++k) v[k] = a + k < b ? qci[a + k] : 0x7fffffff;
#pragma unroll
        for (int k = 1; k < Q_SORT_REG; ++k)  // insertion sort, unrolled: indices stay constant
#pragma unroll
            for (int q = k; q > 0; --q) {
                const int lo = min(v[q - 1], v[q]), hi = max(v[q - 1], v[q]);
                v[q - 1] = lo;
                v[q] = hi;
            }
#pragma unroll
        for (int k = 0; k < Q_SORT_REG; ++k)
            if (a + k < b) {
                qci[a + k] = v[k];
                qv[a + k] = inv(pcnt[v[k]]);
            }
        return;
    }
    for (int p = a + 1; p < b; ++p) {
        const int v = qci[p];
        int q = p;
        while (q > a && qci[q - 1] > v) {
            qci[q] = qci[q - 1];
            --q;
        }
        qci[q] = v;
    }
    for (int p = a; p < b; ++p) qv[p] = inv(pcnt[qci[p]]);
}

// Q's row pointers and (unsorted) entries; cnt and cursor: nc ints of scratch each, adjacent
static void restriction_pattern(int n, int c, const int32_t* pcol, const int32_t* pcnt, int nc, int32_t* cnt,
                                int32_t* qrp, int32_t* qci, cudaStream_t s) {
    BAMG_CK(cudaMemsetAsync(cnt, 0, 2 * sizeof(int32_t) * nc, s));
    BAMG_LAUNCH(k_q_count, blocks_for(n, 256), 256, 0, s, n, c, pcol, pcnt, cnt);
    exclusive_scan(cnt, qrp, nc, s);
    BAMG_LAUNCH(k_q_fill, blocks_for(n, 256), 256, 0, s, n, c, pcol, pcnt, (const int32_t*)qrp, cnt + nc, qci);
}

template <typename T>
void build_restriction(const EllView<T>& P, int nc, DevBuf<int32_t>& qrp, DevBuf<int32_t>& qci, DevBuf<T>& qv,
                       cudaStream_t s) {
    TmpBuf<int32_t> cnt(2 * (size_t)nc, s);
    qrp.alloc(nc + 1);
    const size_t nq = (size_t)P.n * P.c;  // bound: every row of P has at most c entries
    qci.alloc(nq > 0 ? nq : 1);
    qv.alloc(nq > 0 ? nq : 1);
    restriction_pattern(P.n, P.c, P.pcol, P.pcnt, nc, cnt.get(), qrp.get(), qci.get(), s);
    BAMG_LAUNCH(k_q_sort<T>, blocks_for(nc, 128), 128, 0, s, nc, qrp.get(), qci.get(), qv.get(), P.pcnt);
}

// ================================================================ Petrov-Galerkin
// Every product Q[I,i] M[i,j] P[j,J] is enumerated in the order (i, j, slot) for each
// coarse row I, rounded as ((q * m) * p); the products of one (I, J) are then summed in
// that order.  This is the order of the plain definition, so a CPU evaluation of the
// same sum in the same order gives the same bits.
// Products of coarse row I: sum over its Q entries i and the entries (i, j) of B of |P row j|.
// One warp per coarse row: the lanes take the Q entries, then the (i, j) pairs, 32 at a time.
constexpr int GAL_COUNT_WARPS = 4;
__global__ void __launch_bounds__(GAL_COUNT_WARPS * 32)
    k_gal_count(int nc, const int32_t* __restrict__ qrp, const int32_t* __restrict__ qci,
                const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const int32_t* __restrict__ pcnt,
                int32_t* __restrict__ np) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int I = blockIdx.x * GAL_COUNT_WARPS + (threadIdx.x >> 5);
    if (I >= nc) return;
    const int q0 = qrp[I], q1 = qrp[I + 1];
    int s = 0;
    for (int qc = q0; qc < q1; qc += 32) {
        const int qq = qc + lane;
        const int ii = qq < q1 ? qci[qq] : 0;
        const int rb = qq < q1 ? rp[ii] : 0;
        const int rl = qq < q1 ? rp[ii + 1] - rb : 0;
        int rinc = rl;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, rinc, d);
            if (lane >= d) rinc += v;
        }
        const int npairs = __shfl_sync(0xffffffffu, rinc, 31);
        for (int f0 = 0; f0 < npairs; f0 += 32) {
            const int f = f0 + lane;
            int k = 0;
#pragma unroll
            for (int st = 16; st >= 1; st >>= 1) {
                const int ic = __shfl_sync(0xffffffffu, rinc, k + st - 1);
                if (ic <= f) k += st;
            }
            k = min(k, 31);
            const int p = __shfl_sync(0xffffffffu, rb, k) + f - __shfl_sync(0xffffffffu, rinc - rl, k);
            if (f < npairs) s += pcnt[ci[p]];
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) np[I] = s;
}

template <typename T>
__global__ void k_gal_compact(int nc, const int32_t* __restrict__ poff, const int32_t* __restrict__ ucnt,
                              const int32_t* __restrict__ rpc, const int32_t* __restrict__ uJ, const T* __restrict__ ubv,
                              const T* __restrict__ utv, int32_t* __restrict__ ci, T* __restrict__ bv,
                              T* __restrict__ tv) {
    pdl_begin();
    const int lane = threadIdx.x & 31;
    const int I = blockIdx.x * GAL_COUNT_WARPS + (threadIdx.x >> 5);  // one warp per coarse row
    if (I >= nc) return;
    const int o = poff[I], d = rpc[I], cnt = ucnt[I];
    for (int u = lane; u < cnt; u += 32) {
        ci[d + u] = uJ[o + u];
        bv[d + u] = ubv[o + u];
        tv[d + u] = utv[o + u];
    }
}

// Expansion, ordering and summation of one coarse row in one warp, in shared memory: the
// lanes enumerate the row's (Q entry, B entry) pairs in order, each writing the products of
// its pair at their position in the definition order (a warp prefix sum over the pairs'
// product counts).  Every product then finds its J's slot (in order of first appearance, through
// a small open-addressing table) and its place among the slot's products, a counting sort lists
// the products slot by slot, and a lane adds up one slot's products in definition order: half of
// the warp B's, the other half T's.  The slots are finally ranked by J.
// What bounds it in FP64 is the pipe (a warp's operation every 16 cycles, however few lanes take part):
// summing the equal lanes of each chunk of 32 products, first B's and then T's, took 64 additions a
// row of 115 products with a few lanes in each; a row now takes as many as its longest sum (about 30).
// Rows are handled by a first kernel with room for GAL_CAP_S products per warp (most rows); longer
// rows go to a list that a second kernel accumulates in a hash table (below), and beyond its capacity
// by blocks of columns.
constexpr int GAL_WARPS_S = 4;
constexpr int GAL_CAP_S = 256;  // a power of two: also the slots of the row's J table
constexpr int GAL_CAP_LOG = 8;
static_assert((1 << GAL_CAP_LOG) == GAL_CAP_S, "J table size");
constexpr int GAL_BLOCKS_L = 608;

template <typename T>
struct GalArgs {
    int nc;
    const int32_t *qrp, *qci;
    const T* qv;
    const int32_t *rp, *ci;
    const T *bv, *tv;
    const int32_t* pcol;
    const T* pval;
    const int32_t* pcnt;
    int c;
    const int32_t* poff;
    int32_t *ucnt, *uJ;
    T *ubv, *utv;
};
template <typename T>
struct GalRow {  // one warp's row: products, then their slots
    T v[2][GAL_CAP_S];  // B's and T's products
    int J[GAL_CAP_S], hkey[GAL_CAP_S];
    unsigned short cnt[GAL_CAP_S], start[GAL_CAP_S];  // of a slot's products
    unsigned char hval[GAL_CAP_S], slot[GAL_CAP_S], pos[GAL_CAP_S], order[GAL_CAP_S];
};

// One coarse row I of at most GAL_CAP_S products in one warp.
template <typename T>
__device__ void gal_row(const GalArgs<T>& a, int I, GalRow<T>& w) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int o = a.poff[I], np = a.poff[I + 1] - o;
    const int q0 = a.qrp[I], q1 = a.qrp[I + 1];
    int base = 0;
    for (int qc = q0; qc < q1; qc += 32) {  // the Q row's entries in chunks of 32
        // each lane one entry (fine row i, its B row's start and length), prefix of the lengths
        const int qq = qc + lane;
        const int ii = qq < q1 ? a.qci[qq] : 0;
        const int rb = qq < q1 ? a.rp[ii] : 0;
        const int rl = qq < q1 ? a.rp[ii + 1] - rb : 0;
        int rinc = rl;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, rinc, d);
            if (lane >= d) rinc += v;
        }
        const int npairs = __shfl_sync(0xffffffffu, rinc, 31);
        for (int f0 = 0; f0 < npairs; f0 += 32) {
            const int f = f0 + lane;
            int k = 0;  // the chunk entry holding pair f: the first with rinc > f
#pragma unroll
            for (int st = 16; st >= 1; st >>= 1) {
                const int ic = __shfl_sync(0xffffffffu, rinc, k + st - 1);
                if (ic <= f) k += st;
            }
            k = min(k, 31);
            const int i = __shfl_sync(0xffffffffu, ii, k);
            const int p = __shfl_sync(0xffffffffu, rb, k) + f - __shfl_sync(0xffffffffu, rinc - rl, k);
            const int q = qc + k;
            const int j = f < npairs ? a.ci[p] : 0;
            const int cnt = f < npairs ? a.pcnt[j] : 0;
            int incl = cnt;  // inclusive warp prefix sum of the product counts
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += v;
            }
            const int pos0 = base + incl - cnt;
            if (f < npairs) {
                const T qq_ = a.qv[q];
                const T qb = mul_rn(qq_, a.bv[p]);
                const T qt = a.tv ? mul_rn(qq_, a.tv[p]) : (j == i ? qq_ : T(0));
                for (int sl = 0; sl < cnt; ++sl) {
                    const T pv = a.pval[(int64_t)j * a.c + sl];
                    const int e = pos0 + sl;
                    w.J[e] = a.pcol[(int64_t)j * a.c + sl];
                    w.v[0][e] = mul_rn(qb, pv);
                    w.v[1][e] = mul_rn(qt, pv);
                }
            }
            base += __shfl_sync(0xffffffffu, incl, 31);
        }
    }
    {
        int4* h4 = reinterpret_cast<int4*>(w.hkey);  // key J + 1; 0 = free
#pragma unroll
        for (int e = 0; e < GAL_CAP_S / 128; ++e) h4[32 * e + lane] = make_int4(0, 0, 0, 0);
    }
    __syncwarp();
    int U = 0;  // slots so far (U <= e0: each slot took at least one earlier product)
    for (int e0 = 0; e0 < np; e0 += 32) {
        const int e = e0 + lane;
        const int J = e < np ? w.J[e] : -1 - lane;
        const unsigned grp = __match_any_sync(0xffffffffu, J);
        const bool leader = e < np && (grp & lt) == 0u;
        bool claimed = false;
        unsigned h = 0;
        if (leader) {
            h = ((unsigned)J * 2654435761u) >> (32 - GAL_CAP_LOG);
            for (;;) {  // ends: the table has a free entry while U < GAL_CAP_S
                const int k = w.hkey[h];
                if (k == J + 1) break;
                if (k == 0 && atomicCAS(&w.hkey[h], 0, J + 1) == 0) {
                    claimed = true;
                    break;
                }
                h = (h + 1) & (GAL_CAP_S - 1);
            }
        }
        const unsigned cb = __ballot_sync(0xffffffffu, claimed);
        __syncwarp();  // this chunk's J are read before slots overwrite them
        int u = 0, before = 0;
        if (leader) {
            if (claimed) {
                u = U + __popc(cb & lt);  // < e0 + 32: a position already read
                w.hval[h] = (unsigned char)u;
                w.J[u] = J;
            } else {
                u = w.hval[h];
                before = w.cnt[u];
            }
            w.cnt[u] = (unsigned short)(before + __popc(grp));
        }
        const int src = __ffs(grp) - 1;
        u = __shfl_sync(0xffffffffu, u, src);
        before = __shfl_sync(0xffffffffu, before, src);
        if (e < np) {
            w.slot[e] = (unsigned char)u;
            w.pos[e] = (unsigned char)(before + __popc(grp & lt));
        }
        U += __popc(cb);
        __syncwarp();
    }
    int run = 0;
    for (int u0 = 0; u0 < U; u0 += 32) {  // starts of the slots' products
        const int u = u0 + lane, cnt = u < U ? w.cnt[u] : 0;
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        if (u < U) w.start[u] = (unsigned short)(run + incl - cnt);
        run += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    for (int e = lane; e < np; e += 32) w.order[w.start[w.slot[e]] + w.pos[e]] = (unsigned char)e;
    __syncwarp();
    const int h = lane >> 4;  // 0: B's products, 1: T's
    const T* val = w.v[h];
    for (int u = lane & 15; u < U; u += 16) {  // slot u goes to position rank(J) of the row
        const int Ju = w.J[u];
        const unsigned char* ord = w.order + w.start[u];
        const int cnt = w.cnt[u];
        T x = val[ord[0]];
        for (int k = 1; k < cnt; ++k) x = add_rn(x, val[ord[k]]);
        int rank = 0;
        for (int v = 0; v < U; ++v) rank += w.J[v] < Ju;
        (h ? a.utv : a.ubv)[o + rank] = x;
        if (h == 0) a.uJ[o + rank] = (int32_t)Ju;
    }
    if (lane == 0) a.ucnt[I] = U;
    __syncwarp();
}

// rows with at most GAL_CAP_S products; the others are appended to `list`
template <typename T>
__global__ void __launch_bounds__(GAL_WARPS_S * 32)
    k_gal_small(const __grid_constant__ GalArgs<T> a, int32_t* __restrict__ list, int* __restrict__ nlist) {
    pdl_begin();
    __shared__ alignas(16) GalRow<T> s_row[GAL_WARPS_S];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x * GAL_WARPS_S + wid;
    if (I >= a.nc) return;
    const int np = a.poff[I + 1] - a.poff[I];
    if (np > GAL_CAP_S) {
        if (lane == 0) list[atomicAdd(nlist, 1)] = I;
        return;
    }
    gal_row<T>(a, I, s_row[wid]);
}

// Long rows by accumulation instead of sorting: the products of each batch of 32 (Q, B)
// pairs are staged in definition order in shared memory; chunks of 32 staged products
// then find or claim their J in an open-addressing table (GAL_HSLOTS slots), the lanes
// that share a J in a chunk are summed by the lowest one in lane order, so every J
// accumulates its products in definition order.  The table's entries are finally sorted
// by J.  A row with more distinct J than half the table is summed by blocks of them (gal_row_blocks).
constexpr int GAL_HSLOTS = 2048;
constexpr int GAL_STAGE = 32 * 4;  // products of one batch of pairs (caliber <= 4)

// The table's occupied slots by J: skeys[e] = (J, slot) for e below the number of them, which is returned.
__device__ __forceinline__ int gal_sort_slots(const int* hkey, unsigned long long* skeys) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int u = 0;
    for (int e0 = 0; e0 < GAL_HSLOTS; e0 += 32) {
        const int e = e0 + lane;
        const bool occ = hkey[e] >= 0;
        const unsigned bal = __ballot_sync(0xffffffffu, occ);
        if (occ) skeys[u + __popc(bal & lt)] = ((unsigned long long)(unsigned)hkey[e] << 32) | (unsigned)e;
        u += __popc(bal);
    }
    __syncwarp();
    int N = 32;
    while (N < u) N <<= 1;
    for (int e = u + lane; e < N; e += 32) skeys[e] = ~0ull;
    __syncwarp();
    for (int k = 2; k <= N; k <<= 1) {
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int e = lane; e < N; e += 32) {
                const int pe = e ^ jj;
                if (pe > e) {
                    const unsigned long long x = skeys[e], y = skeys[pe];
                    const bool up = (e & k) == 0;
                    if ((x > y) == up) {
                        skeys[e] = y;
                        skeys[pe] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
    return u;
}
// The first u sorted slots to the row's entries from position `at` on; o: the row's product offset.
template <typename T>
__device__ __forceinline__ void gal_write_slots(const GalArgs<T>& a, int o, int at, int u, const T* hvb,
                                                const T* hvt, const unsigned long long* skeys) {
    for (int e = threadIdx.x & 31; e < u; e += 32) {
        const unsigned long long kk = skeys[e];
        const int slot = (int)(kk & 0xffffffffu);
        a.uJ[o + at + e] = (int32_t)(kk >> 32);
        a.ubv[o + at + e] = hvb[slot];
        a.utv[o + at + e] = hvt[slot];
    }
}
// J's slot, claimed if it is not there (linear probing; unrolled, it cost the rows of one
// table 8%); -1 when the table is full.
__device__ __forceinline__ int gal_slot(int* hkey, int J, bool& claimed) {
    unsigned h = ((unsigned)J * 2654435761u) & (GAL_HSLOTS - 1);
#pragma unroll 1
    for (int probe = 0; probe < GAL_HSLOTS; ++probe) {
        const int k = hkey[h];
        if (k == J) return (int)h;
        if (k == -1) {
            const int prev = atomicCAS(&hkey[h], -1, J);
            if (prev == -1 || prev == J) {
                claimed = prev == -1;
                return (int)h;
            }
        }
        h = (h + 1) & (GAL_HSLOTS - 1);
    }
    return -1;
}

template <typename T>
__device__ bool gal_row_hash(const GalArgs<T>& a, int I, int* hkey, T* hvb, T* hvt, int* sJ, T* sb_, T* st_,
                             unsigned long long* skeys) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int o = a.poff[I];
    for (int e = lane; e < GAL_HSLOTS; e += 32) {
        hkey[e] = -1;
        hvb[e] = T(0);
        hvt[e] = T(0);
    }
    __syncwarp();
    const int q0 = a.qrp[I], q1 = a.qrp[I + 1];
    int npairs = 0;
    for (int q = q0; q < q1; ++q) npairs += a.rp[a.qci[q] + 1] - a.rp[a.qci[q]];
    int used = 0;  // claimed slots
    for (int f0 = 0; f0 < npairs; f0 += 32) {
        const int f = f0 + lane;
        int q = q0, acc = 0, i = -1, p = -1;
        if (f < npairs) {
            for (; q < q1; ++q) {
                const int ii = a.qci[q], len = a.rp[ii + 1] - a.rp[ii];
                if (f < acc + len) {
                    i = ii;
                    p = a.rp[ii] + (f - acc);
                    break;
                }
                acc += len;
            }
        }
        const int j = f < npairs ? a.ci[p] : 0;
        const int cnt = f < npairs ? a.pcnt[j] : 0;
        int incl = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        const int pos0 = incl - cnt, nb = __shfl_sync(0xffffffffu, incl, 31);
        if (f < npairs) {  // stage this batch's products in definition order
            const T qq = a.qv[q];
            const T qb = mul_rn(qq, a.bv[p]);
            const T qt = a.tv ? mul_rn(qq, a.tv[p]) : (j == i ? qq : T(0));
            for (int sl = 0; sl < cnt; ++sl) {
                const T pv = a.pval[(int64_t)j * a.c + sl];
                sJ[pos0 + sl] = a.pcol[(int64_t)j * a.c + sl];
                sb_[pos0 + sl] = mul_rn(qb, pv);
                st_[pos0 + sl] = mul_rn(qt, pv);
            }
        }
        __syncwarp();
        for (int e0 = 0; e0 < nb; e0 += 32) {
            const int e = e0 + lane;
            const int J = e < nb ? sJ[e] : -1 - lane;
            const unsigned grp = __match_any_sync(0xffffffffu, J);
            const bool leader = e < nb && (grp & lt) == 0u;
            bool claimed = false;
            if (leader) {
                const int slot = gal_slot(hkey, J, claimed);
                if (slot >= 0) {
                    T vb = hvb[slot], vt = hvt[slot];
                    unsigned m = grp;
                    while (m) {  // the group's products in lane (= definition) order
                        const int l2 = __ffs(m) - 1;
                        m &= m - 1;
                        vb = add_rn(vb, sb_[e0 + l2]);
                        vt = add_rn(vt, st_[e0 + l2]);
                    }
                    hvb[slot] = vb;
                    hvt[slot] = vt;
                }
            }
            used += __popc(__ballot_sync(0xffffffffu, claimed));
            __syncwarp();
        }
        if (used > GAL_HSLOTS / 2) return false;  // too many distinct J: by blocks of them
    }
    const int u = gal_sort_slots(hkey, skeys);
    gal_write_slots(a, o, 0, u, hvb, hvt, skeys);
    if (lane == 0) a.ucnt[I] = u;
    __syncwarp();
    return true;
}

// A row of any length, in passes over its products: a pass sums those with J from lo on, as gal_row_hash
// does, and whenever three quarters of the table are taken keeps the lower half of its columns (hi: the
// first one it gave up, so every J in [lo, hi) has all its products in the table); the next pass begins at
// hi.  What bounds it is the chain of loads and shared-memory operations of the one warp, so the passes
// count: each takes 768 to 1664 columns, whatever the gaps between them.  Ranges of 2048 consecutive J, a range's
// products all added by one lane, took a pass for every range that the row touches: rows of 1,204 columns
// scattered over 100,000 took 9.0 ms in FP32 and 9.3 in FP64, now 0.38 and 0.39; over 1,500 (one range)
// 0.34 and 0.50, now 0.33 and 0.34; rows of 7,800 columns among 10,000 7.0 and 8.1, now 4.5 and 4.6.
template <typename T>
__device__ void gal_row_blocks(const GalArgs<T>& a, int I, int* hkey, T* hvb, T* hvt, int* sJ, T* sb_, T* st_,
                               unsigned long long* skeys) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int o = a.poff[I], q0 = a.qrp[I], q1 = a.qrp[I + 1];
    auto clear = [&] {  // -0: a slot's first product comes out as it is, its sign included
        for (int e = lane; e < GAL_HSLOTS; e += 32) {
            hkey[e] = -1;
            hvb[e] = T(-0.0);
            hvt[e] = T(-0.0);
        }
        __syncwarp();
    };
    int done = 0, lo = 0;  // entries written; J below lo are done
    for (;;) {
        int hi = 0x7fffffff, used = 0;
        clear();
        for (int qc = q0; qc < q1; qc += 32) {  // the Q row's entries in chunks of 32, their pairs in batches of 32
            const int qq = qc + lane;
            const int ii = qq < q1 ? a.qci[qq] : 0;
            const int rb = qq < q1 ? a.rp[ii] : 0;
            const int rl = qq < q1 ? a.rp[ii + 1] - rb : 0;
            int rinc = rl;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, rinc, d);
                if (lane >= d) rinc += v;
            }
            const int npairs = __shfl_sync(0xffffffffu, rinc, 31);
            for (int f0 = 0; f0 < npairs; f0 += 32) {
                const int f = f0 + lane;
                int k = 0;  // the chunk entry holding pair f: the first with rinc > f
#pragma unroll
                for (int st = 16; st >= 1; st >>= 1) {
                    const int ic = __shfl_sync(0xffffffffu, rinc, k + st - 1);
                    if (ic <= f) k += st;
                }
                k = min(k, 31);
                const int i = __shfl_sync(0xffffffffu, ii, k);
                const int p = __shfl_sync(0xffffffffu, rb, k) + f - __shfl_sync(0xffffffffu, rinc - rl, k);
                const int j = f < npairs ? a.ci[p] : 0;
                const int m = f < npairs ? a.pcnt[j] : 0;
                int cnt = 0;  // the pair's products of this pass
                for (int sl = 0; sl < m; ++sl) {
                    const int J = a.pcol[(int64_t)j * a.c + sl];
                    cnt += J >= lo && J < hi;
                }
                int incl = cnt;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const int v = __shfl_up_sync(0xffffffffu, incl, d);
                    if (lane >= d) incl += v;
                }
                const int nb = __shfl_sync(0xffffffffu, incl, 31);
                if (cnt > 0) {  // staged in definition order
                    const T qv = a.qv[qc + k];
                    const T qb = mul_rn(qv, a.bv[p]);
                    const T qt = a.tv ? mul_rn(qv, a.tv[p]) : (j == i ? qv : T(0));
                    int e = incl - cnt;
                    for (int sl = 0; sl < m; ++sl) {
                        const int J = a.pcol[(int64_t)j * a.c + sl];
                        if (J < lo || J >= hi) continue;
                        const T pv = a.pval[(int64_t)j * a.c + sl];
                        sJ[e] = J;
                        sb_[e] = mul_rn(qb, pv);
                        st_[e] = mul_rn(qt, pv);
                        ++e;
                    }
                }
                __syncwarp();
                for (int e0 = 0; e0 < nb; e0 += 32) {
                    const int e = e0 + lane;
                    const int J = e < nb ? sJ[e] : -1 - lane;
                    const unsigned grp = __match_any_sync(0xffffffffu, J);
                    bool claimed = false;
                    if (e < nb && (grp & lt) == 0u) {
                        const int slot = gal_slot(hkey, J, claimed);  // at most 1536 + 128 are taken
                        T vb = hvb[slot], vt = hvt[slot];
                        for (unsigned g = grp; g; g &= g - 1u) {  // the group's products in lane order
                            const int l2 = e0 + __ffs(g) - 1;
                            vb = add_rn(vb, sb_[l2]);
                            vt = add_rn(vt, st_[l2]);
                        }
                        hvb[slot] = vb;
                        hvt[slot] = vt;
                    }
                    used += __popc(__ballot_sync(0xffffffffu, claimed));
                    __syncwarp();
                }
                if (used > GAL_HSLOTS / 4 * 3) {  // keep the lower half: through the row's own place, and back
                    const int mid = gal_sort_slots(hkey, skeys) / 2;
                    hi = (int)(skeys[mid] >> 32);
                    gal_write_slots(a, o, done, mid, hvb, hvt, skeys);
                    __syncwarp();
                    clear();
                    for (int e = lane; e < mid; e += 32) {  // each lane what it has written itself
                        bool c = false;
                        const int slot = gal_slot(hkey, a.uJ[o + done + e], c);
                        hvb[slot] = a.ubv[o + done + e];
                        hvt[slot] = a.utv[o + done + e];
                    }
                    used = mid;
                    __syncwarp();
                }
            }
        }
        const int u = gal_sort_slots(hkey, skeys);
        gal_write_slots(a, o, done, u, hvb, hvt, skeys);
        done += u;
        __syncwarp();
        if (hi == 0x7fffffff) break;
        lo = hi;
    }
    if (lane == 0) a.ucnt[I] = done;
    __syncwarp();
}

// the listed rows, one warp per block, persistent over the list
template <typename T>
__global__ void __launch_bounds__(32) k_gal_large(const __grid_constant__ GalArgs<T> a,
                                                  const int32_t* __restrict__ list, const int* __restrict__ nlist) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char gal_smem[];
    unsigned long long* skeys = reinterpret_cast<unsigned long long*>(gal_smem);  // GAL_HSLOTS
    T* hvb = reinterpret_cast<T*>(skeys + GAL_HSLOTS);
    T* hvt = hvb + GAL_HSLOTS;
    T* sb_ = hvt + GAL_HSLOTS;
    T* st_ = sb_ + GAL_STAGE;
    int* hkey = reinterpret_cast<int*>(st_ + GAL_STAGE);
    int* sJ = hkey + GAL_HSLOTS;
    const int cnt = *nlist;
    for (int k = blockIdx.x; k < cnt; k += gridDim.x) {
        const int I = list[k];
        if (!gal_row_hash<T>(a, I, hkey, hvb, hvt, sJ, sb_, st_, skeys))
            gal_row_blocks<T>(a, I, hkey, hvb, hvt, sJ, sb_, st_, skeys);
    }
}

// The number of entries of B_c alone (the sizing call): every row's distinct J, counted by inserting
// them into a table of GAL_SYM_S slots a warp, or for the rows it lists of GAL_SYM_L slots a block.  A table
// gives up when a probe has passed a quarter of its slots (with J that spread, when it is nearly full): the
// row is listed, or sets *over, after which the products are formed and counted.
constexpr int GAL_SYM_S = 512, GAL_SYM_L = 8192;
constexpr int GAL_SYM_SUMS = 64;  // partial totals, a sector apart: one address would take every row in turn
template <int HS, int THREADS>
__device__ __forceinline__ int gal_distinct(int I, const int32_t* __restrict__ qrp, const int32_t* __restrict__ qci,
                                            const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                                            const int32_t* __restrict__ pcol, const int32_t* __restrict__ pcnt, int c,
                                            int t, int* table, volatile int* full) {
    int mine = 0;  // J this thread claimed
    const int q1 = qrp[I + 1];
    constexpr int G = 8, R = THREADS / G;  // eight lanes walk a row of B
    for (int q = qrp[I] + t / G; q < q1; q += R) {
        const int i = qci[q], pe = rp[i + 1];
        for (int p = rp[i] + (t & (G - 1)); p < pe; p += G) {
            const int j = ci[p], m = pcnt[j];
            for (int sl = 0; sl < m; ++sl) {
                const int J = pcol[(int64_t)j * c + sl];
                unsigned h = ((unsigned)J * 2654435761u) >> (__clz(HS) + 1);
                for (int probe = 0; probe < HS; ++probe, h = (h + 1) & (HS - 1)) {
                    int k = ((volatile int*)table)[h];
                    if (k == -1) {
                        k = atomicCAS(&table[h], -1, J);
                        if (k == -1) ++mine;
                    }
                    if (k == -1 || k == J) break;
                    if (probe == HS / 4) *full = 1;  // long probes: the table is filling up
                }
                if (*full) return mine;
            }
        }
    }
    return mine;
}
__global__ void __launch_bounds__(GAL_WARPS_S * 32)
    k_gal_sym(int nc, const int32_t* __restrict__ qrp, const int32_t* __restrict__ qci, const int32_t* __restrict__ rp,
              const int32_t* __restrict__ ci, const int32_t* __restrict__ pcol, const int32_t* __restrict__ pcnt, int c,
              int32_t* __restrict__ list, int* __restrict__ nlist, int* __restrict__ total) {
    pdl_begin();
    __shared__ alignas(16) int s_table[GAL_WARPS_S][GAL_SYM_S];
    __shared__ int s_full[GAL_WARPS_S];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int I = blockIdx.x * GAL_WARPS_S + wid;
    if (I >= nc) return;
    int4* t4 = reinterpret_cast<int4*>(s_table[wid]);
#pragma unroll
    for (int e = 0; e < GAL_SYM_S / 128; ++e) t4[32 * e + lane] = make_int4(-1, -1, -1, -1);
    if (lane == 0) s_full[wid] = 0;
    __syncwarp();
    int m = gal_distinct<GAL_SYM_S, 32>(I, qrp, qci, rp, ci, pcol, pcnt, c, lane, s_table[wid], &s_full[wid]);
    __syncwarp();
    m = __reduce_add_sync(0xffffffffu, m);
    if (lane == 0) {
        if (s_full[wid])
            list[atomicAdd(nlist, 1)] = I;
        else
            atomicAdd(total + 8 * (blockIdx.x % GAL_SYM_SUMS), m);
    }
}
__global__ void __launch_bounds__(256)
    k_gal_sym_large(const int32_t* __restrict__ qrp, const int32_t* __restrict__ qci, const int32_t* __restrict__ rp,
                    const int32_t* __restrict__ ci, const int32_t* __restrict__ pcol, const int32_t* __restrict__ pcnt,
                    int c, const int32_t* __restrict__ list, const int* __restrict__ nlist, int* __restrict__ total,
                    int* __restrict__ over) {
    pdl_begin();
    __shared__ int s_table[GAL_SYM_L];
    __shared__ int s_full, s_sum;
    const int cnt = *nlist;
    for (int k = blockIdx.x; k < cnt; k += gridDim.x) {
        __syncthreads();
        for (int e = threadIdx.x; e < GAL_SYM_L; e += blockDim.x) s_table[e] = -1;
        if (threadIdx.x == 0) s_full = s_sum = 0;
        __syncthreads();
        const int m = gal_distinct<GAL_SYM_L, 256>(list[k], qrp, qci, rp, ci, pcol, pcnt, c, threadIdx.x, s_table, &s_full);
        atomicAdd(&s_sum, m);
        __syncthreads();
        if (threadIdx.x == 0) {
            if (s_full)
                *over = 1;
            else
                atomicAdd(total, s_sum);
        }
    }
}

// 256-byte aligned slices of one temporary
struct Slices {
    size_t used = 0;
    size_t add(size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) & ~size_t(255);
        return at;
    }
};
// The products of B_c and T_c row by row (at the rows' product offsets poff, ucnt entries each).
template <typename T>
struct GalProducts {
    size_t tot;
    Slices sl;
    size_t o_np, o_poff, o_ucnt, o_list, o_nlist, o_uJ, o_ubv, o_utv;
    GalProducts(const MatView<T>& B, int nc, int c) {
        // bound on the product count: each entry b_ij meets at most c columns of Q and c rows of P
        const size_t bound = (size_t)B.nnz * c * c;
        BAMG_REQUIRE(bound < (size_t)INT32_MAX, BAMG_EINVAL, "galerkin: product count may overflow int32");
        tot = bound > 0 ? bound : 1;
        o_np = sl.add(sizeof(int32_t) * nc);
        o_poff = sl.add(sizeof(int32_t) * ((size_t)nc + 1));
        o_ucnt = sl.add(sizeof(int32_t) * nc);
        o_list = sl.add(sizeof(int32_t) * nc);
        o_nlist = sl.add(sizeof(int));
        o_uJ = sl.add(sizeof(int32_t) * tot);
        o_ubv = sl.add(sizeof(T) * tot);
        o_utv = sl.add(sizeof(T) * tot);
    }
    GalArgs<T> run(char* w, const MatView<T>& B, const T* T_val, const int32_t* qrp, const int32_t* qci, const T* qv,
                   const EllView<T>& P, int nc, cudaStream_t s) const {
        int32_t *np = (int32_t*)(w + o_np), *poff = (int32_t*)(w + o_poff), *list = (int32_t*)(w + o_list);
        int* nlist = (int*)(w + o_nlist);
        BAMG_LAUNCH(k_gal_count, blocks_for(nc, GAL_COUNT_WARPS), GAL_COUNT_WARPS * 32, 0, s, nc, qrp, qci, B.rp, B.ci,
                    P.pcnt, np);
        exclusive_scan(np, poff, nc, s);
        const GalArgs<T> ga{nc,     qrp, qci,  qv, B.rp, B.ci, B.v, T_val, P.pcol, P.pval, P.pcnt, P.c, poff,
                            (int32_t*)(w + o_ucnt), (int32_t*)(w + o_uJ), (T*)(w + o_ubv), (T*)(w + o_utv)};
        BAMG_CK(cudaMemsetAsync(nlist, 0, sizeof(int), s));
        BAMG_LAUNCH(k_gal_small<T>, blocks_for(nc, GAL_WARPS_S), GAL_WARPS_S * 32, 0, s, ga, list, nlist);
        auto large_smem = [](size_t tb) {
            return (size_t)GAL_HSLOTS * (sizeof(unsigned long long) + 2 * tb + sizeof(int)) +
                   GAL_STAGE * (2 * tb + sizeof(int));
        };
        static std::atomic<bool> attr[256] = {};  // per device; idempotent across host threads
        int dev = 0;
        BAMG_CK(cudaGetDevice(&dev));
        BAMG_REQUIRE(dev >= 0 && dev < 256, BAMG_EINVAL, "device ordinal out of range");
        if (!attr[dev]) {
            BAMG_CK(cudaFuncSetAttribute(k_gal_large<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)large_smem(sizeof(T))));
            attr[dev] = true;
        }
        BAMG_LAUNCH(k_gal_large<T>, GAL_BLOCKS_L, 32, large_smem(sizeof(T)), s, ga, (const int32_t*)list,
                    (const int*)nlist);
        return ga;
    }
};
template <typename T>
static void gal_compact(const GalArgs<T>& ga, const int32_t* rp, int32_t* ci, T* bv, T* tv, cudaStream_t s) {
    BAMG_LAUNCH(k_gal_compact<T>, blocks_for(ga.nc, GAL_COUNT_WARPS), GAL_COUNT_WARPS * 32, 0, s, ga.nc, ga.poff, ga.ucnt,
                rp, ga.uJ, ga.ubv, ga.utv, ci, bv, tv);
}

template <typename T>
void galerkin(const MatView<T>& B, const T* T_val, const int32_t* qrp, const int32_t* qci, const T* qv,
              const EllView<T>& P, int nc, GalerkinOut<T>& out, cudaStream_t s, bool defer) {
    const GalProducts<T> gp(B, nc, P.c);
    TmpBuf<char> work(gp.sl.used, s);
    const GalArgs<T> ga = gp.run(work.get(), B, T_val, qrp, qci, qv, P, nc, s);
    out.rp.alloc(nc + 1);
    size_t nz = gp.tot;  // with defer: room for the bound, the count still on its way
    // (only while the bound's arrays stay small: large ones cost more to allocate than the wait)
    if (defer && gp.tot * (sizeof(int32_t) + 2 * sizeof(T)) > ((size_t)64 << 20)) defer = false;
    if (defer) {
        exclusive_scan_total_begin(ga.ucnt, out.rp.get(), nc, s);
        out.nnz = -1;
    } else {
        out.nnz = exclusive_scan_total(ga.ucnt, out.rp.get(), nc, s);
        nz = out.nnz > 0 ? (size_t)out.nnz : 1;
    }
    out.ci.alloc(nz);
    out.bv.alloc(nz);
    out.tv.alloc(nz);
    gal_compact<T>(ga, out.rp.get(), out.ci.get(), out.bv.get(), out.tv.get(), s);
}

// The products into the caller's arrays (capacity cap; out_tv may be null).  Returns the number of
// entries; nothing is written when it exceeds cap.  With cap 0 (the sizing call) only the number is
// formed, from the patterns: it took as long as the products.
template <typename T>
int64_t galerkin_into(const MatView<T>& B, const T* T_val, const EllView<T>& P, int nc, int32_t* out_rp,
                      int32_t* out_ci, T* out_bv, T* out_tv, int64_t cap, cudaStream_t s) {
    const size_t nq = (size_t)P.n * P.c > 0 ? (size_t)P.n * P.c : 1;
    if (cap == 0) {
        Slices sl;
        const size_t o_cnt = sl.add(2 * sizeof(int32_t) * (size_t)nc), o_qrp = sl.add(sizeof(int32_t) * ((size_t)nc + 1)),
                     o_qci = sl.add(sizeof(int32_t) * nq), o_list = sl.add(sizeof(int32_t) * (size_t)nc),
                     o_num = sl.add((8 + 8 * GAL_SYM_SUMS) * sizeof(int));
        GalProducts<T> bound(B, nc, P.c);  // refuses what the products would refuse
        TmpBuf<char> work(sl.used, s);
        int32_t *qrp = (int32_t*)(work.get() + o_qrp), *qci = (int32_t*)(work.get() + o_qci);
        int32_t* list = (int32_t*)(work.get() + o_list);
        int* num = (int*)(work.get() + o_num);  // listed rows, overflow, then the partial totals
        restriction_pattern(P.n, P.c, P.pcol, P.pcnt, nc, (int32_t*)(work.get() + o_cnt), qrp, qci, s);
        int h[8 + 8 * GAL_SYM_SUMS];
        BAMG_CK(cudaMemsetAsync(num, 0, sizeof h, s));
        BAMG_LAUNCH(k_gal_sym, blocks_for(nc, GAL_WARPS_S), GAL_WARPS_S * 32, 0, s, nc, (const int32_t*)qrp,
                    (const int32_t*)qci, B.rp, B.ci, P.pcol, P.pcnt, P.c, list, num, num + 8);
        BAMG_LAUNCH(k_gal_sym_large, GAL_BLOCKS_L, 256, 0, s, (const int32_t*)qrp, (const int32_t*)qci, B.rp, B.ci, P.pcol,
                    P.pcnt, P.c, (const int32_t*)list, (const int*)num, num + 8, num + 1);
        BAMG_CK(cudaMemcpyAsync(h, num, sizeof h, cudaMemcpyDeviceToHost, s));
        BAMG_CK(cudaStreamSynchronize(s));
        int64_t nnz = 0;
        for (int k = 0; k < GAL_SYM_SUMS; ++k) nnz += h[8 + 8 * k];
        if (!h[1] && nnz > 0) return nnz;
    }
    GalProducts<T> gp(B, nc, P.c);
    const size_t o_cnt = gp.sl.add(2 * sizeof(int32_t) * (size_t)nc), o_qrp = gp.sl.add(sizeof(int32_t) * ((size_t)nc + 1)),
                 o_qci = gp.sl.add(sizeof(int32_t) * nq), o_qv = gp.sl.add(sizeof(T) * nq),
                 o_rp = gp.sl.add(sizeof(int32_t) * ((size_t)nc + 1)), o_tv = gp.sl.add(out_tv ? 0 : sizeof(T) * gp.tot);
    TmpBuf<char> work(gp.sl.used, s);
    char* w = work.get();
    int32_t *qrp = (int32_t*)(w + o_qrp), *qci = (int32_t*)(w + o_qci), *rp = (int32_t*)(w + o_rp);
    T* qv = (T*)(w + o_qv);
    restriction_pattern(P.n, P.c, P.pcol, P.pcnt, nc, (int32_t*)(w + o_cnt), qrp, qci, s);
    BAMG_LAUNCH(k_q_sort<T>, blocks_for(nc, 128), 128, 0, s, nc, (const int32_t*)qrp, qci, qv, P.pcnt);
    const GalArgs<T> ga = gp.run(w, B, T_val, qrp, qci, qv, P, nc, s);
    const int64_t nnz = exclusive_scan_total(ga.ucnt, rp, nc, s);
    if (cap < nnz) return nnz;
    BAMG_REQUIRE(out_rp && out_ci && out_bv, BAMG_EINVAL, "null output");
    BAMG_CK(cudaMemcpyAsync(out_rp, rp, sizeof(int32_t) * ((size_t)nc + 1), cudaMemcpyDeviceToDevice, s));
    gal_compact<T>(ga, rp, out_ci, out_bv, out_tv ? out_tv : (T*)(w + o_tv), s);
    BAMG_CK(cudaStreamSynchronize(s));
    return nnz;
}

template <typename T>
void galerkin_nnz(GalerkinOut<T>& out, cudaStream_t s) {
    if (out.nnz < 0) out.nnz = scan_total_wait(s);
}

template <typename T>
__global__ void k_csr_to_dense(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                               const T* __restrict__ v, double* __restrict__ D) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int p = rp[i]; p < rp[i + 1]; ++p) D[(int64_t)i * n + ci[p]] = (double)v[p];
}
template <typename T>
void csr_to_dense(int n, const int32_t* rp, const int32_t* ci, const T* v, double* D, cudaStream_t s) {
    BAMG_CK(cudaMemsetAsync(D, 0, sizeof(double) * n * n, s));
    if (n) BAMG_LAUNCH(k_csr_to_dense<T>, blocks_for(n, 64), 64, 0, s, n, rp, ci, v, D);
}

#define INST(T)                                                                                                     \
    template int interp_ls<T>(int, int, const int32_t*, const int32_t*, const T*, const uint8_t*, const int32_t*,       \
                              const T*, int, int, const double*, int, int, int, double, int32_t*, T*, int32_t*,     \
                              cudaStream_t, int*, const LsOut&);                                                    \
    template int interp_learned<T>(int, int, const int32_t*, const int32_t*, const T*, const uint8_t*, const int32_t*,  \
                                   const T*, int, int, const double*, int, int, int, double, const Model*, bool,    \
                                   int32_t*, T*, int32_t*, cudaStream_t, int*);                                     \
    template void build_restriction<T>(const EllView<T>&, int, DevBuf<int32_t>&, DevBuf<int32_t>&, DevBuf<T>&,      \
                                       cudaStream_t);                                                               \
    template void galerkin<T>(const MatView<T>&, const T*, const int32_t*, const int32_t*, const T*,                \
                              const EllView<T>&, int, GalerkinOut<T>&, cudaStream_t, bool);                         \
    template int64_t galerkin_into<T>(const MatView<T>&, const T*, const EllView<T>&, int, int32_t*, int32_t*, T*,  \
                                      T*, int64_t, cudaStream_t);                                                   \
    template void galerkin_nnz<T>(GalerkinOut<T>&, cudaStream_t);                                                   \
    template void csr_to_dense<T>(int, const int32_t*, const int32_t*, const T*, double*, cudaStream_t);
INST(float)
INST(double)
#undef INST

}  // namespace bamg
