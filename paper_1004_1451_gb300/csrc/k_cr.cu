// Compatible-relaxation coarsening, Algorithm 1 (Section 3.1): an independent set of
// the graph of B to start, then rounds of nu F-relaxation sweeps (Eq. (3.2)) from random
// starts in [1, 2); while the convergence estimate of Eq. (3.3) exceeds theta, an
// independent set of the slow points joins C.  Independent sets use Luby's rule with
// fixed SplitMix64 priorities: an undecided candidate enters when its key (priority,
// index) beats every undecided neighbour's, after which its undecided neighbours leave.
#include <algorithm>

#include "kernels.cuh"

namespace bamg {

__global__ void k_tcount(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                         int32_t* __restrict__ cnt) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int p = rp[i]; p < rp[i + 1]; ++p)
        if (ci[p] != i) atomicAdd(cnt + ci[p], 1);
}
__global__ void k_tfill(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                        const int32_t* __restrict__ rpT, int32_t* __restrict__ cursor, int32_t* __restrict__ ciT) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int p = rp[i]; p < rp[i + 1]; ++p) {
        const int j = ci[p];
        if (j != i) ciT[rpT[j] + atomicAdd(cursor + j, 1)] = i;
    }
}

__device__ __forceinline__ bool beats(uint64_t pi, int i, uint64_t pj, int j) { return pi > pj || (pi == pj && i > j); }

// The independent set in one launch.  Luby's rule with fixed priorities picks the greedy set by
// descending priority whatever the rounds: a candidate is in when every neighbour that beats it is out,
// and out when one of those is in.  So no round needs to end before the next begins: a thread looks
// again at the neighbours that beat it (their states change once, and only from undecided) until its
// own is settled, at most MIS_LOOKS times; what is left undecided (neighbours whose blocks had not
// started, long chains) the next launch settles.  Rounds as two kernels each, four rounds between the
// host's checks, took 8 launches and 46 us where one and 24 us do (planar walk of 65,536 states).
// st: 1 undecided candidate, 0 no candidate or out, 2 in.
//
// G lanes share a row on levels of long rows (lanes_per_row): one lane looking at a row's 30 to 70
// neighbours, one dependent load after the other, took most of the sets' time (46 us a set on average over
// a planar chain of 2^18 states; 24 on its long-row levels with the lanes).
constexpr int MIS_LOOKS = 24;
template <int G>
__global__ void __launch_bounds__(256, 8)
    k_mis(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci, const int32_t* __restrict__ rpT,
          const int32_t* __restrict__ ciT, uint8_t* st, uint8_t* __restrict__ chosen, uint64_t seed, uint64_t stream,
          int* __restrict__ left) {
    pdl_begin();
    constexpr unsigned ALL = 0xffffffffu;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(t / G), sub = (int)(t % G);
    volatile uint8_t* vst = st;
    bool done = i >= n || vst[i] != 1;  // the same in a row's lanes: only they change its state
    if (G == 1 ? done : !__any_sync(ALL, !done)) return;
    // true if p is in any of the row's lanes (all lanes of the warp take part)
    auto any = [&](bool p) {
        if constexpr (G == 1) return p;
        return ((__ballot_sync(ALL, p) >> ((threadIdx.x & 31) & ~(G - 1))) & (ALL >> (32 - G))) != 0;
    };
    const uint64_t pi = counter_u64(seed, stream, (uint64_t)i);
    const int a = done ? 0 : rp[i], na = done ? 0 : rp[i + 1] - a, b = done ? 0 : rpT[i],
              tot = done ? 0 : na + rpT[i + 1] - b;
    auto neighbour = [&](int k) { return k < na ? ci[a + k] : ciT[b + k - na]; };
    unsigned long long beat = 0ull;  // the undecided neighbours that beat i, among this lane's first 64
    bool out = false, wait = false;
    // four neighbours at a time: their states are loaded without waiting for one another (one at a time the
    // set took 30 us).  More lanes a row than lanes_per_row took 12, but the looks then ran out before the
    // chains of waiting rows had settled: the second launch, or four times the looks, cost more (10 us a call).
    constexpr int U = 4;
    auto scan = [&](int k0) {
        for (int k = k0; k < tot && !out; k += U * G) {
            int j[U], q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) j[u] = k + u * G < tot ? neighbour(k + u * G) : i;
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = j[u] != i ? vst[j[u]] : 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (q[u] == 0 || beats(pi, i, counter_u64(seed, stream, (uint64_t)j[u]), j[u])) continue;
                out |= q[u] == 2;
                wait = true;
                if (k + u * G < 64 * G) beat |= 1ull << ((k + u * G) / G);
            }
        }
    };
    scan(sub);
    // settled in the loop, not after it: lanes of the same warp wait for one another
    auto settle = [&] {
        const bool o = any(out), w = any(wait);
        if (done) return;
        done = o || !w;
        if (!done || sub != 0) return;
        vst[i] = o ? 0 : 2;
        if (!o) chosen[i] = 1;
    };
    settle();
    for (int look = 0; look < MIS_LOOKS; ++look) {
        if (G == 1 ? done : !__any_sync(ALL, !done)) break;
        out = wait = false;
        if (!done) {
            for (unsigned long long m = beat; m && !out;) {
                int k[U], q[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    k[u] = m ? __ffsll((long long)m) - 1 : -1;
                    m &= m - 1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) q[u] = k[u] >= 0 ? vst[neighbour(sub + k[u] * G)] : 0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (q[u] == 0 && k[u] >= 0) beat &= ~(1ull << k[u]);
                    out |= q[u] == 2;
                    wait |= q[u] == 1;
                }
            }
            scan(sub + 64 * G);
        }
        settle();
    }
    if (!done && sub == 0) atomicAdd(left, 1);
}

// chosen |= independent set of the candidates (und: 1 on entry; consumed)
static void independent_set(int n, int nnz, const int32_t* rp, const int32_t* ci, const int32_t* rpT,
                            const int32_t* ciT, uint8_t* und, uint8_t* chosen, int* left, uint64_t seed, uint64_t stream,
                            cudaStream_t s) {
    const int G = lanes_per_row(n, nnz);
    for (int round = 0; round <= n; ++round) {  // every launch settles at least one
        BAMG_CK(cudaMemsetAsync(left, 0, sizeof(int), s));
        auto go = [&](auto kern) {
            BAMG_LAUNCH(kern, blocks_for((int64_t)n * G, 256), 256, 0, s, n, rp, ci, rpT, ciT, und, chosen, seed, stream,
                        left);
        };
        switch (G) {
            case 1: go(k_mis<1>); break;
            case 4: go(k_mis<4>); break;
            case 8: go(k_mis<8>); break;
            case 16: go(k_mis<16>); break;
            default: go(k_mis<32>);
        }
        if (read_int(left, s) == 0) return;
    }
    throw Error(BAMG_ETIMEOUT, "independent set did not terminate");
}

// u = 0 on C, the round's random start on F; in the first round (w given) also w_i = omega / b_ii
template <typename T>
__global__ void k_cr_start(int n, const uint8_t* __restrict__ cf, double* __restrict__ u, uint64_t seed,
                           uint64_t stream, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                           const T* __restrict__ bv, double omega, double* __restrict__ w) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    u[i] = cf[i] ? 0.0 : 1.0 + counter_uniform(seed, stream, (uint64_t)i);
    if (w) {
        double d = 0.0;
        for (int p = rp[i]; p < rp[i + 1]; ++p)
            if (ci[p] == i) d = (double)bv[p];
        w[i] = omega * (1.0 / d);
    }
}

// s + b u; a point of C (u = +0) takes no part, whatever the entry's value
__device__ __forceinline__ double cr_term(double s, double b, double u) {
    return __double_as_longlong(u) != 0 ? s + b * u : s;
}

// One F-relaxation sweep.  u is 0 on C and tells the C entries of the row: no load of the flag between
// the index and u.
// The quotient omega / b_ii comes from k_cr_start: an FP64 division a row and sweep took a third of
// the sweep's time on the FP64 pipe (32 us a sweep of 2^18 rows).
template <typename T>
__global__ void k_frelax(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                         const T* __restrict__ bv, const uint8_t* __restrict__ cf, const double* __restrict__ w,
                         const double* __restrict__ u, double* __restrict__ un) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (cf[i]) {
        un[i] = 0.0;
        return;
    }
    double s = 0.0;
    int p = rp[i];
    const int pe = rp[i + 1];
    for (; p + 4 <= pe; p += 4) {  // loads before their uses
        const int j0 = ci[p], j1 = ci[p + 1], j2 = ci[p + 2], j3 = ci[p + 3];
        const T b0 = bv[p], b1 = bv[p + 1], b2 = bv[p + 2], b3 = bv[p + 3];
        const double u0 = u[j0], u1 = u[j1], u2 = u[j2], u3 = u[j3];
        s = cr_term(s, (double)b0, u0);
        s = cr_term(s, (double)b1, u1);
        s = cr_term(s, (double)b2, u2);
        s = cr_term(s, (double)b3, u3);
    }
    for (; p < pe; ++p) s = cr_term(s, (double)bv[p], u[ci[p]]);
    un[i] = u[i] - w[i] * s;
}

// k_frelax with G lanes per row (long rows of coarse levels): strided partial sums added
// by a butterfly.
template <typename T, int G>
__global__ void k_frelax_grp(int n, const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                             const T* __restrict__ bv, const uint8_t* __restrict__ cf, const double* __restrict__ w,
                             const double* __restrict__ u, double* __restrict__ un) {
    pdl_begin();
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int i = (int)(t / G), sub = (int)(t % G);
    double s = 0.0;
    const bool live = i < n && !cf[i];
    if (live) {
        const int pe = rp[i + 1];
#pragma unroll 4
        for (int p = rp[i] + sub; p < pe; p += G) s = cr_term(s, (double)bv[p], u[ci[p]]);
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (i < n && sub == 0) un[i] = live ? u[i] - w[i] * s : 0.0;
}

// sum u0^2 and sum u^2: per-block partials, added up by the block that finishes last (a fixed order)
// and posted to the host.  One thread adding them one by one took 17 us for 256 blocks.
__global__ void __launch_bounds__(256) k_cr_norms(int n, const double* __restrict__ u0, const double* __restrict__ u,
                                                  double* partial, unsigned* __restrict__ ticket, HostPost post) {
    pdl_begin();
    __shared__ double sh[2][8];
    __shared__ int s_last;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double a = 0.0, b = 0.0;
    if (i < n) {
        a = u0[i] * u0[i];
        b = u[i] * u[i];
    }
    a = warp_sum(a);
    b = warp_sum(b);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        sh[0][wid] = a;
        sh[1][wid] = b;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
        partial[(int64_t)blockIdx.x * 2 + threadIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    a = b = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) {
        a += __ldcg(partial + 2 * k);
        b += __ldcg(partial + 2 * k + 1);
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) {
        sh[0][wid] = a;
        sh[1][wid] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = b = 0.0;
        for (int w = 0; w < 8; ++w) {
            a += sh[0][w];
            b += sh[1][w];
        }
        *ticket = 0u;
        const double v[2] = {a, b};
        host_post(post, v, 2);
    }
}

__global__ void k_cr_slow(int n, const uint8_t* __restrict__ cf, const double* __restrict__ up,
                          const double* __restrict__ u, double theta, uint8_t* __restrict__ cand) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    cand[i] = (!cf[i] && fabs(u[i]) / fabs(up[i]) > theta) ? 1 : 0;
}

__global__ void k_u8_to_i32(int n, const uint8_t* __restrict__ a, int32_t* __restrict__ b) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = a[i];
}
__global__ void k_cidx_from_scan(int n, const uint8_t* __restrict__ cf, const int32_t* __restrict__ sc,
                                 int32_t* __restrict__ cidx) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) cidx[i] = cf[i] ? sc[i] : -1;
}

template <typename T>
int coarsen_cr(const MatView<T>& B, int level, uint64_t seed, double theta, int nu, double omega, int max_rounds,
               uint8_t* cf, int32_t* cidx, int* nc_out, cudaStream_t s) {
    const int n = B.n;
    const unsigned g = blocks_for(n, 256);
    const int G = lanes_per_row(n, B.nnz);
    // one allocation: the transposed pattern (cnt and cursor adjacent; cnt is the scan's input and the
    // final numbering's), vectors, masks
    size_t used = 0;
    auto slice = [&](size_t bytes) {
        const size_t at = used;
        used += (bytes + 255) & ~size_t(255);
        return at;
    };
    const size_t ni = sizeof(int32_t) * (size_t)n, nd = sizeof(double) * (size_t)n;
    const size_t o_cnt = slice(2 * ni + 256), o_rpT = slice(ni + sizeof(int32_t)),
                 o_ciT = slice(sizeof(int32_t) * (size_t)std::max(B.nnz, 1)),  // bound: the off-diagonal entries of B
                 o_w = slice(nd), o_u0 = slice(nd), o_ua = slice(nd), o_ub = slice(nd),
                 o_part = slice(2 * sizeof(double) * g), o_und = slice(n), o_cand = slice(n);
    TmpBuf<char> work(used, s);
    char* m = work.get();
    int32_t *cnt = (int32_t*)(m + o_cnt), *cursor = cnt + n, *rpT = (int32_t*)(m + o_rpT), *ciT = (int32_t*)(m + o_ciT);
    unsigned* ticket = (unsigned*)(cursor + n);
    int* left = (int*)ticket + 1;
    double *w = (double*)(m + o_w), *u0 = (double*)(m + o_u0), *part = (double*)(m + o_part);
    uint8_t *und = (uint8_t*)(m + o_und), *cand = (uint8_t*)(m + o_cand);
    BAMG_CK(cudaMemsetAsync(cnt, 0, 2 * ni + 2 * sizeof(int32_t), s));
    BAMG_LAUNCH(k_tcount, g, 256, 0, s, n, B.rp, B.ci, cnt);
    exclusive_scan(cnt, rpT, n, s);
    BAMG_LAUNCH(k_tfill, g, 256, 0, s, n, B.rp, B.ci, (const int32_t*)rpT, cursor, ciT);
    BAMG_CK(cudaMemsetAsync(cf, 0, n, s));
    BAMG_CK(cudaMemsetAsync(und, 1, n, s));
    independent_set(n, B.nnz, B.rp, B.ci, rpT, ciT, und, cf, left, seed, STREAM_MIS + ((uint64_t)level << 8), s);
    int rounds = 0;
    double h[2];
    for (;;) {
        BAMG_LAUNCH(k_cr_start<T>, g, 256, 0, s, n, (const uint8_t*)cf, u0, seed,
                    STREAM_CR + ((uint64_t)level << 8) + rounds, B.rp, B.ci, B.v, omega, rounds == 0 ? w : (double*)nullptr);
        const double* cur = u0;
        double* prev = nullptr;
        double* bufs[2] = {(double*)(m + o_ua), (double*)(m + o_ub)};
        for (int k = 0; k < nu; ++k) {
            double* nxt = bufs[k & 1];
            auto sweep = [&](auto kern, unsigned grid) {
                BAMG_LAUNCH(kern, grid, 256, 0, s, n, B.rp, B.ci, B.v, (const uint8_t*)cf, (const double*)w, cur, nxt);
            };
            const unsigned gg = blocks_for((int64_t)n * G, 256);
            switch (G) {
                case 1: sweep(k_frelax<T>, g); break;
                case 4: sweep(k_frelax_grp<T, 4>, gg); break;
                case 8: sweep(k_frelax_grp<T, 8>, gg); break;
                case 16: sweep(k_frelax_grp<T, 16>, gg); break;
                default: sweep(k_frelax_grp<T, 32>, gg);
            }
            prev = const_cast<double*>(cur);
            cur = nxt;
        }
        const HostPost post = host_post_begin();
        BAMG_LAUNCH(k_cr_norms, g, 256, 0, s, n, (const double*)u0, cur, part, ticket, post);
        host_post_wait(h, 2, s);
        const double rho = std::pow(std::sqrt(h[1]) / std::sqrt(h[0]), 1.0 / nu);
        if (!(rho > theta) || rounds >= max_rounds || h[0] == 0.0) break;
        BAMG_LAUNCH(k_cr_slow, g, 256, 0, s, n, (const uint8_t*)cf, (const double*)prev, cur, theta, cand);
        ++rounds;
        independent_set(n, B.nnz, B.rp, B.ci, rpT, ciT, cand, cf, left, seed,
                        STREAM_MIS + ((uint64_t)level << 8) + rounds, s);
    }
    BAMG_LAUNCH(k_u8_to_i32, g, 256, 0, s, n, (const uint8_t*)cf, cnt);
    exclusive_scan(cnt, rpT, n, s);
    BAMG_LAUNCH(k_cidx_from_scan, g, 256, 0, s, n, (const uint8_t*)cf, (const int32_t*)rpT, cidx);
    *nc_out = read_int(rpT + n, s);
    return rounds;
}

// ---------------------------------------------------------------- colouring of the smoother
// Colour c = an independent set (the rule above, priority stream STREAM_COLOUR + (level <<
// 8) + c) of the states the earlier colours left, in the symmetrised graph of B, until
// every state has a colour.  The classes go out as one row list sorted by (colour, state)
// with host offsets ptr[0..ncol].
__global__ void k_colour_take(int n, const uint8_t* __restrict__ chosen, int c, int32_t* __restrict__ colour,
                              uint8_t* __restrict__ left, int* __restrict__ remaining) {
    pdl_begin();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (chosen[i]) {
        colour[i] = c;
        left[i] = 0;
    } else if (left[i]) {
        atomicAdd(remaining, 1);
    }
}

constexpr int MAX_COLOURS = 255;  // the stream encoding leaves 8 bits for the colour

void colour_classes(int n, int nnz, const int32_t* rp, const int32_t* ci, int level, uint64_t seed,
                    std::vector<int>& ptr, DevBuf<int32_t>& rows, cudaStream_t s) {
    const unsigned g = blocks_for(n, 256);
    TmpBuf<int32_t> cnt(n, s), rpT(n + 1, s), cursor(n, s);
    BAMG_CK(cudaMemsetAsync(cnt.get(), 0, sizeof(int32_t) * n, s));
    BAMG_CK(cudaMemsetAsync(cursor.get(), 0, sizeof(int32_t) * n, s));
    BAMG_LAUNCH(k_tcount, g, 256, 0, s, n, rp, ci, cnt.get());
    exclusive_scan(cnt.get(), rpT.get(), n, s);
    TmpBuf<int32_t> ciT(nnz > 0 ? nnz : 1, s);
    BAMG_LAUNCH(k_tfill, g, 256, 0, s, n, rp, ci, rpT.get(), cursor.get(), ciT.get());
    TmpBuf<uint8_t> left(n, s), und(n, s), chosen(n, s);
    TmpBuf<int32_t> colour(n, s);
    TmpBuf<int> rem(1, s), undecided(1, s);
    BAMG_CK(cudaMemsetAsync(left.get(), 1, n, s));
    int ncol = 0;
    for (int c = 0; c < MAX_COLOURS; ++c) {
        BAMG_CK(cudaMemcpyAsync(und.get(), left.get(), n, cudaMemcpyDeviceToDevice, s));
        BAMG_CK(cudaMemsetAsync(chosen.get(), 0, n, s));
        independent_set(n, nnz, rp, ci, rpT.get(), ciT.get(), und.get(), chosen.get(), undecided.get(), seed,
                        STREAM_COLOUR + ((uint64_t)level << 8) + (uint64_t)c, s);
        BAMG_CK(cudaMemsetAsync(rem.get(), 0, sizeof(int), s));
        BAMG_LAUNCH(k_colour_take, g, 256, 0, s, n, (const uint8_t*)chosen.get(), c, colour.get(), left.get(),
                    rem.get());
        if (read_int(rem.get(), s) == 0) {
            ncol = c + 1;
            break;
        }
    }
    BAMG_REQUIRE(ncol > 0, BAMG_ETIMEOUT, "colouring: more than 255 colours");
    std::vector<int32_t> hc(n), hr(n);
    BAMG_CK(cudaMemcpyAsync(hc.data(), colour.get(), sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    BAMG_CK(cudaStreamSynchronize(s));
    ptr.assign(ncol + 1, 0);
    for (int i = 0; i < n; ++i) ptr[hc[i] + 1]++;
    for (int c = 0; c < ncol; ++c) ptr[c + 1] += ptr[c];
    std::vector<int> at(ptr.begin(), ptr.end() - 1);
    for (int i = 0; i < n; ++i) hr[at[hc[i]]++] = i;  // ascending states within a colour
    rows.alloc(n);
    BAMG_CK(cudaMemcpyAsync(rows.get(), hr.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice, s));
    BAMG_CK(cudaStreamSynchronize(s));
}

template int coarsen_cr<float>(const MatView<float>&, int, uint64_t, double, int, double, int, uint8_t*, int32_t*,
                               int*, cudaStream_t);
template int coarsen_cr<double>(const MatView<double>&, int, uint64_t, double, int, double, int, uint8_t*, int32_t*,
                                int*, cudaStream_t);

}  // namespace bamg
