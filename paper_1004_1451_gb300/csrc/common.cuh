// Shared host/device helpers of the GB300 Bootstrap AMG library.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <iterator>
#include <map>
#include <set>
#include <stdexcept>
#include <string>
#include <utility>
#include <vector>

#include "../../include/bamg.h"

namespace bamg {

struct Error : std::runtime_error {
    int code;
    Error(int c, const std::string& m) : std::runtime_error(m), code(c) {}
};

void count_launch();
void count_launches(int64_t k);  // adds k (may be negative: graph capture bookkeeping)
void set_last_error(const std::string& msg);

#define BAMG_CK(call)                                                                              \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            cudaGetLastError(); /* this call's answer, not the next launch's */                     \
            throw ::bamg::Error(e_ == cudaErrorMemoryAllocation ? BAMG_ENOMEM : BAMG_ECUDA,        \
                                std::string(#call) + ": " + cudaGetErrorString(e_));               \
        }                                                                                          \
    } while (0)

#define BAMG_REQUIRE(cond, code, msg)                                                              \
    do {                                                                                           \
        if (!(cond)) throw ::bamg::Error((code), (msg));                                           \
    } while (0)

// Programmatic dependent launch: while pdl_enabled() is set (the default; BAMG_PDL=0 in
// the environment clears it) every launch lets the kernel start before its predecessor in
// the stream finishes.  Every kernel of the library calls pdl_begin() before its first
// access to memory written by earlier work: it waits until the predecessor grid has
// completed and its writes are visible, and signals that its own dependents may launch.
// Without the attribute both instructions return at once.
bool& pdl_enabled();
__device__ __forceinline__ void pdl_begin() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" :::);
}
struct PdlScope {
    bool prev;
    PdlScope() : prev(pdl_enabled()) { pdl_enabled() = true; }
    ~PdlScope() { pdl_enabled() = prev; }
};
#define BAMG_LAUNCH_PDL(kernel, grid, block, smem, strm_, ...)                                      \
    do {                                                                                           \
        if (::bamg::pdl_enabled()) {                                                               \
            cudaLaunchConfig_t cfg_ = {};                                                          \
            cfg_.gridDim = dim3(grid);                                                             \
            cfg_.blockDim = dim3(block);                                                           \
            cfg_.dynamicSmemBytes = (smem);                                                        \
            cfg_.stream = (strm_);                                                                  \
            cudaLaunchAttribute at_[1];                                                            \
            at_[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;                        \
            at_[0].val.programmaticStreamSerializationAllowed = 1;                                 \
            cfg_.attrs = at_;                                                                      \
            cfg_.numAttrs = 1;                                                                     \
            BAMG_CK(cudaLaunchKernelEx(&cfg_, kernel, __VA_ARGS__));                               \
        } else {                                                                                   \
            kernel<<<(grid), (block), (smem), (strm_)>>>(__VA_ARGS__);                              \
        }                                                                                          \
        ::bamg::count_launch();                                                                    \
        BAMG_CK(cudaGetLastError());                                                               \
    } while (0)
// Every kernel of the library goes through this macro so the process-wide launch
// counter is exact.
#define BAMG_LAUNCH(kernel, grid, block, smem, stream, ...) \
    BAMG_LAUNCH_PDL(kernel, grid, block, smem, stream, __VA_ARGS__)

inline unsigned blocks_for(int64_t work, int per_block) {
    int64_t b = (work + per_block - 1) / per_block;
    return (unsigned)(b < 1 ? 1 : b);
}

// Device memory comes from a pool of the library's own (one per device, made at its first use):
// cudaMallocAsync's default pool gives every unused byte back to the system at each
// synchronisation, and mapping a call's temporaries again took 100 to 400 us (two thirds of a
// galerkin call).  This pool keeps up to MEM_POOL_KEEP unused bytes at a synchronisation and gives the
// rest back; bamg_release_memory() gives back the rest too.  Blocks are ordered by stream as
// cudaMallocAsync's are, across threads and streams.
constexpr uint64_t MEM_POOL_KEEP = uint64_t(512) << 20;
void pool_alloc(void** p, size_t bytes, cudaStream_t s);
void pool_trim();  // of the current device

// A solver's small long-lived buffers: slices of chunks from the pool, given out by size and taken
// back into a free list (at once, for buffers are reused in the order of the solver's streams, which
// are fenced against one another).  A setup allocates some 200 of them, at 2 us each, and at 30 us with
// eight host threads in the allocator at a time.  Blocks above MAX_SLICE come from the pool
// directly.  The chunks are freed with the solver, so what they hold beyond its buffers is a live handle's
// cost: the first has the size that the owner expects, each later one a sixth of what is there; a free slice
// larger than asked for gives up its rest, and neighbours that are free join.  (With chunks from 2 MiB
// doubling up to 32 and whole slices up to twice the size, 62 MiB of chunks held 27 of buffers on
// 200 x 200 states in FP64, now 33.)
struct DevArena {
    static constexpr size_t MAX_SLICE = size_t(4) << 20, MIN_CHUNK = size_t(512) << 10, MAX_CHUNK = size_t(24) << 20;
    struct Chunk {
        char* base;
        size_t cap, top;
        cudaStream_t s;
    };
    struct Slice {
        size_t bytes;
        size_t chunk;
        bool free;
    };
    std::vector<Chunk> chunks;
    std::map<char*, Slice> slices;              // every slice, in the order of addresses
    std::set<std::pair<size_t, char*>> unused;  // the free ones by size
    size_t held = 0, first = 0;
    void expect(size_t bytes) { first = bytes < MAX_CHUNK ? (bytes + 255) & ~size_t(255) : MAX_CHUNK; }
    void* alloc(size_t bytes, cudaStream_t s) {
        bytes = (bytes + 255) & ~size_t(255);
        const auto it = unused.lower_bound({bytes, nullptr});
        if (it != unused.end()) {
            char* p = it->second;
            unused.erase(it);
            Slice& sl = slices.at(p);
            sl.free = false;
            if (sl.bytes > bytes) {
                slices.emplace(p + bytes, Slice{sl.bytes - bytes, sl.chunk, true});
                unused.insert({sl.bytes - bytes, p + bytes});
                sl.bytes = bytes;
            }
            return p;
        }
        if (chunks.empty() || chunks.back().top + bytes > chunks.back().cap) {
            if (!chunks.empty() && chunks.back().top < chunks.back().cap) {  // its rest, for smaller buffers
                Chunk& c = chunks.back();
                slices.emplace(c.base + c.top, Slice{c.cap - c.top, chunks.size() - 1, true});
                unused.insert({c.cap - c.top, c.base + c.top});
                c.top = c.cap;
            }
            const size_t next = chunks.empty() ? first : (held / 6 + 255) & ~size_t(255);
            const size_t cap = next < MIN_CHUNK ? MIN_CHUNK : next < MAX_CHUNK ? next : MAX_CHUNK;
            Chunk c{nullptr, cap > bytes ? cap : bytes, 0, s};
            pool_alloc((void**)&c.base, c.cap, s);
            chunks.push_back(c);
            held += c.cap;
        }
        Chunk& c = chunks.back();
        char* p = c.base + c.top;
        c.top += bytes;
        slices.emplace(p, Slice{bytes, chunks.size() - 1, false});
        return p;
    }
    void free(void* q) {
        auto it = slices.find((char*)q);
        it->second.free = true;
        const auto join = [&](std::map<char*, Slice>::iterator lo, std::map<char*, Slice>::iterator hi) {
            lo->second.bytes += hi->second.bytes;
            slices.erase(hi);
        };
        const auto next = std::next(it);
        if (next != slices.end() && next->second.free && next->second.chunk == it->second.chunk) {
            unused.erase({next->second.bytes, next->first});
            join(it, next);
        }
        if (it != slices.begin()) {
            const auto prev = std::prev(it);
            if (prev->second.free && prev->second.chunk == it->second.chunk) {
                unused.erase({prev->second.bytes, prev->first});
                join(prev, it);
                it = prev;
            }
        }
        unused.insert({it->second.bytes, it->first});
    }
    DevArena() = default;
    ~DevArena() {
        for (Chunk& c : chunks) cudaFreeAsync(c.base, c.s);
    }
    DevArena(const DevArena&) = delete;
    DevArena& operator=(const DevArena&) = delete;
};

// Stream on which DevBuf allocations are ordered (set by the owner of the work: the
// handle's stream during setup and solve), and the arena small ones come from (null: the pool).
// Thread-local.
cudaStream_t& alloc_stream();
DevArena*& dev_arena();
// Sets both for a scope.
struct AllocStream {
    cudaStream_t prev;
    DevArena* prev_a;
    explicit AllocStream(cudaStream_t s, DevArena* a = nullptr) : prev(alloc_stream()), prev_a(dev_arena()) {
        alloc_stream() = s;
        dev_arena() = a;
    }
    ~AllocStream() {
        alloc_stream() = prev;
        dev_arena() = prev_a;
    }
};

// Owning device buffer from the arena or the pool, ordered on alloc_stream(), so building a
// hierarchy does not synchronise the device for every allocation.
// Callers synchronise their streams before the owner is destroyed.
template <typename T>
struct DevBuf {
    T* p = nullptr;
    size_t n = 0;
    cudaStream_t s = nullptr;
    DevArena* a = nullptr;
    DevBuf() = default;
    explicit DevBuf(size_t n_) { alloc(n_); }
    void alloc(size_t n_) {
        release();
        s = alloc_stream();
        const size_t bytes = n_ * sizeof(T);
        a = bytes <= DevArena::MAX_SLICE ? dev_arena() : nullptr;
        if (n_) {
            if (a)
                p = static_cast<T*>(a->alloc(bytes, s));
            else
                pool_alloc((void**)&p, bytes, s);
        }
        n = n_;
    }
    void ensure(size_t n_) {
        if (n_ > n) alloc(n_);
    }
    void release() {
        if (p) {
            if (a)
                a->free(p);
            else
                cudaFreeAsync(p, s);
        }
        p = nullptr;
        n = 0;
    }
    ~DevBuf() { release(); }
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    DevBuf(DevBuf&& o) noexcept : p(o.p), n(o.n), s(o.s), a(o.a) { o.p = nullptr; o.n = 0; }
    DevBuf& operator=(DevBuf&& o) noexcept {
        release();
        p = o.p;
        n = o.n;
        s = o.s;
        a = o.a;
        o.p = nullptr;
        o.n = 0;
        return *this;
    }
    T* get() const { return p; }
};

// A block of mapped pinned host memory (PINNED_SLOT bytes), from pages that live as long as the
// process: a cudaHostAlloc takes 130 us and stops the other threads' allocations.
constexpr size_t PINNED_SLOT = 256;
void* pinned_acquire();
void pinned_release(void* p);

// Stack allocator for the temporaries of one stream: chunks from the stream-ordered pool,
// handed out in 256-byte aligned slices and taken back when the slices are released (any
// order; space is reclaimed from the top).  A slice released here can be handed out again
// at once: its next user is ordered after its last one on the same stream.  Spares the
// pool calls of the many short-lived buffers of a setup.
struct StackArena {
    struct Chunk {
        char* base;
        size_t cap, top;
    };
    struct Slice {
        int chunk;
        size_t prev;
        char* p;
        bool live;
    };
    cudaStream_t s;
    std::vector<Chunk> chunks;
    std::vector<Slice> stack;
    static constexpr size_t MIN_CHUNK = size_t(16) << 20;
    explicit StackArena(cudaStream_t st) : s(st) {}
    void* push(size_t bytes) {
        bytes = (bytes + 255) & ~size_t(255);
        size_t c = stack.empty() ? 0 : (size_t)stack.back().chunk;
        while (c < chunks.size() && chunks[c].top + bytes > chunks[c].cap) ++c;
        if (c == chunks.size()) {
            Chunk k{nullptr, bytes > MIN_CHUNK ? bytes : MIN_CHUNK, 0};
            pool_alloc((void**)&k.base, k.cap, s);
            chunks.push_back(k);
        }
        Chunk& k = chunks[c];
        stack.push_back(Slice{(int)c, k.top, k.base + k.top, true});
        k.top += bytes;
        return stack.back().p;
    }
    void pop(void* p) {
        for (size_t q = stack.size(); q-- > 0;)
            if (stack[q].p == p && stack[q].live) {
                stack[q].live = false;
                break;
            }
        while (!stack.empty() && !stack.back().live) {
            chunks[stack.back().chunk].top = stack.back().prev;
            stack.pop_back();
        }
    }
    // returns the chunks to the pool once no slice is live
    void release() {
        if (!stack.empty()) return;
        for (Chunk& k : chunks) cudaFreeAsync(k.base, s);
        chunks.clear();
    }
    ~StackArena() {
        stack.clear();
        release();
    }
    StackArena(const StackArena&) = delete;
    StackArena& operator=(const StackArena&) = delete;
};
// The arena that TmpBufs on its stream draw from (thread-local; null: the pool directly).
StackArena*& tmp_arena();
struct ArenaScope {  // sets tmp_arena() for a scope and releases the arena's chunks after
    StackArena* prev;
    StackArena& a;
    explicit ArenaScope(StackArena& a_) : prev(tmp_arena()), a(a_) { tmp_arena() = &a; }
    ~ArenaScope() {
        tmp_arena() = prev;
        a.release();
    }
};

// Stream-ordered temporary: a slice of the current StackArena when it serves this stream,
// else a block of the pool.
template <typename T>
struct TmpBuf {
    T* p = nullptr;
    cudaStream_t s = nullptr;
    StackArena* a = nullptr;
    TmpBuf(size_t n, cudaStream_t st) : s(st) {
        if (!n) return;
        StackArena* cur = tmp_arena();
        if (cur && cur->s == st) {
            a = cur;
            p = static_cast<T*>(a->push(n * sizeof(T)));
        } else {
            pool_alloc((void**)&p, n * sizeof(T), s);
        }
    }
    ~TmpBuf() {
        if (!p) return;
        if (a)
            a->pop(p);
        else
            cudaFreeAsync(p, s);
    }
    TmpBuf(const TmpBuf&) = delete;
    TmpBuf& operator=(const TmpBuf&) = delete;
    T* get() const { return p; }
};

// ------------------------------------------------------------------ device helpers
// SplitMix64 (Steele, Lea, Flood, OOPSLA 2014): state s + t * gamma, then the published
// 64-bit finaliser.  Draw number (stream * 2^40 + idx + 1) of `seed`.
__host__ __device__ __forceinline__ uint64_t splitmix64_output(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
__host__ __device__ __forceinline__ uint64_t counter_u64(uint64_t seed, uint64_t stream, uint64_t idx) {
    uint64_t ctr = stream * (1ull << 40) + idx + 1ull;
    return splitmix64_output(seed + ctr * 0x9E3779B97F4A7C15ull);
}
__device__ __forceinline__ double counter_uniform(uint64_t seed, uint64_t stream, uint64_t idx) {
    return (double)(counter_u64(seed, stream, idx) >> 11) * 0x1.0p-53;
}

constexpr uint64_t STREAM_TV = 0;
constexpr uint64_t STREAM_CR = 1ull << 22;
constexpr uint64_t STREAM_MIS = 1ull << 23;
constexpr uint64_t STREAM_COLOUR = 1ull << 21;  // + (level << 8) + colour: the smoother's colouring

// 16-byte vector of T: 2 doubles or 4 floats.
template <typename T>
struct V16;
template <>
struct V16<double> {
    using type = double2;
    static constexpr int W = 2;
    __device__ static void load(const double* p, double* o) {
        double2 v = *reinterpret_cast<const double2*>(p);
        o[0] = v.x;
        o[1] = v.y;
    }
    __device__ static void store(double* p, const double* o) { *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]); }
};
template <>
struct V16<float> {
    using type = float4;
    static constexpr int W = 4;
    __device__ static void load(const float* p, float* o) {
        float4 v = *reinterpret_cast<const float4*>(p);
        o[0] = v.x;
        o[1] = v.y;
        o[2] = v.z;
        o[3] = v.w;
    }
    __device__ static void store(float* p, const float* o) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    }
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Multiply and add with rounding after each operation (no contraction into an FMA),
// so that sums computed in the same order match a plain CPU evaluation bit for bit.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// w / h rounded to nearest, given r = 1 / h rounded to nearest: q0 = w r lies within an ulp
// of the quotient, the remainder w - q0 h is exact in one fma, and q0 + rem r rounded once is
// the correctly rounded quotient (Markstein's theorem: P. Markstein, IBM J. Res. Dev. 34(1),
// 1990).  Three FP64 operations instead of a full division, for the many quotients by one
// divisor; it holds for quotients in the normal range.  A zero remainder keeps q0, and with
// it the sign of a zero quotient.
__device__ __forceinline__ double div_by_recip(double w, double h, double r) {
    const double q0 = __dmul_rn(w, r);
    const double rem = __fma_rn(-q0, h, w);
    return rem == 0.0 ? q0 : __fma_rn(rem, r, q0);
}

// ------------------------------------------------------------------ host helpers
// d_out has n + 1 entries; with h_total (the device address of mapped host memory) the total
// is also stored there
void exclusive_scan(const int32_t* d_in, int32_t* d_out, int n, cudaStream_t s, int32_t* h_total = nullptr);
int32_t exclusive_scan_total(const int32_t* d_in, int32_t* d_out, int n, cudaStream_t s);  // the total, to the host
int32_t read_int(const int32_t* d_p, cudaStream_t s);  // a device int, to the host (after s's earlier work)
// Up to 16 doubles a kernel posts to this thread's mapped host block: host_post_begin before the
// launch, host_post by one thread of the kernel, host_post_wait after it.  The same block carries
// read_int's and the scans' counts: one at a time.
struct HostPost {
    int32_t* flag = nullptr;
    double* val = nullptr;
};
HostPost host_post_begin();
void host_post_wait(double* out, int k, cudaStream_t s);
__device__ __forceinline__ void host_post(const HostPost& p, const double* v, int k) {
    for (int q = 0; q < k; ++q) *(volatile double*)(p.val + q) = v[q];
    __threadfence_system();
    *(volatile int32_t*)p.flag = 1;
    __threadfence_system();
}

}  // namespace bamg
