// Shared device helpers for the AMG/GCIN library (sm_103a).
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <string>

namespace amg {

// Process-wide count of kernels this library has launched (reported by
// amg_launch_count; every launch site is followed by AMG_COUNT()).
extern std::atomic<long long> g_launches;
#define AMG_COUNT() (::amg::g_launches.fetch_add(1, std::memory_order_relaxed))

constexpr int kBlock = 256;          // threads per block of the row kernels
constexpr int kNumSMs = 152;         // GB300

// Contiguous device arena: lay out every buffer with 256-byte alignment in
// one pass that only counts, allocate once, then lay out again for real.
struct Planner {
    char *base = nullptr;
    size_t off = 0;
    template <class T>
    T *take(size_t count) {
        size_t a = (off + 255) & ~static_cast<size_t>(255);
        off = a + count * sizeof(T);
        return base ? reinterpret_cast<T *>(base + a) : nullptr;
    }
};

// Sum over the TPR lanes of one row group (TPR divides 32; whole warp active).
template <int TPR, class T>
__device__ __forceinline__ T group_sum(T v) {
#pragma unroll
    for (int o = TPR / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, TPR);
    return v;
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP32 pair h + l (about 48 bits): sums that want more than FP32 where FP64
// would bind (GB300: 2 FP64 FMAs a clock and SM against 128 in FP32).
struct FloatPair {
    float h, l;
};
// a += p + e (Knuth's error-free sum; the _rn intrinsics keep the compiler
// from contracting it)
__device__ __forceinline__ void pair_add(FloatPair &a, float p, float e = 0.f) {
    const float s = __fadd_rn(a.h, p);
    const float z = __fadd_rn(s, -a.h);
    const float t = __fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -z)), __fadd_rn(p, -z));
    a.h = s;
    a.l = __fadd_rn(a.l, __fadd_rn(t, e));
}

// Dot product of one CSR row with a gathered operand, split over the TPR
// lanes of a row group: lane `lane` takes entries p0 + lane, p0 + lane + TPR,
// ... and adds them in that order.  Each step issues the col / value loads of
// four entries before their four gathers, so a lane has up to eight loads in
// flight instead of one dependent pair per entry.
template <int TPR, class T, class X>
__device__ __forceinline__ T row_dot(int lane, int p0, int e, const int *__restrict__ col,
                                     const T *__restrict__ val, const X &xg) {
    T acc = T(0);
    for (int base = p0 + lane; base < e; base += 4 * TPR) {
        int c[4];
        T v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = base + j * TPR;
            c[j] = p < e ? __ldg(col + p) : 0;
            v[j] = p < e ? __ldg(val + p) : T(0);
        }
        T x[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j] = (base + j * TPR < e) ? xg(c[j]) : T(0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (base + j * TPR < e) acc += v[j] * x[j];
    }
    return acc;
}

// The first batch of a row-group lane's entries (row bounds, columns and
// values), fetched before griddepcontrol.wait: matrices do not change while
// a V-cycle runs, so these loads overlap the previous kernel and only the
// gathers of the vector it produced remain after the wait.
template <class T> struct RowBatch {
    int base = 0, e = 0, row = 0;
    int c[4] = {0, 0, 0, 0};
    T v[4] = {T(0), T(0), T(0), T(0)};
};

// An ordinary load that is issued here: the compiler would sink the load of a
// row's own value (b_i, u_i) to its use behind the row's sum, where it costs a
// memory round trip of its own; issued with the gathers it costs none (2.5M
// rows: residual pass 32.9 -> 30.5 us; 280k rows: 4.5 -> 4.2 us).
__device__ __forceinline__ float load_now(const float *p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double load_now(const double *p) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

// Loads whose lines leave L2 first (a policy made once per thread).
__device__ __forceinline__ unsigned long long evict_first_policy() {
    unsigned long long pol;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ float load_passing(const float *p, unsigned long long pol) {
    float v;
    asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ double load_passing(const double *p, unsigned long long pol) {
    double v;
    asm("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
    return v;
}

// How a pass reads its columns and values and which block of rows a CTA takes.
// const int *: CSR columns.  ColDelta: columns of a square matrix stored as
// 16-bit offsets from the row (j = i + d_p; used where every |j - i| < 2^15,
// e.g. a mesh in RCM order), 2 instead of 4 bytes per entry on the HBM-bound
// passes.  ColStream: the same on a level whose A and Q^-1 together pass L2.
// Its values come back only after the other matrix has passed, so they leave
// L2 first and the columns (shared by A and Q^-1) and vectors stay; and
// every other pass takes the rows in reverse, starting with what the pass
// before it touched last.
struct ColDelta {
    const short *__restrict__ d;
};
struct ColStream {
    const short *__restrict__ d;
    int reverse;
};
__device__ __forceinline__ int col_at(const int *__restrict__ col, int p, int) { return __ldg(col + p); }
__device__ __forceinline__ int col_at(const ColDelta &cd, int p, int row) { return row + static_cast<int>(__ldg(cd.d + p)); }
__device__ __forceinline__ int col_at(const ColStream &cd, int p, int row) { return row + static_cast<int>(__ldg(cd.d + p)); }
template <class CS> __device__ __forceinline__ int pass_block(const CS &) { return blockIdx.x; }
__device__ __forceinline__ int pass_block(const ColStream &cs) { return cs.reverse ? gridDim.x - 1 - blockIdx.x : blockIdx.x; }
template <class T, class CS> __device__ __forceinline__ T val_at(const T *__restrict__ val, int p, const CS &, unsigned long long) { return __ldg(val + p); }
template <class T> __device__ __forceinline__ T val_at(const T *__restrict__ val, int p, const ColStream &, unsigned long long pol) { return load_passing(val + p, pol); }
template <class CS> __device__ __forceinline__ unsigned long long pass_policy(const CS &) { return 0; }
__device__ __forceinline__ unsigned long long pass_policy(const ColStream &) { return evict_first_policy(); }

template <int TPR, class T, class CS>
__device__ __forceinline__ void row_prefetch(RowBatch<T> &rb, bool live, int lane, const int *__restrict__ rp,
                                             int row, const CS &col, const T *__restrict__ val) {
    if (!live) return;
    const int p0 = __ldg(rp + row);
    rb.e = __ldg(rp + row + 1);
    rb.base = p0 + lane;
    rb.row = row;
    const unsigned long long pol = pass_policy(col);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int p = rb.base + j * TPR;
        rb.c[j] = p < rb.e ? col_at(col, p, row) : 0;
        rb.v[j] = p < rb.e ? val_at(val, p, col, pol) : T(0);
    }
}

// row_dot with the first batch taken from a RowBatch (same entries, same order).
template <int TPR, class T, class CS, class X>
__device__ __forceinline__ T row_dot_pref(const RowBatch<T> &rb, const CS &col,
                                          const T *__restrict__ val, const X &xg) {
    T acc = T(0);
    if (rb.base >= rb.e) return acc;
    T x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) x[j] = (rb.base + j * TPR < rb.e) ? xg(rb.c[j]) : T(0);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (rb.base + j * TPR < rb.e) acc += rb.v[j] * x[j];
    const unsigned long long pol = pass_policy(col);
    for (int base = rb.base + 4 * TPR; base < rb.e; base += 4 * TPR) {
        int c[4];
        T v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int p = base + j * TPR;
            c[j] = p < rb.e ? col_at(col, p, rb.row) : 0;
            v[j] = p < rb.e ? val_at(val, p, col, pol) : T(0);
        }
        T y[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) y[j] = (base + j * TPR < rb.e) ? xg(c[j]) : T(0);
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (base + j * TPR < rb.e) acc += v[j] * y[j];
    }
    return acc;
}

template <class T> struct Gather {
    const T *__restrict__ x;
    __device__ __forceinline__ T operator()(int j) const { return x[j]; }
};

// Programmatic dependent launch (PDL).  A solve-path kernel first waits for
// its predecessor grid to finish and flush (griddepcontrol.wait), touching no
// memory before that, then lets its own dependents start launching, so the
// next kernel's launch and block scheduling overlap this kernel's tail.
__device__ __forceinline__ void pdl_wait_and_release() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       Args... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
    AMG_COUNT();
}

// Threads per row of the row-group CSR kernels (a power of two, 1..32).
// Large matrices (>= 2^21 entries, HBM-bound) get about four entries per
// lane, one four-deep load batch per lane with the most rows per warp;
// smaller ones (L2-resident, latency-bound) about two, so more lanes share
// each row's short dependent chain.  Measured on GB300: the 2.5M-row
// residual pass 48 -> 41 us, the 50k-row V-cycle 103 -> 92 us against a
// uniform three entries per lane.
inline int pick_tpr(long long nnz, int n) {
    if (n <= 0) return 1;
    const double per_lane = static_cast<double>(nnz) / n / (nnz >= (1LL << 21) ? 4.0 : 2.0);
    int t = 1;
    while (t * 2 <= per_lane && t < 32) t *= 2;
    return t;
}

inline int grid_for(long long threads) {
    long long g = (threads + kBlock - 1) / kBlock;
    return static_cast<int>(g < 1 ? 1 : g);
}

}  // namespace amg
