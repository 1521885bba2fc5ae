// GCIN coefficient network (Sec. 3.2, App. A.1; Algorithm 1 steps 1-6 and
// the network half of step 13) on sm_103a: forward, backward and Adam.
//
// The batch is the disjoint union of every level graph (Algorithm 1 step 5):
// one concatenated CSR whose entries are the edges (weight a_ij; the
// diagonal entry is the self-loop of A_hat with weight a_ii).  Nodes are cut
// into tiles of <= 64 consecutive nodes inside one graph; one block owns a
// tile.  Per layer (forward):
//   aggregation + linear   h_i = sum_j w_ij x_j, y = h Theta + b   (warp per
//                          node, lanes own feature pairs) and, in the same
//                          kernel, the tile's mean / M2 of y per feature
//   statistics             per graph: Chan combination of tile partials
//   normalise + pool       x = ReLU((y - mu) rstd gamma + beta) and the
//                          tile's sum / max / argmax of x
//   pooling                per graph: combination of tile partials
// Head (block per graph): 4 readout linears 128->32, LayerNorm(128),
// sigmoid, Linear 128->128 + ReLU, Linear 128->64 + ReLU, Linear 64->5.
// Backward mirrors these steps; every parameter gradient is a fixed-order
// sum of per-tile or per-graph partials, so gradients are bit-reproducible.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <mutex>
#include <vector>

#include "gcin.cuh"

namespace amg {

constexpr float kEps = 1e-5f;
__constant__ ParamLayout kPLd[2] = {make_layout(kHidden), make_layout(kHidden32)};   // device copies of the offsets
template <int H>
__device__ __forceinline__ const ParamLayout &PL() { return kPLd[H == kHidden ? 0 : 1]; }
template <int H>
__host__ __device__ constexpr int num_params() { return make_layout(H).total; }

// ---------------------------------------------------------------------------
// batch construction
// ---------------------------------------------------------------------------
__global__ void k_cat_graph(int n, int nnz, const int *__restrict__ rp, const int *__restrict__ col,
                            const double *__restrict__ v, const double *__restrict__ diag, int node_off,
                            int edge_off, int g, int *__restrict__ rp_out, int *__restrict__ col_out,
                            float *__restrict__ w_out, double *__restrict__ w64_out, double *__restrict__ x0,
                            int *__restrict__ gid) {
    const int t = blockIdx.x * kBlock + threadIdx.x;
    if (t < n) {
        rp_out[node_off + t] = rp[t] + edge_off;
        gid[node_off + t] = g;
        // raw features [a_ii, deg_i] (Algorithm 1 step 3; deg = off-diagonal
        // pattern entries, every row holding its diagonal)
        x0[2 * static_cast<size_t>(node_off + t)] = diag[t];
        x0[2 * static_cast<size_t>(node_off + t) + 1] = static_cast<double>(rp[t + 1] - rp[t] - 1);
    }
    if (t < nnz) {
        col_out[edge_off + t] = col[t] + node_off;
        w_out[edge_off + t] = static_cast<float>(v[t]);
        w64_out[edge_off + t] = v[t];
    }
}

__global__ void k_set_int(int *p, int v) { *p = v; }

void gcin_batch_free(GcinBatch &b) {
    if (b.arena) cudaFree(b.arena);
    b = GcinBatch{};
}

static void batch_layout(GcinBatch &b, Planner &pl, bool backward) {
    const size_t N = b.N, G = b.G, NT = b.NT, E = std::max<long long>(1, b.E);
    b.rp = pl.take<int>(N + 1);
    b.col = pl.take<int>(E);
    b.w = pl.take<float>(E);
    b.w64 = pl.take<double>(E);
    b.gptr = pl.take<int>(G + 1);
    b.gid = pl.take<int>(N);
    b.tstart = pl.take<int>(NT + 1);
    b.tgraph = pl.take<int>(NT);
    b.gtile = pl.take<int>(G + 1);
    const size_t NC = b.NC;
    b.ctile = pl.take<int>(NC + 1);
    b.cnode = pl.take<int>(NC + 1);
    b.gchunk = pl.take<int>(G + 1);
    b.cmean = pl.take<float>(NC * kHidden);
    b.cm2 = pl.take<float>(NC * kHidden);
    b.cmax = pl.take<float>(NC * kHidden);
    b.csum = pl.take<double>(NC * kHidden);
    b.carg = pl.take<int>(NC * kHidden);
    b.x0 = pl.take<double>(N * 2);
    b.h1 = pl.take<float>(N * 2);
    for (int l = 0; l < kLayers; ++l) {
        b.h[l] = (l == 0) ? nullptr : pl.take<float>(N * kHidden);
        b.y[l] = pl.take<float>(N * kHidden);
        b.x[l] = pl.take<float>(N * kHidden);
        b.mu[l] = pl.take<float>(G * kHidden);
        b.rstd[l] = pl.take<float>(G * kHidden);
    }
    b.tmean = pl.take<float>(NT * kHidden);
    b.tm2 = pl.take<float>(NT * kHidden);
    b.tsum = pl.take<double>(NT * kHidden);
    b.tsum2 = pl.take<double>(NT * kHidden);
    b.tmax = pl.take<float>(NT * kHidden);
    b.targ = pl.take<int>(NT * kHidden);
    b.pooled = pl.take<float>(G * kLayers * 2 * kHidden);
    b.argmax = pl.take<int>(G * kLayers * kHidden);
    b.head = pl.take<float>(G * kHeadScratch);
    b.c = pl.take<float>(G * 5);
    b.err = pl.take<int>(4);
    if (backward) {
        b.dc = pl.take<float>(G * 5);
        b.dhead = pl.take<float>(G * kHeadGrad);
        b.dpooled = pl.take<float>(G * kLayers * 2 * kHidden);
        b.dx = pl.take<float>(N * kHidden);
        b.dh = pl.take<float>(N * kHidden);
        b.dy = pl.take<float>(N * kHidden);
        b.gS1 = pl.take<double>(G * kHidden);
        b.gS2 = pl.take<double>(G * kHidden);
        b.dWt = pl.take<float>(NT * (kHidden * kHidden + kHidden));
        b.dWc = pl.take<double>(static_cast<size_t>(kGradChunks) * (kHidden * kHidden + kHidden));
    }
}

int gcin_batch_build(GcinBatch &b, int n_problems, amg_ctx *const *problems, cudaStream_t s, std::string &err,
                     bool backward) {
    gcin_batch_free(b);
    std::vector<int> gptr(1, 0), tstart, tgraph, gtile;
    long long E = 0;
    for (int m = 0; m < n_problems; ++m) {
        const amg_ctx *c = problems[m];
        if (!c || c->lev.empty()) {
            err = "problem " + std::to_string(m) + " has no hierarchy";
            return AMG_ERR_STATE;
        }
        for (const auto &L : c->lev) {
            const int g = static_cast<int>(gptr.size()) - 1;
            gtile.push_back(static_cast<int>(tstart.size()));
            for (int a = gptr.back(); a < gptr.back() + L.n; a += kTile) {
                tstart.push_back(a);
                tgraph.push_back(g);
            }
            gptr.push_back(gptr.back() + L.n);
            E += L.A.nnz;
        }
    }
    if (E > 2000000000LL || gptr.back() <= 0 || gptr.back() > 200000000) {
        err = "batch graph too large or empty";
        return AMG_ERR_ARG;
    }
    b.G = static_cast<int>(gptr.size()) - 1;
    b.N = gptr.back();
    b.NT = static_cast<int>(tstart.size());
    b.E = E;
    tstart.push_back(b.N);
    gtile.push_back(b.NT);
    std::vector<int> ctile, cnode, gchunk;
    for (int g = 0; g < b.G; ++g) {
        gchunk.push_back(static_cast<int>(ctile.size()));
        // about sqrt(tiles) tiles per chunk: both reduction stages then loop
        // over about as many parts per lane (at least kChunkTiles per chunk)
        const int nt_g = gtile[g + 1] - gtile[g];
        const int ct = std::max(kChunkTiles, static_cast<int>(std::ceil(std::sqrt(static_cast<double>(nt_g)))));
        for (int t = gtile[g]; t < gtile[g + 1]; t += ct) {
            ctile.push_back(t);
            cnode.push_back(tstart[t]);
        }
    }
    b.NC = static_cast<int>(ctile.size());
    ctile.push_back(b.NT);
    cnode.push_back(b.N);
    gchunk.push_back(b.NC);
    Planner pl;
    batch_layout(b, pl, backward);
    cudaError_t e = cudaMalloc(&b.arena, pl.off);
    if (e != cudaSuccess) {
        err = std::string("cudaMalloc batch: ") + cudaGetErrorString(e);
        b.arena = nullptr;
        return AMG_ERR_CUDA;
    }
    b.bytes = pl.off;
    pl = Planner{};
    pl.base = b.arena;
    batch_layout(b, pl, backward);
    cudaMemcpyAsync(b.gptr, gptr.data(), sizeof(int) * gptr.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.tstart, tstart.data(), sizeof(int) * tstart.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.tgraph, tgraph.data(), sizeof(int) * tgraph.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.gtile, gtile.data(), sizeof(int) * gtile.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.ctile, ctile.data(), sizeof(int) * ctile.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.cnode, cnode.data(), sizeof(int) * cnode.size(), cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(b.gchunk, gchunk.data(), sizeof(int) * gchunk.size(), cudaMemcpyHostToDevice, s);
    int g = 0;
    long long eoff = 0;
    for (int m = 0; m < n_problems; ++m) {
        for (const auto &L : problems[m]->lev) {
            const int work = std::max(L.n, L.A.nnz);
            k_cat_graph<<<grid_for(work), kBlock, 0, s>>>(L.n, L.A.nnz, L.A.rp, L.A.col, L.A.v64, L.diag, gptr[g],
                                                          static_cast<int>(eoff), g, b.rp, b.col, b.w, b.w64, b.x0,
                                                          b.gid); AMG_COUNT();
            eoff += L.A.nnz;
            ++g;
        }
    }
    k_set_int<<<1, 1, 0, s>>>(b.rp + b.N, static_cast<int>(E)); AMG_COUNT();
    cudaMemsetAsync(b.err, 0, sizeof(int) * 4, s);
    e = cudaStreamSynchronize(s);   // host vectors above must outlive the async copies
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        err = std::string("batch build: ") + cudaGetErrorString(e);
        return AMG_ERR_CUDA;
    }
    return AMG_OK;
}

// ---------------------------------------------------------------------------
// forward kernels
// ---------------------------------------------------------------------------
// mean and M2 (sum of squared deviations) per feature of the tile's y rows;
// the block's threads form kBlock / H groups of H (one thread per feature)
template <int H, int YS = H + 1>
__device__ __forceinline__ void tile_stats(const float (*sY)[YS], int nn, float *tmean, float *tm2) {
    constexpr int Q = kBlock / H;
    __shared__ float red[Q][H];
    __shared__ float smean[H];
    const int f = threadIdx.x % H, q = threadIdx.x / H;
    float s = 0.f;
    for (int k = q; k < nn; k += Q) s += sY[k][f];
    red[q][f] = s;
    __syncthreads();
    if (q == 0) {
        float t = red[0][f];
#pragma unroll
        for (int j = 1; j < Q; ++j) t += red[j][f];
        smean[f] = t / nn;
    }
    __syncthreads();
    const float m = smean[f];
    float v = 0.f;
    for (int k = q; k < nn; k += Q) {
        const float d = sY[k][f] - m;
        v = fmaf(d, d, v);
    }
    __syncthreads();
    red[q][f] = v;
    __syncthreads();
    if (q == 0) {
        float t = red[0][f];
#pragma unroll
        for (int j = 1; j < Q; ++j) t += red[j][f];
        tmean[f] = m;
        tm2[f] = t;
    }
}

// bfloat16 copy of four FP32 values (round to nearest even), as 8 bytes
__device__ __forceinline__ uint2 bf16x4(float a, float b, float c, float d) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<unsigned *>(&lo), *reinterpret_cast<unsigned *>(&hi));
}

// Layer 1: h = A_hat x0 (FP64 sums of the raw features, two lanes per node),
// y = h W + b (K = 2: FMA units); tile stats.  YB (BF16 inference): y only
// feeds the tile statistics (FP32); h1 is stored and the normalisation pass
// recomputes y from it (8 bytes per node instead of 128).
// Bound by the FP64 pipe (two DFMAs per entry, 2 lanes a clock and SM): two
// lanes per node waste less of it on short rows than four and exchange their
// sums with one addition each.  A thread owns one feature and keeps its column
// of W, so y needs no shared memory; its two accumulators per statistic are
// the groups of tile_stats.  1.95M nodes: 228 us with four lanes, y staged in
// shared memory and W read per node (L1 pipe 84 %).  Twelve CTAs an SM leave
// 40 registers, at which it spills 16 bytes a thread (28 read back).
constexpr int kL1Threads = 2 * kTile;
template <int H, bool YB = false>
__global__ void __launch_bounds__(kL1Threads, 12) k_layer1_tile(const int *__restrict__ rp, const int *__restrict__ col,
                                                                const double *__restrict__ w64,
                                                                const double *__restrict__ x0,
                                                                const float *__restrict__ W,
                                                                const float *__restrict__ bias,
                                                                const int *__restrict__ tstart, float *__restrict__ h1,
                                                                float *__restrict__ y, float *__restrict__ tmean,
                                                                float *__restrict__ tm2) {
    constexpr int Q = kL1Threads / H;            // threads per feature; 2 Q groups of nodes
    __shared__ float2 sH[kTile];
    __shared__ float red[2 * Q][H];
    const int t = blockIdx.x, a = tstart[t], nn = tstart[t + 1] - a;
    {
        const int k = threadIdx.x >> 1, q = threadIdx.x & 1;
        double a0 = 0.0, a1 = 0.0;
        if (k < nn) {
            const int e = rp[a + k + 1];
            for (int p = rp[a + k] + q; p < e; p += 8) {
                int c[4];
                double w[4];
                double2 x[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    c[j] = p + 2 * j < e ? col[p + 2 * j] : 0;
                    w[j] = p + 2 * j < e ? w64[p + 2 * j] : 0.0;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (p + 2 * j < e) x[j] = reinterpret_cast<const double2 *>(x0)[c[j]];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (p + 2 * j < e) {
                        a0 = fma(w[j], x[j].x, a0);
                        a1 = fma(w[j], x[j].y, a1);
                    }
                }
            }
        }
        // lane 0 ends with the first feature's sum, lane 1 with the second's
        const double other = __shfl_xor_sync(0xffffffffu, q ? a0 : a1, 1);
        const float h = static_cast<float>((q ? a1 : a0) + other);
        if (k < nn) {
            h1[2 * static_cast<size_t>(a) + threadIdx.x] = h;
            reinterpret_cast<float *>(sH)[threadIdx.x] = h;
        }
    }
    const int f = threadIdx.x % H, q = threadIdx.x / H;
    const float w0 = W[f], w1 = W[H + f], bf = bias[f];
    __syncthreads();
    auto yval = [&](int k) {
        const float2 h = sH[k];
        return fmaf(h.x, w0, fmaf(h.y, w1, bf));
    };
    float s0 = 0.f, s1 = 0.f;                    // groups q and q + Q of the tile's nodes
#pragma unroll 4
    for (int k = q; k < nn; k += 2 * Q) {
        const float v0 = yval(k);
        s0 += v0;
        if (!YB) y[static_cast<size_t>(a + k) * H + f] = v0;
        if (k + Q < nn) {
            const float v1 = yval(k + Q);
            s1 += v1;
            if (!YB) y[static_cast<size_t>(a + k + Q) * H + f] = v1;
        }
    }
    auto total = [&](float g0, float g1) {       // the groups' sums in group order
        red[q][f] = g0;
        red[q + Q][f] = g1;
        __syncthreads();
        float r = red[0][f];
#pragma unroll
        for (int j = 1; j < 2 * Q; ++j) r += red[j][f];
        __syncthreads();
        return r;
    };
    const float m = total(s0, s1) / nn;
    float v0 = 0.f, v1 = 0.f;
#pragma unroll 4
    for (int k = q; k < nn; k += 2 * Q) {
        const float d0 = yval(k) - m;
        v0 = fmaf(d0, d0, v0);
        if (k + Q < nn) {
            const float d1 = yval(k + Q) - m;
            v1 = fmaf(d1, d1, v1);
        }
    }
    const float m2 = total(v0, v1);
    if (q == 0) {
        tmean[static_cast<size_t>(t) * H + f] = m;
        tm2[static_cast<size_t>(t) * H + f] = m2;
    }
}

// h_i = sum_p w_p x_{col p} with L = H / 4 lanes per row and 32 / L rows per
// warp (two rows for H = 64, four for H = 32): lane j of a row's group owns
// features 4 j .. 4 j + 3, and entries are added in row order.  Up to L
// (col, w) pairs per row come in with one coalesced load and are broadcast by
// shuffles; each lane keeps four 16-byte gathers in flight, so a warp has
// eight H = 64 (or sixteen H = 32) feature rows in flight.  Called by a whole
// warp (the loop runs to the longest row of the warp, shorter rows predicated
// off).
template <int H, class XR = const float4 *>
__device__ __forceinline__ float4 agg_rows(int p0, int p1, const int *__restrict__ col, const float *__restrict__ w,
                                           const XR &x4, int hl) {
    constexpr int L = H / 4;
    float4 h = make_float4(0.f, 0.f, 0.f, 0.f);
    const int deg = p1 - p0;
    int maxdeg = deg;
#pragma unroll
    for (int o = L; o < 32; o <<= 1) maxdeg = max(maxdeg, __shfl_xor_sync(0xffffffffu, maxdeg, o));
    for (int base = 0; base < maxdeg; base += L) {
        int cj = 0;
        float wj = 0.f;
        if (base + hl < deg) {
            cj = col[p0 + base + hl];
            wj = w[p0 + base + hl];
        }
        const int cnt = deg - base;                  // entries of this row in the chunk (may be <= 0)
        const int cmax = min(L, maxdeg - base);
        int k = 0;
        for (; k + 4 <= cmax; k += 4) {
            int c[4];
            float wk[4];
            float4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                c[j] = __shfl_sync(0xffffffffu, cj, k + j, L);
                wk[j] = __shfl_sync(0xffffffffu, wj, k + j, L);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                v[j] = (k + j < cnt) ? x4[static_cast<size_t>(c[j]) * L + hl] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (k + j < cnt) {
                    h.x = fmaf(wk[j], v[j].x, h.x);
                    h.y = fmaf(wk[j], v[j].y, h.y);
                    h.z = fmaf(wk[j], v[j].z, h.z);
                    h.w = fmaf(wk[j], v[j].w, h.w);
                }
            }
        }
        for (; k < cmax; ++k) {
            const int c = __shfl_sync(0xffffffffu, cj, k, L);
            const float wk = __shfl_sync(0xffffffffu, wj, k, L);
            if (k < cnt) {
                const float4 v = x4[static_cast<size_t>(c) * L + hl];
                h.x = fmaf(wk, v.x, h.x);
                h.y = fmaf(wk, v.y, h.y);
                h.z = fmaf(wk, v.z, h.z);
                h.w = fmaf(wk, v.w, h.w);
            }
        }
    }
    return h;
}

// Layers 2..4: h = A_hat x (H features), y = h W + b; tile stats.
template <int H>
__global__ void __launch_bounds__(kBlock) k_agg_lin_tile(const int *__restrict__ rp, const int *__restrict__ col,
                                                         const float *__restrict__ w, const float *__restrict__ x,
                                                         const float *__restrict__ W, const float *__restrict__ bias,
                                                         const int *__restrict__ tstart, float *__restrict__ hout,
                                                         float *__restrict__ y, float *__restrict__ tmean,
                                                         float *__restrict__ tm2) {
    constexpr int L = H / 4, R = 32 / L;   // lanes per row, rows per warp
    __shared__ float4 sW[H * L];   // W[m][4 j .. 4 j + 3]
    __shared__ float sY[kTile][H + 1];
    for (int t2 = threadIdx.x; t2 < H * L; t2 += kBlock) sW[t2] = reinterpret_cast<const float4 *>(W)[t2];
    __syncthreads();
    const int t = blockIdx.x, a = tstart[t], nn = tstart[t + 1] - a;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, grp = lane / L, hl = lane % L;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    const float4 b4 = reinterpret_cast<const float4 *>(bias)[hl];
    for (int k0 = R * warp; k0 < nn; k0 += R * (kBlock / 32)) {
        const int k = k0 + grp;
        const bool live = k < nn;                    // the last rows of the last group may be absent
        const int i = a + (live ? k : k0);
        const int p0 = rp[i], p1 = live ? rp[i + 1] : p0;
        const float4 hv = agg_rows<H>(p0, p1, col, w, x4, hl);
        if (live && hout) reinterpret_cast<float4 *>(hout)[static_cast<size_t>(i) * L + hl] = hv;
        float4 yv = b4;
#pragma unroll 4
        for (int m = 0; m < H; ++m) {
            const float hsrc = (m & 3) == 0 ? hv.x : (m & 3) == 1 ? hv.y : (m & 3) == 2 ? hv.z : hv.w;
            const float hm = __shfl_sync(0xffffffffu, hsrc, m >> 2, L);
            const float4 wm = sW[m * L + hl];
            yv.x = fmaf(hm, wm.x, yv.x);
            yv.y = fmaf(hm, wm.y, yv.y);
            yv.z = fmaf(hm, wm.z, yv.z);
            yv.w = fmaf(hm, wm.w, yv.w);
        }
        if (live) {
            reinterpret_cast<float4 *>(y)[static_cast<size_t>(i) * L + hl] = yv;
            sY[k][4 * hl] = yv.x;
            sY[k][4 * hl + 1] = yv.y;
            sY[k][4 * hl + 2] = yv.z;
            sY[k][4 * hl + 3] = yv.w;
        }
    }
    __syncthreads();
    tile_stats<H>(sY, nn, tmean + static_cast<size_t>(t) * H, tm2 + static_cast<size_t>(t) * H);
}

// Fixed-order sum over the 16 tile lanes of one feature (16 H-thread blocks:
// f = tid % H, lane = tid / H); every thread receives the total.
constexpr int kLanes = 16;
template <int H>
constexpr int combine_threads() { return kLanes * H; }
template <int H>
__device__ __forceinline__ double lanes_sum(double v, double (*red)[H]) {
    const int f = threadIdx.x % H, q = threadIdx.x / H;
    red[q][f] = v;
    __syncthreads();
    for (int w = kLanes / 2; w > 0; w >>= 1) {
        if (q < w) red[q][f] += red[q + w][f];
        __syncthreads();
    }
    const double t = red[0][f];
    __syncthreads();
    return t;
}

// The same for FP32 pairs; the total in the threads with tid < H.
template <int H>
__device__ __forceinline__ FloatPair lanes_sum_pair(FloatPair v, FloatPair (*red)[H]) {
    const int f = threadIdx.x % H, q = threadIdx.x / H;
    red[q][f] = v;
    __syncthreads();
    for (int w = kLanes / 2; w > 0; w >>= 1) {
        if (q < w) {
            const FloatPair o = red[q + w][f];
            pair_add(v, o.h, o.l);
            red[q][f] = v;
        }
        __syncthreads();
    }
    return v;
}
__device__ __forceinline__ double pair_value(const FloatPair &v) { return static_cast<double>(v.h) + static_cast<double>(v.l); }

// A pair sum that leaves FP32's range (or meets an infinity) ends with a
// non-finite l; it is then taken again in FP64.  Such a total as a pair: h
// scaled by 2^-64 and l = -inf, which no finite sum has.
constexpr double kPairWide = 18446744073709551616.0;   // 2^64
__device__ __forceinline__ FloatPair pair_of(double d) {
    const float h = static_cast<float>(d);
    if (isfinite(h)) return {h, static_cast<float>(d - static_cast<double>(h))};
    return {static_cast<float>(d / kPairWide), -INFINITY};
}
__device__ __forceinline__ double pair_decode(const FloatPair &v) {
    return v.l == -INFINITY ? static_cast<double>(v.h) * kPairWide : pair_value(v);
}

// The statistics' sums of one feature in FP64 (out of line: the threads that
// need it are rare, and inlined it cost the others registers).
__device__ __noinline__ double stats_sum_wide(int a, int e, int f, int H, const int *tstart, const float *tmean) {
    double d = 0.0;
    for (int t = a; t < e; ++t)
        d += static_cast<double>(static_cast<float>(tstart[t + 1] - tstart[t]) * tmean[static_cast<size_t>(t) * H + f]);
    return d;
}
__device__ __noinline__ double stats_m2_wide(int a, int e, int f, int H, const int *tstart, const float *tmean,
                                             const float *tm2, float mean) {
    double v = 0.0;
    for (int t = a; t < e; ++t) {
        const float d = tmean[static_cast<size_t>(t) * H + f] - mean;
        v += static_cast<double>(fmaf(static_cast<float>(tstart[t + 1] - tstart[t]) * d, d, tm2[static_cast<size_t>(t) * H + f]));
    }
    return v;
}

// Group statistics from part statistics (biased variance):
// mean = sum_t n_t mean_t / n, M2 = sum_t [M2_t + n_t (mean_t - mean)^2].
// Parts t of group g are gtile[g] .. gtile[g+1] with node ranges
// tstart[t] .. tstart[t+1].  Run twice: tiles -> chunks (final = 0: writes
// the chunk mean and M2 into mu / rstd) and chunks -> graphs (final = 1:
// writes the instance-norm mean and 1/sqrt(var + eps)).  16 lanes of parts
// per feature, summed as FP32 pairs; FP64 for the totals' divisions and for
// sums past FP32's range (features of matrices with entries of 1e9 and more).
// In FP64 each part cost two instructions of 64 cycles on a sub-partition's
// FP64 unit (7 of a stage's 12 us on a 50k-node mesh); the part loops are
// unrolled so that a thread's loads are in flight together.  With the
// normalisation pass's and the head's reductions: prediction on 50k rows 363
// -> 314 us and, with pairs here and in the pooling, 301 -> 263 us; on 1.2M rows
// 2698 -> 2487 and 2235 -> 2114 us (the checks for sums past FP32's range take
// 12 us of the 1.2M rows, nothing on 50k).
template <int H>
__global__ void __launch_bounds__(kLanes * H) k_stats_combine(const int *__restrict__ gtile, const int *__restrict__ gptr,
                                                            const int *__restrict__ tstart,
                                                            const float *__restrict__ tmean,
                                                            const float *__restrict__ tm2, float *__restrict__ mu,
                                                            float *__restrict__ rstd, int final) {
    __shared__ FloatPair red[kLanes][H];
    __shared__ float smean[H];
    const int g = blockIdx.x, f = threadIdx.x % H, q = threadIdx.x / H;
    const int t0 = gtile[g] + q, t1 = gtile[g + 1];
    FloatPair s{0.f, 0.f};
#pragma unroll 8
    for (int t = t0; t < t1; t += kLanes)
        pair_add(s, static_cast<float>(tstart[t + 1] - tstart[t]) * tmean[static_cast<size_t>(t) * H + f]);
    s = lanes_sum_pair<H>(s, red);
    const int n = gptr[g + 1] - gptr[g];
    if (q == 0)
        smean[f] = static_cast<float>((isfinite(s.l) ? pair_value(s) : stats_sum_wide(t0, t1, f, H, tstart, tmean)) / n);
    __syncthreads();
    const float mf = smean[f];
    FloatPair v{0.f, 0.f};
#pragma unroll 8
    for (int t = t0; t < t1; t += kLanes) {
        const float d = tmean[static_cast<size_t>(t) * H + f] - mf;
        pair_add(v, fmaf(static_cast<float>(tstart[t + 1] - tstart[t]) * d, d, tm2[static_cast<size_t>(t) * H + f]));
    }
    v = lanes_sum_pair<H>(v, red);
    if (q == 0) {
        const double m2 = isfinite(v.l) ? pair_value(v) : stats_m2_wide(t0, t1, f, H, tstart, tmean, tm2, mf);
        mu[static_cast<size_t>(g) * H + f] = mf;
        rstd[static_cast<size_t>(g) * H + f] =
            final ? static_cast<float>(1.0 / sqrt(m2 / n + static_cast<double>(kEps))) : static_cast<float>(m2);
    }
}

// x = ReLU((y - mu) rstd gamma + beta); tile sum / max / argmax of x
// (groups of H / 4 threads, four features per thread, kBlock / (H / 4) rows
// at a time).  x is stored in
// FP32 (x), in bfloat16 (xb: BF16 inference) or not at all (both null: the
// last layer in inference); the pooling always reads the FP32 value.
// YM: 0 FP32 y; 1 bfloat16 y (BF16 inference); 2 layer 1 in BF16 inference:
// y = h1 W1 + b1 recomputed from the stored h1 with the same FMAs as
// k_layer1_tile, rounded to bfloat16 as a stored y would be.
// The 16 row groups' partial sums and maxima go through shared memory as
// 16-byte vectors (four features of a thread; as 8-byte FP64 values at a
// stride of four they kept the L1 pipe at 85 to 94 %), and a feature's 16
// sums are added as an FP32 pair (the 32 FP64 operations per feature and tile
// were 100 us of a 1.95M-node pass).  Six CTAs an SM leave 40 registers: at
// width 64 it spills 92 to 152 bytes a thread (184 to 244 read back).
template <int H, int YM = 0>
__global__ void __launch_bounds__(kBlock, 6) k_norm_relu_pool_tile(const int *__restrict__ tstart,
                                                                const int *__restrict__ tgraph,
                                                                const float *__restrict__ y,
                                                                const float *__restrict__ mu,
                                                                const float *__restrict__ rstd,
                                                                const float *__restrict__ gamma,
                                                                const float *__restrict__ beta, float *__restrict__ x,
                                                                __nv_bfloat16 *__restrict__ xb,
                                                                FloatPair *__restrict__ tsum, float *__restrict__ tmax,
                                                                int *__restrict__ targ,
                                                                const float *__restrict__ h1 = nullptr,
                                                                const float *__restrict__ W1 = nullptr,
                                                                const float *__restrict__ b1 = nullptr) {
    constexpr int F = H / 4, Q = kBlock / F;   // threads per row (4 features each), rows at a time
    __shared__ float4 rs[Q][F], rm[Q][F];
    __shared__ int4 ri[Q][F];
    const int t = blockIdx.x, a = tstart[t], e = tstart[t + 1], g = tgraph[t];
    const int f = 4 * (threadIdx.x % F), q = threadIdx.x / F;
    const float4 m = *reinterpret_cast<const float4 *>(mu + g * H + f);
    const float4 r = *reinterpret_cast<const float4 *>(rstd + g * H + f);
    const float4 ga = *reinterpret_cast<const float4 *>(gamma + f);
    const float4 be = *reinterpret_cast<const float4 *>(beta + f);
    // FP32 partial sums of at most kTile / Q values per thread (GB300's FP64
    // pipe is narrow); tile and graph sums are FP32 pairs
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
    int mi[4] = {a, a, a, a};
    static_assert(kTile % Q == 0, "rows per thread");
    float4 w0, w1, wb;
    if (YM == 2) {
        w0 = *reinterpret_cast<const float4 *>(W1 + f);
        w1 = *reinterpret_cast<const float4 *>(W1 + H + f);
        wb = *reinterpret_cast<const float4 *>(b1 + f);
    }
    // every row's load first (predicated), so a thread's kTile / Q loads are in flight together
    float4 yr[kTile / Q];
#pragma unroll
    for (int r4 = 0; r4 < kTile / Q; ++r4) {
        const int i = a + q + r4 * Q;
        const size_t o = static_cast<size_t>(i < e ? i : a) * H + f;
        if (YM == 1) {   // bfloat16 y (BF16 inference), widened exactly
            const uint2 u = *reinterpret_cast<const uint2 *>(reinterpret_cast<const __nv_bfloat16 *>(y) + o);
            yr[r4] = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u),
                                 __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xFFFF0000u));
        } else if (YM == 2) {
            const float2 hh = reinterpret_cast<const float2 *>(h1)[i < e ? i : a];
            auto yb = [&](float a0, float a1, float c) {
                return __bfloat162float(__float2bfloat16_rn(fmaf(hh.x, a0, fmaf(hh.y, a1, c))));
            };
            yr[r4] = make_float4(yb(w0.x, w1.x, wb.x), yb(w0.y, w1.y, wb.y), yb(w0.z, w1.z, wb.z), yb(w0.w, w1.w, wb.w));
        } else {
            yr[r4] = *reinterpret_cast<const float4 *>(y + o);
        }
    }
#pragma unroll
    for (int r4 = 0; r4 < kTile / Q; ++r4) {
        const int i = a + q + r4 * Q;
        if (i >= e) break;
        const size_t o = static_cast<size_t>(i) * H + f;
        const float4 yv = yr[r4];
        float v[4];
        v[0] = fmaxf((yv.x - m.x) * r.x * ga.x + be.x, 0.f);
        v[1] = fmaxf((yv.y - m.y) * r.y * ga.y + be.y, 0.f);
        v[2] = fmaxf((yv.z - m.z) * r.z * ga.z + be.z, 0.f);
        v[3] = fmaxf((yv.w - m.w) * r.w * ga.w + be.w, 0.f);
        if (xb) {   // inference: the next aggregation's BF16 input
            *reinterpret_cast<uint2 *>(xb + o) = bf16x4(v[0], v[1], v[2], v[3]);
        } else if (x) {
            *reinterpret_cast<float4 *>(x + o) = make_float4(v[0], v[1], v[2], v[3]);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            s[j] += v[j];
            if (v[j] > mx[j]) { mx[j] = v[j]; mi[j] = i; }
        }
    }
    rs[q][f / 4] = make_float4(s[0], s[1], s[2], s[3]);
    rm[q][f / 4] = make_float4(mx[0], mx[1], mx[2], mx[3]);
    if (targ) ri[q][f / 4] = make_int4(mi[0], mi[1], mi[2], mi[3]);
    __syncthreads();
    if (threadIdx.x < H) {
        const int ff = threadIdx.x;
        const float *ps = reinterpret_cast<const float *>(rs) + ff, *pm = reinterpret_cast<const float *>(rm) + ff;
        const int *pi = reinterpret_cast<const int *>(ri) + ff;
        FloatPair ts{0.f, 0.f};
        float bm = -INFINITY;
#pragma unroll 4
        for (int k = 0; k < Q; ++k) {
            pair_add(ts, ps[k * H]);
            bm = fmaxf(bm, pm[k * H]);
        }
        if (!isfinite(ts.l)) {                   // past FP32's range
            double d = 0.0;
#pragma unroll 1
            for (int k = 0; k < Q; ++k) d += static_cast<double>(ps[k * H]);
            ts = pair_of(d);
        }
        tsum[static_cast<size_t>(t) * H + ff] = ts;
        tmax[static_cast<size_t>(t) * H + ff] = bm;
        if (targ) {                              // the first node of the maximum
            int bi = a;
            bool found = false;
#pragma unroll 4
            for (int k = 0; k < Q; ++k) {
                if (pm[k * H] == bm && (!found || pi[k * H] < bi)) {
                    bi = pi[k * H];
                    found = true;
                }
            }
            targ[static_cast<size_t>(t) * H + ff] = bi;
        }
    }
}

// A pooled sum of one feature in FP64.
__device__ __noinline__ FloatPair pool_sum_wide(int a, int e, int f, int H, const FloatPair *tsum) {
    double d = 0.0;
    for (int t = a; t < e; ++t) d += pair_decode(tsum[static_cast<size_t>(t) * H + f]);
    return pair_of(d);
}

// Group sum and max (first index of the max kept) from part partials; as
// for the statistics, tiles -> chunks (csum != nullptr: writes the chunk sum,
// max and argmax) and chunks -> graphs (writes the pooled mean and max).
template <int H>
__global__ void __launch_bounds__(kLanes * H) k_pool_combine(const int *__restrict__ gtile, const int *__restrict__ gptr,
                                                           const FloatPair *__restrict__ tsum,
                                                           const float *__restrict__ tmax,
                                                           const int *__restrict__ targ, float *__restrict__ pooled,
                                                           int *__restrict__ argmax, int layer,
                                                           FloatPair *__restrict__ csum, float *__restrict__ cmax,
                                                           int *__restrict__ carg) {
    __shared__ FloatPair red[kLanes][H];
    __shared__ float rm[kLanes][H];
    __shared__ int ri[kLanes][H];
    const int g = blockIdx.x, f = threadIdx.x % H, q = threadIdx.x / H;
    FloatPair s{0.f, 0.f};
    float bm = -INFINITY;
    int bi = gptr[g];
    const int t0 = gtile[g] + q, t1 = gtile[g + 1];
    if (targ) {
#pragma unroll 8
        for (int t = t0; t < t1; t += kLanes) {
            const size_t o = static_cast<size_t>(t) * H + f;
            const float m = tmax[o];
            const int a = targ[o];
            const FloatPair p = tsum[o];
            pair_add(s, p.h, p.l);
            if (m > bm) { bm = m; bi = a; }   // tiles ascend, so the first max wins
        }
    } else {                                  // inference: no backward asks for the node
#pragma unroll 8
        for (int t = t0; t < t1; t += kLanes) {
            const size_t o = static_cast<size_t>(t) * H + f;
            const FloatPair p = tsum[o];
            pair_add(s, p.h, p.l);
            bm = fmaxf(bm, tmax[o]);
        }
    }
    rm[q][f] = bm;
    ri[q][f] = bi;
    FloatPair total = lanes_sum_pair<H>(s, red);
    if (q == 0) {
        for (int k = 1; k < kLanes; ++k)
            if (rm[k][f] > bm || (rm[k][f] == bm && ri[k][f] < bi)) { bm = rm[k][f]; bi = ri[k][f]; }
        if (!isfinite(total.l)) total = pool_sum_wide(t0, t1, f, H, tsum);   // past FP32's range
        if (csum) {
            const size_t o = static_cast<size_t>(g) * H + f;
            csum[o] = total;
            cmax[o] = bm;
            if (carg) carg[o] = bi;
            return;
        }
        float *P = pooled + (static_cast<size_t>(g) * kLayers + layer) * 2 * H;
        P[f] = static_cast<float>(pair_decode(total) / (gptr[g + 1] - gptr[g]));
        P[H + f] = bm;
        if (targ) argmax[(static_cast<size_t>(g) * kLayers + layer) * H + f] = bi;
    }
}

// Sum over the block's first 128 threads (called by exactly those).
__device__ __forceinline__ float block128_sum(float v, float *red) {
    v = warp_sum(v);
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = v;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    float t = red[0] + red[1] + red[2] + red[3];
    asm volatile("bar.sync 1, 128;" ::: "memory");
    return t;
}

// Head scratch layout per graph: z[128] | zh[128] | sig[128] | a1[128] | a2[64] | mean | rstd
constexpr int kSz = 0, kSzh = kEmb, kSsg = 2 * kEmb, kSa1 = 3 * kEmb, kSa2 = 3 * kEmb + 128,
              kSmean = 3 * kEmb + 192, kSrs = 3 * kEmb + 193;
// Head gradient layout per graph: dz1[128] | dz2[64] | dzh[128] | dz[128]
constexpr int kGdz1 = 0, kGdz2 = 128, kGdzh = 192, kGdz = 192 + kEmb;

// Bias plus a dot product of n terms over a column of W (row stride ld).
// Inference takes four lanes per output, each with an unrolled quarter: the
// three dependent layers are then a few load round trips each (128 serial
// terms per lane took 33 us on seven graphs).  Training, whose loss passes the
// coefficients' last bits on through the V-cycles, adds the terms in one chain.
template <int LANES>
__device__ __forceinline__ float head_dot(float bias, const float *v, const float *__restrict__ W, int n, int ld, int q) {
    if (LANES == 1) {
#pragma unroll 32
        for (int m = 0; m < n; ++m) bias = fmaf(v[m], W[m * ld], bias);
        return bias;
    }
    float a = 0.f;
#pragma unroll 32
    for (int m = q; m < n; m += LANES) a = fmaf(v[m], W[m * ld], a);
#pragma unroll
    for (int o = 1; o < LANES; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return bias + a;
}

// Readout + head for one graph (four threads per element of the 128-vectors).
template <int H, int LANES>
__global__ void __launch_bounds__(LANES * kEmb) k_head(const float *__restrict__ pooled, const float *__restrict__ th,
                                                       float *__restrict__ scratch, float *__restrict__ c) {
    __shared__ float sp[kLayers * 2 * H];
    __shared__ float sz[kEmb], ss[kEmb], sa1[128], sa2[64];
    __shared__ float red[4];
    constexpr int kHeadThreads = LANES * kEmb;
    const int g = blockIdx.x, t = threadIdx.x / LANES, q = threadIdx.x % LANES;
    for (int k = threadIdx.x; k < kLayers * 2 * H; k += kHeadThreads)
        sp[k] = pooled[static_cast<size_t>(g) * kLayers * 2 * H + k];
    __syncthreads();
    float *S = scratch + static_cast<size_t>(g) * kHeadScratch;
    // readout linears: z[32 l + k] = [mean_l, max_l] . W_l[:, k] + b_l[k]
    {
        const int l = t / kRo, k = t % kRo;
        const float z = head_dot<LANES>(th[PL<H>().roB[l] + k], sp + l * 2 * H, th + PL<H>().roW[l] + k, 2 * H, kRo, q);
        if (q == 0) sz[t] = z;
    }
    __syncthreads();
    // layer norm over the 128-vector (the first 128 threads)
    if (threadIdx.x < kEmb) {
        const int i = threadIdx.x;
        const float z = sz[i];
        const float mean = block128_sum(z, red) / kEmb;
        const float d = z - mean;
        const float var = block128_sum(d * d, red) / kEmb;
        const float rs = rsqrtf(var + kEps);
        const float zh = d * rs * th[PL<H>().lnG + i] + th[PL<H>().lnB + i];
        const float sg = 1.f / (1.f + expf(-zh));
        S[kSz + i] = z;
        S[kSzh + i] = zh;
        S[kSsg + i] = sg;
        if (i == 0) {
            S[kSmean] = mean;
            S[kSrs] = rs;
        }
        ss[i] = sg;
    }
    __syncthreads();
    const float a1 = fmaxf(head_dot<LANES>(th[PL<H>().h1B + t], ss, th + PL<H>().h1W + t, kEmb, 128, q), 0.f);
    if (q == 0) {
        sa1[t] = a1;
        S[kSa1 + t] = a1;
    }
    __syncthreads();
    if (t < 64) {
        const float a2 = fmaxf(head_dot<LANES>(th[PL<H>().h2B + t], sa1, th + PL<H>().h2W + t, 128, 64, q), 0.f);
        if (q == 0) {
            sa2[t] = a2;
            S[kSa2 + t] = a2;
        }
    }
    __syncthreads();
    if (threadIdx.x < 32) {                       // one whole warp; five outputs
        const int o = min(t, 4);
        const float v = head_dot<LANES>(th[PL<H>().h3B + o], sa2, th + PL<H>().h3W + o, 64, 5, q);
        if (q == 0 && t < 5) c[g * 5 + t] = v;
    }
}

}  // namespace amg
#include "gcin_tc.cuh"
namespace amg {

void gcin_prepare_device() {
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return;
    cudaFuncSetAttribute(k_agg_lin_tc<kHidden>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem<kHidden>());
    cudaFuncSetAttribute(k_agg_lin_tc<kHidden32>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem<kHidden32>());
    cudaFuncSetAttribute(k_agg_lin_tc<kHidden, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem<kHidden>());
    cudaFuncSetAttribute(k_agg_lin_tc<kHidden32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         tc_smem<kHidden32>());
    cudaFuncSetAttribute(k_bwd_lin_tc<kHidden>, cudaFuncAttributeMaxDynamicSharedMemorySize, tcb_smem<kHidden>());
    cudaFuncSetAttribute(k_bwd_lin_tc<kHidden32>, cudaFuncAttributeMaxDynamicSharedMemorySize, tcb_smem<kHidden32>());
    done[dev] = true;
}

template <int H>
static void forward_impl(GcinBatch &b, const float *th, cudaStream_t s) {
    const ParamLayout &pl = host_layout(H);
    const int N = b.N, G = b.G, NT = b.NT;
    constexpr int CT = combine_threads<H>();
    const bool xb16 = b.bf16 && b.infer;   // BF16 inference on the tensor cores
    const bool xbf = xb16 && kInferBF16Acts;   // ... with y and x stored in bfloat16
    for (int l = 0; l < kLayers; ++l) {
        if (l == 0 && xbf) {
            k_layer1_tile<H, true><<<NT, kL1Threads, 0, s>>>(b.rp, b.col, b.w64, b.x0, th + pl.convW[0],
                                                         th + pl.convB[0], b.tstart, b.h1, b.y[0], b.tmean,
                                                         b.tm2); AMG_COUNT();
        } else if (l == 0) {
            k_layer1_tile<H><<<NT, kL1Threads, 0, s>>>(b.rp, b.col, b.w64, b.x0, th + pl.convW[0], th + pl.convB[0],
                                                   b.tstart, b.h1, b.y[0], b.tmean, b.tm2); AMG_COUNT();
        } else if (xb16) {
            k_agg_lin_tc<H, true><<<(NT + 1) / 2, kBlock, tc_smem<H>(), s>>>(
                b.rp, b.col, b.w, b.x[l - 1], nullptr, b.wtile + static_cast<size_t>(l - 1) * tc_b_bytes<H>(),
                th + pl.convB[l], b.tstart, NT, nullptr, b.y[l], b.tmean, b.tm2, b.err, 0); AMG_COUNT();
        } else if (b.bf16) {
            k_agg_lin_tc<H><<<(NT + 1) / 2, kBlock, tc_smem<H>(), s>>>(b.rp, b.col, b.w, b.x[l - 1],
                                                                     th + pl.convW[l], nullptr, th + pl.convB[l],
                                                                     b.tstart, NT, b.infer ? nullptr : b.h[l], b.y[l],
                                                                     b.tmean, b.tm2, b.err, 0); AMG_COUNT();
        } else {
            k_agg_lin_tile<H><<<NT, kBlock, 0, s>>>(b.rp, b.col, b.w, b.x[l - 1], th + pl.convW[l],
                                                    th + pl.convB[l], b.tstart, b.infer ? nullptr : b.h[l], b.y[l],
                                                    b.tmean, b.tm2); AMG_COUNT();
        }
        k_stats_combine<H><<<b.NC, CT, 0, s>>>(b.ctile, b.cnode, b.tstart, b.tmean, b.tm2, b.cmean, b.cm2, 0); AMG_COUNT();
        k_stats_combine<H><<<G, CT, 0, s>>>(b.gchunk, b.gptr, b.cnode, b.cmean, b.cm2, b.mu[l], b.rstd[l], 1); AMG_COUNT();
        // inference keeps only what the next aggregation reads (bfloat16 with
        // the tensor-core linears, nothing after the last layer)
        const bool last = l == kLayers - 1;
        FloatPair *tsum = reinterpret_cast<FloatPair *>(b.tsum), *csum = reinterpret_cast<FloatPair *>(b.csum);
        int *targ = b.infer ? nullptr : b.targ, *carg = b.infer ? nullptr : b.carg;
        float *xo = (b.infer && (xbf || last)) ? nullptr : b.x[l];
        __nv_bfloat16 *xbo = (xbf && !last) ? reinterpret_cast<__nv_bfloat16 *>(b.x[l]) : nullptr;
        if (xbf && l == 0) {
            k_norm_relu_pool_tile<H, 2><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.y[l], b.mu[l], b.rstd[l],
                                                              th + pl.inG[l], th + pl.inB[l], xo, xbo, tsum,
                                                              b.tmax, targ, b.h1, th + pl.convW[0],
                                                              th + pl.convB[0]); AMG_COUNT();
        } else if (xbf) {
            k_norm_relu_pool_tile<H, 1><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.y[l], b.mu[l], b.rstd[l],
                                                              th + pl.inG[l], th + pl.inB[l], xo, xbo, tsum,
                                                              b.tmax, targ); AMG_COUNT();
        } else {
            k_norm_relu_pool_tile<H><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.y[l], b.mu[l], b.rstd[l],
                                                           th + pl.inG[l], th + pl.inB[l], xo, xbo, tsum, b.tmax,
                                                           targ); AMG_COUNT();
        }
        k_pool_combine<H><<<b.NC, CT, 0, s>>>(b.ctile, b.cnode, tsum, b.tmax, targ, nullptr, nullptr, l,
                                              csum, b.cmax, carg); AMG_COUNT();
        k_pool_combine<H><<<G, CT, 0, s>>>(b.gchunk, b.gptr, csum, b.cmax, carg, b.pooled, b.argmax, l,
                                           nullptr, nullptr, nullptr); AMG_COUNT();
    }
    if (b.infer) k_head<H, 4><<<G, 4 * kEmb, 0, s>>>(b.pooled, th, b.head, b.c);
    else k_head<H, 1><<<G, kEmb, 0, s>>>(b.pooled, th, b.head, b.c); AMG_COUNT();
}

// The layer 2..4 B tiles of BF16 inference, laid out when the parameters are
// loaded (gnn_load_params) instead of in every prediction.
static void pack_wtiles(int H, const float *th, unsigned char *out, cudaStream_t s) {
    const ParamLayout &pl = host_layout(H);
    if (H == kHidden32)
        k_pack_wtile<kHidden32><<<kLayers - 1, kBlock, 0, s>>>(th + pl.convW[1], th + pl.convW[2], th + pl.convW[3], out);
    else
        k_pack_wtile<kHidden><<<kLayers - 1, kBlock, 0, s>>>(th + pl.convW[1], th + pl.convW[2], th + pl.convW[3], out);
    AMG_COUNT();
}

void gcin_forward(GcinBatch &b, const float *th, cudaStream_t s) {
    gcin_prepare_device();
    // the tensor-core kernel's wait-timeout flag belongs to this forward pass
    // only: clear it first (a captured inference graph replays this too), so
    // one timed-out pass does not fail every later one
    cudaMemsetAsync(b.err, 0, sizeof(int) * 4, s);
    if (b.hidden == kHidden32) forward_impl<kHidden32>(b, th, s);
    else forward_impl<kHidden>(b, th, s);
}

// ---------------------------------------------------------------------------
// backward kernels
// ---------------------------------------------------------------------------
// Head backward for one graph: dc -> dz2, dz1, dzh, dz (readout outputs) and
// the pooled-feature gradient dpooled.
template <int H>
__global__ void __launch_bounds__(128) k_head_bwd(const float *__restrict__ scratch, const float *__restrict__ th,
                                                  const float *__restrict__ dc, float *__restrict__ dhead,
                                                  float *__restrict__ dpooled) {
    __shared__ float sdc[5], sdz2[64], sdz1[128], sdz[kEmb];
    __shared__ float red[4];
    const int g = blockIdx.x, t = threadIdx.x;
    const float *S = scratch + static_cast<size_t>(g) * kHeadScratch;
    float *D = dhead + static_cast<size_t>(g) * kHeadGrad;
    if (t < 5) sdc[t] = dc[g * 5 + t];
    __syncthreads();
    if (t < 64) {
        float da2 = 0.f;
        for (int k = 0; k < 5; ++k) da2 = fmaf(sdc[k], th[PL<H>().h3W + t * 5 + k], da2);
        const float dz2 = S[kSa2 + t] > 0.f ? da2 : 0.f;
        sdz2[t] = dz2;
        D[kGdz2 + t] = dz2;
    }
    __syncthreads();
    float da1 = 0.f;
#pragma unroll 32   // the lane's loads of its weight row in flight together
    for (int k = 0; k < 64; ++k) da1 = fmaf(sdz2[k], th[PL<H>().h2W + t * 64 + k], da1);
    const float dz1 = S[kSa1 + t] > 0.f ? da1 : 0.f;
    sdz1[t] = dz1;
    D[kGdz1 + t] = dz1;
    __syncthreads();
    float ds = 0.f;
#pragma unroll 32
    for (int k = 0; k < 128; ++k) ds = fmaf(sdz1[k], th[PL<H>().h1W + t * 128 + k], ds);
    const float sg = S[kSsg + t];
    const float dzh = ds * sg * (1.f - sg);
    D[kGdzh + t] = dzh;
    // layer norm backward
    const float rs = S[kSrs], mean = S[kSmean];
    const float zn = (S[kSz + t] - mean) * rs;
    const float dzn = dzh * th[PL<H>().lnG + t];
    const float m1 = block128_sum(dzn, red) / kEmb;
    const float m2 = block128_sum(dzn * zn, red) / kEmb;
    const float dz = rs * (dzn - m1 - zn * m2);
    sdz[t] = dz;
    D[kGdz + t] = dz;
    __syncthreads();
    // readout linears: dpooled_l[m] = sum_k dz[32 l + k] W_l[m][k]
    for (int j = t; j < kLayers * 2 * H; j += 128) {
        const int l = j / (2 * H), m = j % (2 * H);
        const float *W = th + PL<H>().roW[l] + m * kRo;
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < kRo; ++k) acc = fmaf(sdz[l * kRo + k], W[k], acc);
        dpooled[static_cast<size_t>(g) * kLayers * 2 * H + j] = acc;
    }
}

// Gradients of the readout / layer-norm / head parameters: one thread per
// parameter, sum over graphs in graph order.
template <int H>
__global__ void k_head_param_grad(int G, const float *__restrict__ pooled, const float *__restrict__ scratch,
                                  const float *__restrict__ dhead, const float *__restrict__ dc,
                                  float *__restrict__ grad) {
    const int p = PL<H>().roW[0] + blockIdx.x * kBlock + threadIdx.x;
    if (p >= num_params<H>()) return;
    double acc = 0.0;
    int l = -1;
    for (int k = 0; k < kLayers; ++k)
        if (p >= PL<H>().roW[k] && p < PL<H>().roB[k] + kRo) l = k;
    for (int g = 0; g < G; ++g) {
        const float *S = scratch + static_cast<size_t>(g) * kHeadScratch;
        const float *D = dhead + static_cast<size_t>(g) * kHeadGrad;
        double v;
        if (l >= 0) {
            if (p < PL<H>().roB[l]) {
                const int o = p - PL<H>().roW[l], m = o / kRo, k = o % kRo;
                v = static_cast<double>(pooled[(static_cast<size_t>(g) * kLayers + l) * 2 * H + m]) *
                    D[kGdz + l * kRo + k];
            } else {
                v = D[kGdz + l * kRo + (p - PL<H>().roB[l])];
            }
        } else if (p < PL<H>().lnB) {
            const int k = p - PL<H>().lnG;
            v = static_cast<double>(D[kGdzh + k]) * ((S[kSz + k] - S[kSmean]) * S[kSrs]);
        } else if (p < PL<H>().h1W) {
            v = D[kGdzh + (p - PL<H>().lnB)];
        } else if (p < PL<H>().h1B) {
            const int o = p - PL<H>().h1W, m = o / 128, k = o % 128;
            v = static_cast<double>(S[kSsg + m]) * D[kGdz1 + k];
        } else if (p < PL<H>().h2W) {
            v = D[kGdz1 + (p - PL<H>().h1B)];
        } else if (p < PL<H>().h2B) {
            const int o = p - PL<H>().h2W, m = o / 64, k = o % 64;
            v = static_cast<double>(S[kSa1 + m]) * D[kGdz2 + k];
        } else if (p < PL<H>().h3W) {
            v = D[kGdz2 + (p - PL<H>().h2B)];
        } else if (p < PL<H>().h3B) {
            const int o = p - PL<H>().h3W, m = o / 5, k = o % 5;
            v = static_cast<double>(S[kSa2 + m]) * dc[g * 5 + k];
        } else {
            v = dc[g * 5 + (p - PL<H>().h3B)];
        }
        acc += v;
    }
    grad[p] = static_cast<float>(acc);
}

// Layer backward, part 1 (per tile): dX = dx_next + pooling routes; the
// ReLU mask gives d(yn); tile sums S1 = sum d(yn), S2 = sum d(yn) * yhat.
template <int H>
__global__ void __launch_bounds__(kBlock) k_bwd_relu_tile(const int *__restrict__ tstart,
                                                          const int *__restrict__ tgraph, const int *__restrict__ gptr,
                                                          const float *__restrict__ x, const float *__restrict__ y,
                                                          const float *__restrict__ mu, const float *__restrict__ rstd,
                                                          const float *__restrict__ dx, const float *__restrict__ dpooled,
                                                          const int *__restrict__ argmax, int layer,
                                                          float *__restrict__ dyn, double *__restrict__ tsum,
                                                          double *__restrict__ tsum2) {
    constexpr int Q = kBlock / H;
    __shared__ double r1[Q][H], r2[Q][H];
    const int t = blockIdx.x, a = tstart[t], e = tstart[t + 1], g = tgraph[t];
    const int f = threadIdx.x % H, q = threadIdx.x / H;
    const float *dp = dpooled + (static_cast<size_t>(g) * kLayers + layer) * 2 * H;
    const float dmean = dp[f] / (gptr[g + 1] - gptr[g]), dmax = dp[H + f];
    const int am = argmax[(static_cast<size_t>(g) * kLayers + layer) * H + f];
    const float m = mu[g * H + f], r = rstd[g * H + f];
    float s1 = 0.f, s2 = 0.f;                 // FP32 per thread, FP64 from the tile sum on
    for (int i = a + q; i < e; i += Q) {
        const size_t o = static_cast<size_t>(i) * H + f;
        float dX = dmean + (i == am ? dmax : 0.f);
        if (dx) dX += dx[o];
        const float d = x[o] > 0.f ? dX : 0.f;
        dyn[o] = d;
        s1 += d;
        s2 = fmaf(d, (y[o] - m) * r, s2);
    }
    r1[q][f] = static_cast<double>(s1);
    r2[q][f] = static_cast<double>(s2);
    __syncthreads();
    if (q == 0) {
        double t1 = r1[0][f], t2 = r2[0][f];
        for (int k = 1; k < Q; ++k) {
            t1 += r1[k][f];
            t2 += r2[k][f];
        }
        tsum[static_cast<size_t>(t) * H + f] = t1;
        tsum2[static_cast<size_t>(t) * H + f] = t2;
    }
}

template <int H>
__global__ void __launch_bounds__(kLanes * H) k_bwd_combine(const int *__restrict__ gtile,
                                                            const double *__restrict__ tsum,
                                                            const double *__restrict__ tsum2,
                                                            double *__restrict__ gS1, double *__restrict__ gS2) {
    __shared__ double red[kLanes][H];
    const int g = blockIdx.x, f = threadIdx.x % H, q = threadIdx.x / H;
    double s1 = 0.0, s2 = 0.0;
    const int t1e = gtile[g + 1];
#pragma unroll 4
    for (int t = gtile[g] + q; t < t1e; t += kLanes) {
        s1 += tsum[static_cast<size_t>(t) * H + f];
        s2 += tsum2[static_cast<size_t>(t) * H + f];
    }
    const double t1 = lanes_sum<H>(s1, red);
    const double t2 = lanes_sum<H>(s2, red);
    if (q == 0) {
        gS1[g * H + f] = t1;
        gS2[g * H + f] = t2;
    }
}

// FPL = H / 32 consecutive floats of row i owned by lane `lane` (float2 for H = 64)
template <int FPL>
__device__ __forceinline__ void lane_load(const float *__restrict__ p, size_t i, int lane, float (&v)[FPL]) {
    if constexpr (FPL == 2) {
        const float2 t = reinterpret_cast<const float2 *>(p)[i * 32 + lane];
        v[0] = t.x;
        v[1] = t.y;
    } else {
        v[0] = p[i * 32 + lane];
    }
}

// Instance-norm backward of a lane's features of one node:
// dy = rstd (gamma d(yn) - gamma S1/n - yhat gamma S2/n).
template <int FPL> struct NormBwd {
    float ga[FPL], m[FPL], r[FPL], c1[FPL], c2[FPL];
    __device__ __forceinline__ NormBwd(int g, int H, int lane, float inv_n, const float *__restrict__ mu,
                                       const float *__restrict__ rstd, const float *__restrict__ gamma,
                                       const double *__restrict__ gS1, const double *__restrict__ gS2) {
#pragma unroll
        for (int j = 0; j < FPL; ++j) {
            const int f = FPL * lane + j;
            ga[j] = gamma[f];
            m[j] = mu[g * H + f];
            r[j] = rstd[g * H + f];
            c1[j] = ga[j] * static_cast<float>(gS1[g * H + f]) * inv_n;
            c2[j] = ga[j] * static_cast<float>(gS2[g * H + f]) * inv_n;
        }
    }
    __device__ __forceinline__ float dy(int j, float d, float y) const {
        const float yh = (y - m[j]) * r[j];
        return r[j] * (ga[j] * d - c1[j] - yh * c2[j]);
    }
};

// Layer backward, part 2, layers 2..4 in FP32 (per tile): the instance norm's
// backward, then dh = dy W^T and the tile's partial weight and bias gradients
// sum_i h_i^T dy_i, sum_i dy_i.  Both products are bound by shared memory, so
// each thread holds a block of outputs in registers (H = 64: 4 x 4 of either)
// and reads 16 bytes at a time: 8 loads for 64 FMAs where a load and a
// shuffle fed two.  dy and W^T come first; the tile's h waits in registers and
// takes W^T's place for the second product.  Sums run in the order of k and of
// the nodes.  Five 8k-row meshes (61k nodes): a training batch 5003 -> 4759 us
// (the old form took 127 us a layer).
template <int H>
__global__ void __launch_bounds__(kBlock) k_bwd_lin_tile(const int *__restrict__ tstart, const int *__restrict__ tgraph,
                                                         const int *__restrict__ gptr, const float *__restrict__ y,
                                                         const float *__restrict__ mu, const float *__restrict__ rstd,
                                                         const float *__restrict__ gamma, const double *__restrict__ gS1,
                                                         const double *__restrict__ gS2, const float *__restrict__ W,
                                                         const float *__restrict__ hin, const float *__restrict__ dyn,
                                                         float *__restrict__ dh, float *__restrict__ dWt, int round_w) {
    constexpr int FPL = H / 32, LD = H + 4, TX = H / 4, TY = kBlock / TX;
    constexpr int R = kTile / TY, RW = H / TY;            // output rows per thread: dh, weight gradient
    constexpr int HV = kTile * H / 4 / kBlock;            // 16-byte pieces of h per thread
    static_assert(R * TY == kTile && RW * TY == H && HV * kBlock * 4 == kTile * H, "whole blocks");
    __shared__ __align__(16) float sD[kTile * LD];
    __shared__ __align__(16) float sB[(H > kTile ? H : kTile) * LD];   // W^T, then h
    const int t = blockIdx.x, a = tstart[t], nn = tstart[t + 1] - a, g = tgraph[t];
    const float inv_n = 1.f / (gptr[g + 1] - gptr[g]);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    float4 hv[HV];
#pragma unroll
    for (int q = 0; q < HV; ++q) {
        const int e = q * kBlock + threadIdx.x;
        hv[q] = e / TX < nn ? reinterpret_cast<const float4 *>(hin)[static_cast<size_t>(a) * TX + e]
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int e = threadIdx.x; e < H * H; e += kBlock) {
        float wv = W[e];
        if (round_w) wv = __bfloat162float(__float2bfloat16_rn(wv));   // the forward multiplied by the BF16-rounded weights
        sB[(e % H) * LD + e / H] = wv;
    }
    const NormBwd<FPL> nb(g, H, lane, inv_n, mu, rstd, gamma, gS1, gS2);
#pragma unroll 4
    for (int k = warp; k < nn; k += kBlock / 32) {
        float d[FPL], yv[FPL];
        lane_load<FPL>(dyn, a + k, lane, d);
        lane_load<FPL>(y, a + k, lane, yv);
#pragma unroll
        for (int j = 0; j < FPL; ++j) sD[k * LD + FPL * lane + j] = nb.dy(j, d[j], yv[j]);
    }
    __syncthreads();
    const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
    auto at4 = [](const float *p) { return *reinterpret_cast<const float4 *>(p); };
    if (R * ty < nn) {                                    // rows past the tile's nodes are computed, not stored
        float acc[R][4] = {};
#pragma unroll 4
        for (int k = 0; k < H; k += 4) {
            float av[R][4];
#pragma unroll
            for (int i = 0; i < R; ++i) *reinterpret_cast<float4 *>(av[i]) = at4(sD + (R * ty + i) * LD + k);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w4 = at4(sB + (k + q) * LD + 4 * tx);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    acc[i][0] = fmaf(av[i][q], w4.x, acc[i][0]);
                    acc[i][1] = fmaf(av[i][q], w4.y, acc[i][1]);
                    acc[i][2] = fmaf(av[i][q], w4.z, acc[i][2]);
                    acc[i][3] = fmaf(av[i][q], w4.w, acc[i][3]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (R * ty + i < nn)
                reinterpret_cast<float4 *>(dh)[static_cast<size_t>(a + R * ty + i) * TX + tx] =
                    make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < HV; ++q) {
        const int e = q * kBlock + threadIdx.x;
        *reinterpret_cast<float4 *>(sB + (e / TX) * LD + 4 * (e % TX)) = hv[q];
    }
    __syncthreads();
    float *out = dWt + static_cast<size_t>(t) * (H * H + H);
    float acc[RW][4] = {}, bias[4] = {};
#pragma unroll 4
    for (int j = 0; j < nn; ++j) {
        const float4 d4 = at4(sD + j * LD + 4 * tx);
        float hj[RW];
        if constexpr (RW == 4) *reinterpret_cast<float4 *>(hj) = at4(sB + j * LD + 4 * ty);
        else
            for (int i = 0; i < RW; ++i) hj[i] = sB[j * LD + RW * ty + i];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
            acc[i][0] = fmaf(hj[i], d4.x, acc[i][0]);
            acc[i][1] = fmaf(hj[i], d4.y, acc[i][1]);
            acc[i][2] = fmaf(hj[i], d4.z, acc[i][2]);
            acc[i][3] = fmaf(hj[i], d4.w, acc[i][3]);
        }
        if (ty == 0) {
            bias[0] += d4.x;
            bias[1] += d4.y;
            bias[2] += d4.z;
            bias[3] += d4.w;
        }
    }
#pragma unroll
    for (int i = 0; i < RW; ++i)
        *reinterpret_cast<float4 *>(out + (RW * ty + i) * H + 4 * tx) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
    if (ty == 0) *reinterpret_cast<float4 *>(out + H * H + 4 * tx) = make_float4(bias[0], bias[1], bias[2], bias[3]);
}

// The same for layer 1 (two input features, no dh): a warp takes one node,
// lane j owns features FPL j .. FPL j + FPL - 1 (FPL = H / 32).
template <int H>
__global__ void __launch_bounds__(kBlock) k_bwd_lin1_tile(const int *__restrict__ tstart, const int *__restrict__ tgraph,
                                                          const int *__restrict__ gptr, const float *__restrict__ y,
                                                          const float *__restrict__ mu, const float *__restrict__ rstd,
                                                          const float *__restrict__ gamma, const double *__restrict__ gS1,
                                                          const double *__restrict__ gS2, const float *__restrict__ hin,
                                                          const float *__restrict__ dyn, float *__restrict__ dWt) {
    constexpr int FPL = H / 32;
    __shared__ float sH[kTile][3];
    __shared__ float sD[kTile][H + 1];
    const int t = blockIdx.x, a = tstart[t], nn = tstart[t + 1] - a, g = tgraph[t];
    const float inv_n = 1.f / (gptr[g + 1] - gptr[g]);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const NormBwd<FPL> nb(g, H, lane, inv_n, mu, rstd, gamma, gS1, gS2);
    for (int k = warp; k < nn; k += kBlock / 32) {
        float d[FPL], yv[FPL];
        lane_load<FPL>(dyn, a + k, lane, d);
        lane_load<FPL>(y, a + k, lane, yv);
#pragma unroll
        for (int j = 0; j < FPL; ++j) sD[k][FPL * lane + j] = nb.dy(j, d[j], yv[j]);
        if (lane < 2) sH[k][lane] = hin[static_cast<size_t>(a + k) * 2 + lane];
    }
    __syncthreads();
    float *out = dWt + static_cast<size_t>(t) * (H * H + H);
    for (int e = threadIdx.x; e < 2 * H; e += kBlock) {
        const int mm = e / H, kk = e % H;
        float acc = 0.f;
        for (int j = 0; j < nn; ++j) acc = fmaf(sH[j][mm], sD[j][kk], acc);
        out[e] = acc;
    }
    if (threadIdx.x < H) {
        float acc = 0.f;
        for (int j = 0; j < nn; ++j) acc += sD[j][threadIdx.x];
        out[H * H + threadIdx.x] = acc;
    }
}

// dx = A_hat dh (A_hat symmetric), H features, 32 / (H / 4) nodes per warp.
template <int H>
__global__ void __launch_bounds__(kBlock) k_agg_plain(int N, const int *__restrict__ rp, const int *__restrict__ col,
                                                      const float *__restrict__ w, const float *__restrict__ v,
                                                      float *__restrict__ out) {
    constexpr int L = H / 4, R = 32 / L;
    const int wid = (blockIdx.x * kBlock + threadIdx.x) / 32, lane = threadIdx.x % 32, hl = lane % L;
    const int i0 = R * wid;
    if (i0 >= N) return;                         // warp-uniform
    const int i = i0 + lane / L;
    const bool live = i < N;
    const int p0 = rp[live ? i : i0], p1 = live ? rp[i + 1] : p0;
    const float4 h = agg_rows<H>(p0, p1, col, w, reinterpret_cast<const float4 *>(v), hl);
    if (live) reinterpret_cast<float4 *>(out)[static_cast<size_t>(i) * L + hl] = h;
}

// Conv weight/bias gradient: tile partials summed per chunk of tiles (FP64,
// tile order), then the chunks in order; instance-norm affine gradients are
// the per-graph sums added in graph order.
template <int H>
constexpr int grad_stride() { return H * H + H; }
template <int H>
__global__ void k_layer_param_partial(int NT, int fin, const float *__restrict__ dWt, double *__restrict__ chunk) {
    const int e = blockIdx.x * kBlock + threadIdx.x, c = blockIdx.y;
    const int nW = fin * H;
    if (e >= nW + H) return;
    const int src = (e < nW) ? e : H * H + (e - nW);
    const int t0 = static_cast<int>(static_cast<long long>(NT) * c / kGradChunks);
    const int t1 = static_cast<int>(static_cast<long long>(NT) * (c + 1) / kGradChunks);
    double acc = 0.0;
    for (int t = t0; t < t1; ++t) acc += dWt[static_cast<size_t>(t) * grad_stride<H>() + src];
    chunk[static_cast<size_t>(c) * grad_stride<H>() + e] = acc;
}

template <int H>
__global__ void k_layer_param_final(int G, int fin, const double *__restrict__ chunk, const double *__restrict__ gS1,
                                    const double *__restrict__ gS2, float *__restrict__ gW, float *__restrict__ gB,
                                    float *__restrict__ gG, float *__restrict__ gBeta) {
    const int e = blockIdx.x * kBlock + threadIdx.x;
    const int nW = fin * H;
    if (e < nW + H) {
        double acc = 0.0;
        for (int c = 0; c < kGradChunks; ++c) acc += chunk[static_cast<size_t>(c) * grad_stride<H>() + e];
        if (e < nW) gW[e] = static_cast<float>(acc);
        else gB[e - nW] = static_cast<float>(acc);
    } else if (e < nW + 2 * H) {
        const int f = e - nW - H;
        double s1 = 0.0, s2 = 0.0;
        for (int g = 0; g < G; ++g) {
            s1 += gS1[g * H + f];
            s2 += gS2[g * H + f];
        }
        gG[f] = static_cast<float>(s2);
        gBeta[f] = static_cast<float>(s1);
    }
}

template <int H>
static void backward_impl(GcinBatch &b, const float *th, float *grad, cudaStream_t s) {
    const ParamLayout &pl = host_layout(H);
    const int N = b.N, G = b.G, NT = b.NT;
    k_head_bwd<H><<<G, 128, 0, s>>>(b.head, th, b.dc, b.dhead, b.dpooled); AMG_COUNT();
    const int nhead = pl.total - pl.roW[0];
    k_head_param_grad<H><<<grid_for(nhead), kBlock, 0, s>>>(G, b.pooled, b.head, b.dhead, b.dc, grad); AMG_COUNT();
    constexpr int R = 32 / (H / 4);                                          // nodes per warp
    const int warp_grid = grid_for((static_cast<long long>(N) + R - 1) / R * 32);
    for (int l = kLayers - 1; l >= 0; --l) {
        k_bwd_relu_tile<H><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.gptr, b.x[l], b.y[l], b.mu[l], b.rstd[l],
                                                 l == kLayers - 1 ? nullptr : b.dx, b.dpooled, b.argmax, l, b.dy,
                                                 b.tsum, b.tsum2); AMG_COUNT();
        k_bwd_combine<H><<<G, combine_threads<H>(), 0, s>>>(b.gtile, b.tsum, b.tsum2, b.gS1, b.gS2); AMG_COUNT();
        if (l > 0 && b.bf16) {
            // the forward's node linear ran on the tensor cores: so does its backward
            k_bwd_lin_tc<H><<<(NT + 1) / 2, kBlock, tcb_smem<H>(), s>>>(b.tstart, b.tgraph, b.gptr, NT, b.y[l], b.mu[l],
                                                                      b.rstd[l], th + pl.inG[l], b.gS1, b.gS2,
                                                                      th + pl.convW[l], b.h[l], b.dy, b.dh, b.dWt,
                                                                      b.err); AMG_COUNT();
            k_agg_plain<H><<<warp_grid, kBlock, 0, s>>>(N, b.rp, b.col, b.w, b.dh, b.dx); AMG_COUNT();
        } else if (l > 0) {
            k_bwd_lin_tile<H><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.gptr, b.y[l], b.mu[l], b.rstd[l],
                                                    th + pl.inG[l], b.gS1, b.gS2, th + pl.convW[l], b.h[l], b.dy, b.dh,
                                                    b.dWt, b.bf16); AMG_COUNT();
            k_agg_plain<H><<<warp_grid, kBlock, 0, s>>>(N, b.rp, b.col, b.w, b.dh, b.dx); AMG_COUNT();
        } else {
            k_bwd_lin1_tile<H><<<NT, kBlock, 0, s>>>(b.tstart, b.tgraph, b.gptr, b.y[l], b.mu[l], b.rstd[l],
                                                     th + pl.inG[l], b.gS1, b.gS2, b.h1, b.dy, b.dWt); AMG_COUNT();
        }
        const int fin = (l == 0) ? 2 : H;
        k_layer_param_partial<H><<<dim3(grid_for(fin * H + H), kGradChunks), kBlock, 0, s>>>(NT, fin, b.dWt,
                                                                                          b.dWc); AMG_COUNT();
        k_layer_param_final<H><<<grid_for(fin * H + 2 * H), kBlock, 0, s>>>(
            G, fin, b.dWc, b.gS1, b.gS2, grad + pl.convW[l], grad + pl.convB[l], grad + pl.inG[l],
            grad + pl.inB[l]); AMG_COUNT();
    }
}

void gcin_backward(GcinBatch &b, const float *th, float *grad, cudaStream_t s) {
    if (b.hidden == kHidden32) backward_impl<kHidden32>(b, th, grad, s);
    else backward_impl<kHidden>(b, th, grad, s);
}

// ---------------------------------------------------------------------------
// optimiser: global-norm clipping + Adam (Table train_hyper)
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock) k_sq_partial_f(int n, const float *__restrict__ v, double *__restrict__ part) {
    __shared__ double red[kBlock / 32];
    double s = 0.0;
    for (int i = blockIdx.x * kBlock + threadIdx.x; i < n; i += gridDim.x * kBlock) s += static_cast<double>(v[i]) * v[i];
    s = warp_sum(s);
    if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < kBlock / 32; ++k) t += red[k];
        part[blockIdx.x] = t;
    }
}

__global__ void k_norm_from_partials(int np, const double *__restrict__ part, double *__restrict__ out) {
    if (threadIdx.x != 0) return;
    double s = 0.0;
    for (int i = 0; i < np; ++i) s += part[i];
    *out = sqrt(s);
}

// clip to max_norm (scale = min(1, max_norm / (||g|| + 1e-6))), then Adam
__global__ void k_adam(int n, float *__restrict__ theta, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, const double *__restrict__ gnorm, double max_norm, double lr,
                       double b1, double b2, double eps, double bc1, double bc2) {
    const int i = blockIdx.x * kBlock + threadIdx.x;
    if (i >= n) return;
    const double scale = fmin(1.0, max_norm / (*gnorm + 1e-6));
    const double gi = g[i] * scale;
    const double mi = b1 * m[i] + (1.0 - b1) * gi;
    const double vi = b2 * v[i] + (1.0 - b2) * gi * gi;
    m[i] = static_cast<float>(mi);
    v[i] = static_cast<float>(vi);
    theta[i] = static_cast<float>(theta[i] - lr * (mi / bc1) / (sqrt(vi / bc2) + eps));
}

void gcin_engine_free(GcinEngine *e) {
    if (!e) return;
    if (e->exec) cudaGraphExecDestroy(e->exec);
    gcin_batch_free(e->batch);
    if (e->theta) cudaFree(e->theta);
    delete e;
}

}  // namespace amg

using namespace amg;

struct gcin_trainer {
    int device = 0;
    int bf16 = 0;
    int hidden = kHidden;            // GCIN width of the parameters
    int n = kNumParams;              // parameter count
    std::string err;
    cudaStream_t stream = nullptr;
    float *theta = nullptr, *grad = nullptr, *m = nullptr, *v = nullptr;
    double *part = nullptr;          // norm partials + the norm
    long long step = 0;
    GcinBatch batch;
    std::vector<const amg_ctx *> key;
    std::vector<long long> versions;
    bool have_forward = false;
};

static int tr_fail(gcin_trainer *t, int rc, const std::string &msg) {
    if (t) t->err = msg;
    return rc;
}

static int tr_cuda(gcin_trainer *t, cudaError_t e, const char *what) {
    if (e == cudaSuccess) return AMG_OK;
    return tr_fail(t, AMG_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

constexpr int kNormBlocks = 64;

extern "C" {

int gnn_load_params(amg_ctx *c, const float *theta, long long n) {
    if (!c) return AMG_ERR_ARG;
    c->err.clear();
    const int H = hidden_of(n);
    if (!theta || !H) return ctx_fail(c, "expected 55045 (hidden 64) or 37189 (hidden 32) parameters"), AMG_ERR_ARG;
    cudaError_t e = cudaSetDevice(c->opt.device);
    if (e != cudaSuccess) return ctx_cuda_check(c, e, "cudaSetDevice");
    if (!c->gnn) {
        c->gnn = new GcinEngine();
        // the parameters and, 256-byte aligned behind them, the packed B tiles
        const size_t tb = (sizeof(float) * kNumParams + 255) / 256 * 256;
        e = cudaMalloc(&c->gnn->theta, tb + static_cast<size_t>(kLayers - 1) * kHidden * kHidden * 2);
        if (e == cudaSuccess) c->gnn->wtile = reinterpret_cast<unsigned char *>(c->gnn->theta) + tb;
        if (e != cudaSuccess) {
            delete c->gnn;
            c->gnn = nullptr;
            return ctx_cuda_check(c, e, "cudaMalloc params");
        }
    }
    e = cudaMemcpyAsync(c->gnn->theta, theta, sizeof(float) * n, cudaMemcpyHostToDevice, c->stream);
    if (e == cudaSuccess) {
        pack_wtiles(H, c->gnn->theta, c->gnn->wtile, c->stream);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess) return ctx_cuda_check(c, e, "upload params");
    c->gnn->have_params = true;
    c->gnn->hidden = H;
    return AMG_OK;
}

int gnn_predict_coeffs(amg_ctx *c, double *c_out) {
    if (!c) return AMG_ERR_ARG;
    c->err.clear();
    if (c->lev.empty()) return ctx_fail(c, "no hierarchy loaded"), AMG_ERR_STATE;
    if (!c->gnn || !c->gnn->have_params) return ctx_fail(c, "no GCIN parameters loaded"), AMG_ERR_STATE;
    cudaError_t e = cudaSetDevice(c->opt.device);
    if (e != cudaSuccess) return ctx_cuda_check(c, e, "cudaSetDevice");
    GcinEngine *g = c->gnn;
    cudaStream_t s = c->stream;
    if (g->batch_version != c->hier_version || g->batch.G != static_cast<int>(c->lev.size())) {
        std::string err;
        amg_ctx *one[1] = {c};
        int rc = gcin_batch_build(g->batch, 1, one, s, err, false);
        if (rc) return ctx_fail(c, err), rc;
        g->batch_version = c->hier_version;
    }
    g->batch.bf16 = (c->opt.gnn_precision == AMG_GNN_BF16) ? 1 : 0;
    g->batch.infer = 1;
    g->batch.hidden = g->hidden;
    g->batch.wtile = g->wtile;
    // forward + smoother assembly (straight from the device coefficients) run
    // as one CUDA graph, captured once per batch and arithmetic: 28 small
    // kernels whose host launch cost would otherwise exceed their run time
    const int key = g->batch.bf16 + 2 * c->opt.precision + 4 * (g->hidden == kHidden32 ? 1 : 0);
    if (!g->exec || g->exec_version != g->batch_version || g->exec_key != key) {
        if (g->exec) cudaGraphExecDestroy(g->exec);
        g->exec = nullptr;
        gcin_prepare_device();
        cudaGraph_t graph = nullptr;
        e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return ctx_cuda_check(c, e, "GCIN capture begin");
        const long long before = g_launches.load();
        gcin_forward(g->batch, g->theta, s);
        const int rc0 = enqueue_coeff_assembly(c, g->batch.c, s);
        g->exec_kernels = g_launches.load() - before;
        g_launches.fetch_sub(g->exec_kernels);
        e = cudaStreamEndCapture(s, &graph);
        if (rc0) {
            if (graph) cudaGraphDestroy(graph);
            return rc0;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&g->exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            g->exec = nullptr;
            return ctx_cuda_check(c, e, "GCIN graph");
        }
        g->exec_version = g->batch_version;
        g->exec_key = key;
    }
    e = cudaGraphLaunch(g->exec, s);
    if (e != cudaSuccess) return ctx_cuda_check(c, e, "GCIN graph launch");
    g_launches.fetch_add(g->exec_kernels);
    c->have_q = true;
    c->q_nodes = false;
    c->tail[1].ok = false;                         // re-formed by the next V-cycle
    c->q64_stale = c->opt.precision != AMG_FP64;   // the graph assembled the FP32 values only
    c->smoother = AMG_SMOOTHER_GNN;
    int dflag = 0;
    const int G = g->batch.G;
    std::vector<float> cf(static_cast<size_t>(G) * 5);
    e = cudaMemcpyAsync(cf.data(), g->batch.c, sizeof(float) * cf.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&dflag, g->batch.err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return ctx_cuda_check(c, e, "GCIN forward and smoother assembly");
    bool finite = true;
    for (size_t k = 0; k < static_cast<size_t>(G - 1) * 5; ++k) finite = finite && std::isfinite(cf[k]);   // smoothed levels
    if (dflag || !finite) {
        c->have_q = false;
        c->smoother = AMG_SMOOTHER_JACOBI;
        if (dflag) return ctx_fail(c, "tensor-core GCIN kernel timed out waiting for its MMAs"), AMG_ERR_DEVICE_FLAG;
        return ctx_fail(c, "non-finite coefficient"), AMG_ERR_ARG;
    }
    if (c_out) std::copy(cf.begin(), cf.end(), c_out);
    return AMG_OK;
}

int gcin_tc_selftest(int device, int no_commit, const float *x, const float *W, const float *bias, float *y,
                     float *h, int *flag) {
    if (!x || !W || !bias || !y || !h || !flag) return AMG_ERR_ARG;
    if (cudaSetDevice(device) != cudaSuccess) return AMG_ERR_CUDA;
    gcin_prepare_device();
    constexpr int n = kTcRows;
    // identity graph (h = x), two 64-node tiles
    std::vector<int> rp(n + 1), col(n), tstart = {0, kTile, 2 * kTile};
    std::vector<float> w(n, 1.0f);
    for (int i = 0; i <= n; ++i) rp[i] = i;
    for (int i = 0; i < n; ++i) col[i] = i;
    char *mem = nullptr;
    Planner pl;
    auto lay = [&](Planner &P) {
        struct L { int *rp, *col, *ts, *err; float *w, *x, *W, *b, *h, *y, *tm, *t2; } l{};
        l.rp = P.take<int>(n + 1); l.col = P.take<int>(n); l.ts = P.take<int>(3); l.err = P.take<int>(4);
        l.w = P.take<float>(n); l.x = P.take<float>(n * kHidden); l.W = P.take<float>(kHidden * kHidden);
        l.b = P.take<float>(kHidden); l.h = P.take<float>(n * kHidden); l.y = P.take<float>(n * kHidden);
        l.tm = P.take<float>(2 * kHidden); l.t2 = P.take<float>(2 * kHidden);
        return l;
    };
    lay(pl);
    if (cudaMalloc(&mem, pl.off) != cudaSuccess) return AMG_ERR_CUDA;
    Planner p2;
    p2.base = mem;
    auto L = lay(p2);
    cudaError_t e = cudaMemset(mem, 0, p2.off);
    if (e == cudaSuccess) e = cudaMemcpy(L.rp, rp.data(), sizeof(int) * rp.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.col, col.data(), sizeof(int) * col.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.ts, tstart.data(), sizeof(int) * 3, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.w, w.data(), sizeof(float) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.x, x, sizeof(float) * n * kHidden, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.W, W, sizeof(float) * kHidden * kHidden, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(L.b, bias, sizeof(float) * kHidden, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        k_agg_lin_tc<kHidden><<<1, kBlock, tc_smem<kHidden>()>>>(L.rp, L.col, L.w, L.x, L.W, nullptr, L.b, L.ts, 2, L.h, L.y, L.tm, L.t2, L.err,
                                             no_commit ? 1 : 0); AMG_COUNT();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(y, L.y, sizeof(float) * n * kHidden, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(h, L.h, sizeof(float) * n * kHidden, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(flag, L.err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(mem);
    return e == cudaSuccess ? AMG_OK : AMG_ERR_CUDA;
}

int gcin_trainer_create(gcin_trainer **out, int device, int precision, const float *theta0, long long n_params) {
    if (!out || !theta0 || (precision != AMG_GNN_FP32 && precision != AMG_GNN_BF16) || !hidden_of(n_params))
        return AMG_ERR_ARG;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return AMG_ERR_CUDA;
    gcin_trainer *t = new gcin_trainer();
    t->device = device;
    t->bf16 = (precision == AMG_GNN_BF16) ? 1 : 0;
    t->hidden = hidden_of(n_params);
    t->n = static_cast<int>(n_params);
    cudaError_t e = cudaStreamCreateWithFlags(&t->stream, cudaStreamNonBlocking);
    const size_t P = t->n;
    const size_t fbytes = ((sizeof(float) * 4 * P + 255) / 256) * 256;
    if (e == cudaSuccess) e = cudaMalloc(&t->theta, fbytes + sizeof(double) * (kNormBlocks + 1));
    if (e != cudaSuccess) {
        if (t->stream) cudaStreamDestroy(t->stream);
        delete t;
        return AMG_ERR_CUDA;
    }
    t->grad = t->theta + P;
    t->m = t->grad + P;
    t->v = t->m + P;
    t->part = reinterpret_cast<double *>(reinterpret_cast<char *>(t->theta) + fbytes);
    e = cudaMemcpyAsync(t->theta, theta0, sizeof(float) * P, cudaMemcpyHostToDevice, t->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(t->grad, 0, sizeof(float) * 3 * P, t->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(t->stream);
    if (e != cudaSuccess) {
        gcin_trainer_destroy(t);
        return AMG_ERR_CUDA;
    }
    *out = t;
    return AMG_OK;
}

void gcin_trainer_destroy(gcin_trainer *t) {
    if (!t) return;
    cudaSetDevice(t->device);
    if (t->stream) cudaStreamSynchronize(t->stream);
    gcin_batch_free(t->batch);
    if (t->theta) cudaFree(t->theta);
    if (t->stream) cudaStreamDestroy(t->stream);
    delete t;
}

const char *gcin_trainer_last_error(const gcin_trainer *t) { return t ? t->err.c_str() : "trainer is NULL"; }

int gcin_trainer_get_params(const gcin_trainer *tc, float *theta_out) {
    gcin_trainer *t = const_cast<gcin_trainer *>(tc);
    if (!t || !theta_out) return AMG_ERR_ARG;
    int rc = tr_cuda(t, cudaSetDevice(t->device), "cudaSetDevice");
    if (rc) return rc;
    rc = tr_cuda(t, cudaMemcpyAsync(theta_out, t->theta, sizeof(float) * t->n, cudaMemcpyDeviceToHost, t->stream),
                 "params download");
    if (rc) return rc;
    return tr_cuda(t, cudaStreamSynchronize(t->stream), "sync");
}

int gcin_trainer_set_params(gcin_trainer *t, const float *theta, long long n) {
    if (!t) return AMG_ERR_ARG;
    t->err.clear();
    if (!theta || n != t->n) return tr_fail(t, AMG_ERR_ARG, "parameter count differs from the trainer's");
    int rc = tr_cuda(t, cudaSetDevice(t->device), "cudaSetDevice");
    if (rc) return rc;
    rc = tr_cuda(t, cudaMemcpyAsync(t->theta, theta, sizeof(float) * n, cudaMemcpyHostToDevice, t->stream),
                 "params upload");
    if (rc) return rc;
    t->have_forward = false;
    return tr_cuda(t, cudaStreamSynchronize(t->stream), "sync");
}

int gcin_trainer_forward(gcin_trainer *t, int n_problems, amg_ctx *const *problems, double *c_out) {
    if (!t) return AMG_ERR_ARG;
    t->err.clear();
    if (n_problems < 1 || !problems || !c_out) return tr_fail(t, AMG_ERR_ARG, "need at least one problem and c_out");
    int rc = tr_cuda(t, cudaSetDevice(t->device), "cudaSetDevice");
    if (rc) return rc;
    std::vector<const amg_ctx *> key(problems, problems + n_problems);
    std::vector<long long> versions;
    for (int m = 0; m < n_problems; ++m) {
        if (!problems[m]) return tr_fail(t, AMG_ERR_ARG, "NULL problem");
        versions.push_back(problems[m]->hier_version);
    }
    if (key != t->key || versions != t->versions || !t->batch.arena) {
        std::string err;
        rc = gcin_batch_build(t->batch, n_problems, problems, t->stream, err, true);
        if (rc) return tr_fail(t, rc, err);
        t->key = key;
        t->versions = versions;
    }
    t->batch.bf16 = t->bf16;
    t->batch.hidden = t->hidden;
    gcin_forward(t->batch, t->theta, t->stream);
    std::vector<float> cf(static_cast<size_t>(t->batch.G) * 5);
    int dflag = 0;
    rc = tr_cuda(t, cudaGetLastError(), "GCIN forward");
    if (!rc) rc = tr_cuda(t, cudaMemcpyAsync(cf.data(), t->batch.c, sizeof(float) * cf.size(), cudaMemcpyDeviceToHost,
                                             t->stream), "coefficients download");
    if (!rc) rc = tr_cuda(t, cudaMemcpyAsync(&dflag, t->batch.err, sizeof(int), cudaMemcpyDeviceToHost, t->stream),
                          "flag download");
    if (!rc) rc = tr_cuda(t, cudaStreamSynchronize(t->stream), "sync");
    if (rc) return rc;
    if (dflag) return tr_fail(t, AMG_ERR_DEVICE_FLAG, "tensor-core GCIN kernel timed out waiting for its MMAs");
    std::copy(cf.begin(), cf.end(), c_out);
    t->have_forward = true;
    return AMG_OK;
}

int gcin_trainer_backward(gcin_trainer *t, const double *dc, double *dtheta_out) {
    if (!t) return AMG_ERR_ARG;
    t->err.clear();
    if (!dc) return tr_fail(t, AMG_ERR_ARG, "dc is NULL");
    if (!t->have_forward) return tr_fail(t, AMG_ERR_STATE, "backward without a forward");
    int rc = tr_cuda(t, cudaSetDevice(t->device), "cudaSetDevice");
    if (rc) return rc;
    std::vector<float> df(dc, dc + static_cast<size_t>(t->batch.G) * 5);
    rc = tr_cuda(t, cudaMemcpyAsync(t->batch.dc, df.data(), sizeof(float) * df.size(), cudaMemcpyHostToDevice,
                                    t->stream), "dc upload");
    if (rc) return rc;
    gcin_backward(t->batch, t->theta, t->grad, t->stream);
    rc = tr_cuda(t, cudaGetLastError(), "GCIN backward");
    if (rc) return rc;
    std::vector<float> g(t->n);
    if (dtheta_out) {
        rc = tr_cuda(t, cudaMemcpyAsync(g.data(), t->grad, sizeof(float) * t->n, cudaMemcpyDeviceToHost,
                                        t->stream), "gradient download");
        if (rc) return rc;
    }
    int dflag = 0;   // the tensor-core backward's bounded MMA wait
    rc = tr_cuda(t, cudaMemcpyAsync(&dflag, t->batch.err, sizeof(int), cudaMemcpyDeviceToHost, t->stream),
                 "flag download");
    if (rc) return rc;
    rc = tr_cuda(t, cudaStreamSynchronize(t->stream), "sync");
    if (rc) return rc;
    if (dflag) return tr_fail(t, AMG_ERR_DEVICE_FLAG, "tensor-core GCIN kernel timed out waiting for its MMAs");
    if (dtheta_out) std::copy(g.begin(), g.end(), dtheta_out);
    return AMG_OK;
}

int gcin_trainer_adam_step(gcin_trainer *t, double lr, double max_norm) {
    if (!t) return AMG_ERR_ARG;
    t->err.clear();
    if (!(lr >= 0.0) || !(max_norm > 0.0)) return tr_fail(t, AMG_ERR_ARG, "bad lr or max_norm");
    int rc = tr_cuda(t, cudaSetDevice(t->device), "cudaSetDevice");
    if (rc) return rc;
    t->step += 1;
    const double b1 = 0.9, b2 = 0.999, eps = 1e-8;
    const double bc1 = 1.0 - std::pow(b1, static_cast<double>(t->step));
    const double bc2 = 1.0 - std::pow(b2, static_cast<double>(t->step));
    k_sq_partial_f<<<kNormBlocks, kBlock, 0, t->stream>>>(t->n, t->grad, t->part); AMG_COUNT();
    k_norm_from_partials<<<1, 32, 0, t->stream>>>(kNormBlocks, t->part, t->part + kNormBlocks); AMG_COUNT();
    k_adam<<<grid_for(t->n), kBlock, 0, t->stream>>>(t->n, t->theta, t->grad, t->m, t->v,
                                                           t->part + kNormBlocks, max_norm, lr, b1, b2, eps, bc1,
                                                           bc2); AMG_COUNT();
    rc = tr_cuda(t, cudaGetLastError(), "adam");
    if (rc) return rc;
    return tr_cuda(t, cudaStreamSynchronize(t->stream), "sync");
}

}  // extern "C"
