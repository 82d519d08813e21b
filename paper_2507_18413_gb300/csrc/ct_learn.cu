// ct_learn.cu -- the learned branching order: per-variable features of a
// network's state, and the 8 -> 64 -> 64 -> 1 scoring network with its
// training (not in the paper, whose solver branches first-fail; Sec. 4).
//
// Features (kNF = 8 per variable, zero for |D(x)| < 2). With s = |D(x)|, d0
// the initial size, deg(x) the tables holding x (degmax the largest, >= 1),
// smax the largest |D| among the unfixed variables of the same node, and for
// every table c holding x with live_c > 0 valid tuples (tuples whose every
// value is in its current domain: the live bits of currTable),
// p_c(a) = |{valid tuples of c with x = a}| / live_c = popcount(supports[x,a]
// AND currTable) / popcount(currTable):
//   f0 = s / d0, f1 = log2(s) / 8, f2 = deg / degmax,
//   f3 = mean_c s * min_a p_c(a), f4 = mean_c max_a p_c(a),
//   f5 = mean_c (-sum_a p_c(a) log2 p_c(a)) / log2(s),
//   f6 = mean_c log2(1 + live_c) / 32, f7 = s / smax.
// The counts are integers (a warp per (table, segment), lane per chunk, or on
// small networks a CTA per variable and table); what is made of them is float.
//
// Network: h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), out = W3 . h2 + b3,
// float32, weights flat as W1[64][8], b1, W2[64][64], b2, W3[64], b3.
// Training: loss sum (out - y)^2 / (2B) per batch, Adam (Kingma and Ba, 2015;
// beta1 0.9, beta2 0.999, eps 1e-8, bias-corrected), one cluster of CTAs that
// keeps the weights and the batch's activations in shared memory and the
// moments in registers and walks the given epoch orders in consecutive batches.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "ct_learn.cuh"

using namespace ctk;

struct ct_mlp {
    float* d_w = nullptr;  // [kNW]
    float* d_m = nullptr;  // Adam first moment
    float* d_v = nullptr;  // Adam second moment
    int64_t t = 0;         // Adam steps taken
    cudaStream_t stream = nullptr;
    bool ownStream = false;
};

namespace {

struct FeatArgs {
    const TableDev* tabs;
    const uint32_t* dom;
    const uint8_t* nodeActive;
    const int32_t* rowBase;
    const int32_t* unitBase;
    const int32_t* scopeBase;
    const int32_t* scopeOff;
    const int32_t* adjBase;
    const int2* adj;
    const int32_t* varOff;
    const int32_t* varNW;
    const int32_t* varD0;
    const int32_t* deg;
    uint32_t* counts;
    uint32_t* live;
    float* feat;
    int32_t nt, nv, T, V, degmax, totalUnits;
    // the one-kernel path
    const int32_t* pairVar;
    float4* pairStat;
    unsigned* ticket;
    int32_t pairs;
    float* publish;  // mapped host memory, or null
};

__device__ __forceinline__ uint32_t popc4(const uint4& v) {
    return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}

__device__ __forceinline__ uint32_t warp_sum(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ uint32_t warp_min(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ uint32_t warp_max(uint32_t v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

__device__ __forceinline__ float warp_sum_f32(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Valid tuples per supports row and per table: one warp per (table, segment,
// scope variable, domain word) unit, lane l holding live chunk 32 * segment +
// l. Only the rows of the word's present values are read, none for a fixed
// variable (its features are zero), eight row loads in flight; the unit of the
// first word of the first scope variable also counts the segment's valid
// tuples.
__global__ void ct_counts_kernel(const FeatArgs A) {
    const int lane = threadIdx.x & 31;
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int u = gwarp; u < A.totalUnits; u += nwarps) {
        int lo = 0, hi = A.nt - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&A.unitBase[mid]) <= u) lo = mid;
            else hi = mid - 1;
        }
        const int t = lo;
        if (A.nodeActive && !A.nodeActive[t / A.T]) continue;
        const TableDev& T = A.tabs[t];
        const int s0 = __ldg(&A.scopeBase[t]);
        const int ar = __ldg(&A.scopeBase[t + 1]) - s0;
        int sw = 0;
        for (int k = 0; k < ar; ++k) sw += __ldg(&T.varNW[k]);
        const int local = u - __ldg(&A.unitBase[t]);
        const int seg = local / sw;
        int i = 0, q = local - seg * sw;
        while (i < ar && q >= __ldg(&T.varNW[i])) q -= __ldg(&T.varNW[i++]);
        if (i >= ar) continue;
        const uint32_t mask = T.segMask[seg];
        if (mask == 0u) continue;
        const int w = seg * 32 + lane;
        const bool act = (mask >> lane) & 1u;
        const uint4 cur = act ? T.curr[w] : make_uint4(0u, 0u, 0u, 0u);
        if (i == 0 && q == 0) {
            const uint32_t lv = warp_sum(popc4(cur));
            if (lane == 0 && lv) atomicAdd(&A.live[t], lv);
        }
        const uint32_t* dv = A.dom + __ldg(&A.scopeOff[s0 + i]);
        const int nw = __ldg(&T.varNW[i]);
        uint32_t sz = 0;
        for (int k = lane; k < nw; k += 32) sz += __popc(dv[k]);
        if (warp_sum(sz) < 2u) continue;
        const int row0 = __ldg(&T.varRow0[i]);
        const int base = __ldg(&A.rowBase[t]) + row0;
        const size_t W4 = (size_t)T.W4;
        const uint4* sp = T.sup + (size_t)row0 * W4 + w;
        {
            uint32_t bits = dv[q];
            while (bits) {
                int a[8];
                uint32_t n[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    a[j] = bits ? 32 * q + __ffs(bits) - 1 : -1;
                    bits &= bits - 1u;
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    n[j] = 0u;
                    if (a[j] >= 0 && act) {
                        const uint4 s = __ldg(sp + (size_t)a[j] * W4);
                        n[j] = popc4(make_uint4(s.x & cur.x, s.y & cur.y, s.z & cur.z, s.w & cur.w));
                    }
                }
                // sums of the eight rows over the warp: three halving exchanges
                // leave lane l one row (4 b4 + 2 b3 + b2 of l), two more add it up
                const bool h4 = lane & 16, h3 = lane & 8, h2 = lane & 4;
                uint32_t m4[4], m2[2];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    m4[k] = (h4 ? n[k + 4] : n[k]) + __shfl_xor_sync(0xffffffffu, h4 ? n[k] : n[k + 4], 16);
#pragma unroll
                for (int k = 0; k < 2; ++k)
                    m2[k] = (h3 ? m4[k + 2] : m4[k]) + __shfl_xor_sync(0xffffffffu, h3 ? m4[k] : m4[k + 2], 8);
                uint32_t v = (h2 ? m2[1] : m2[0]) + __shfl_xor_sync(0xffffffffu, h2 ? m2[0] : m2[1], 4);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                const int jr = (h4 ? 4 : 0) + (h3 ? 2 : 0) + (h2 ? 1 : 0);
                int ar = a[0];
#pragma unroll
                for (int j = 1; j < 8; ++j) ar = jr == j ? a[j] : ar;
                if ((lane & 3) == 0 && ar >= 0 && v) atomicAdd(&A.counts[base + ar], v);
            }
        }
    }
}

// Features of a node's variables: `perNode` CTAs per node, one warp per
// variable, lane l holding the values 32 q + l. Every CTA first takes the
// node's largest unfixed domain. Minimum and maximum counts are taken on the
// integers; the rest is float: a lane sums the entropy terms of its values
// (d / 32 of a domain of d values) before the warp reduction, a relative error
// of a few 1e-7 up to about a thousand values.
__global__ void ct_features_kernel(const FeatArgs A, int perNode) {
    const int node = blockIdx.x / perNode;
    if (A.nodeActive && !A.nodeActive[node]) return;
    __shared__ int red[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    const int firstVar = (blockIdx.x - node * perNode) * nwarp;
    int mx = 0;
    for (int lx = tid; lx < A.V; lx += blockDim.x) {
        const int v = node * A.V + lx;
        int s = 0;
        for (int q = 0; q < A.varNW[v]; ++q) s += __popc(A.dom[A.varOff[v] + q]);
        if (s >= 2 && s > mx) mx = s;
    }
    mx = (int)warp_max((uint32_t)mx);
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    int smax = 0;
    for (int k = 0; k < nwarp; ++k) smax = max(smax, red[k]);
    for (int lx = firstVar + warp; lx < A.V && lx < firstVar + nwarp; lx += nwarp) {
        const int v = node * A.V + lx;
        float* f = A.feat + (size_t)v * kNF;
        const uint32_t* d = A.dom + A.varOff[v];
        const int nw = A.varNW[v];
        uint32_t su = 0;
        for (int q = lane; q < nw; q += 32) su += __popc(d[q]);
        const int s = (int)warp_sum(su);
        if (s < 2) {
            if (lane < kNF) f[lane] = 0.0f;
            continue;
        }
        float bal = 0.0f, top = 0.0f, ent = 0.0f, liv = 0.0f;
        int cnt = 0;
        const float ls = log2f((float)s);
        for (int j = A.adjBase[v]; j < A.adjBase[v + 1]; ++j) {
            const int2 e = A.adj[j];
            const uint32_t live = A.live[e.x];
            if (live == 0u) continue;
            const int row0 = A.tabs[e.x].varRow0[e.y];
            const uint32_t* c = A.counts + A.rowBase[e.x] + row0;
            const float fl = (float)live;
            uint32_t cmin = 0xffffffffu, cmax = 0u;
            float hl = 0.0f;
            for (int q0 = 0; q0 < nw; q0 += 4) {
                bool pr[4];
                uint32_t cq[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int q = q0 + k;
                    pr[k] = q < nw && ((d[q] >> lane) & 1u);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) cq[k] = pr[k] ? c[(q0 + k) * 32 + lane] : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (!pr[k]) continue;
                    cmin = min(cmin, cq[k]);
                    cmax = max(cmax, cq[k]);
                    if (cq[k]) {
                        const float p = (float)cq[k] / fl;
                        hl -= p * log2f(p);
                    }
                }
            }
            cmin = warp_min(cmin);
            cmax = warp_max(cmax);
            hl = warp_sum_f32(hl);
            bal += (float)s * ((float)cmin / fl);
            top += (float)cmax / fl;
            ent += hl / ls;
            liv += log2f(1.0f + fl) / 32.0f;
            ++cnt;
        }
        if (lane == 0) {
            const float inv = cnt ? 1.0f / (float)cnt : 0.0f;
            f[0] = (float)s / (float)A.varD0[v];
            f[1] = ls / 8.0f;
            f[2] = (float)A.deg[v] / (float)A.degmax;
            f[3] = bal * inv;
            f[4] = top * inv;
            f[5] = ent * inv;
            f[6] = liv * inv;
            f[7] = (float)s / (float)smax;
        }
    }
}

// The features of networks of small tables in one kernel: a CTA per (variable,
// table) entry counts the table's valid tuples for every value of the variable
// in shared memory and stores the entry's part of the features; the node's last
// CTA adds the parts up per variable, in the order and with the operations of
// ct_features_kernel. What bounds it is the chain of round trips of one CTA:
// the two kernels above with their two memsets took 42 us per node on 25
// variables and 40 tables of up to 157 chunks, this one 10. For one network the
// last CTA also writes the features where the host reads them, and a word that
// the host waits for (a copy and a stream synchronisation took 6 us more of
// ct_model_features' 28). The line to the two kernels, which spread the counts
// and the sums over the grid, lies where those catch up (ct_model_features in us,
// this kernel and those):
//   an entry's values x chunks, all one CTA's: 128 x 256 57 and 60 us (3 tables)
//   or 61 and 74 (40 tables), 512 x 64 57 and 62, 60 and 87; beyond, 192 x 256 68
//   and 59, 125 and 94, 1,024 x 64 89 and 62;
//   a node's variables, one per thread of its last CTA: 256 in 8 tables each 52
//   and 75, in 24 each 95 and 105; beyond, 384 73 and 76, 140 and 118, 512 79 and
//   78, 157 and 124, 2,048 221 and 117, 636 and 315.
// Batches of nodes (the batched search with a policy, ms, this kernel and those):
// many entries of short tables leave it bound by its CTAs, 600 of 16 chunks at 200
// variables 60.6 and 59.9 on 8 nodes, 30.6 and 26.4 on 64; 300 of 94 chunks at
// 100 variables 7.2 and 7.3 on 64; 192 of 40 chunks at 64 variables 12.2 and 12.8.
constexpr int kFeatNodeVars = 64, kFeatEntries = 16384;
constexpr int kFeatThreads = 256, kFeatVars = kFeatThreads;
constexpr int kFeatChunks = 256, kFeatValues = 1024, kFeatTests = 32768;  // of a table, a variable, an entry

__global__ void __launch_bounds__(kFeatThreads) ct_features_small_kernel(const FeatArgs A) {
    __shared__ uint4 cur[kFeatChunks];
    __shared__ uint32_t counts[kFeatValues];
    __shared__ uint32_t s_live;
    __shared__ int s_last, s_size[kFeatVars], red[kFeatThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int nwarp = kFeatThreads / 32;
    const int p = blockIdx.x, node = p / A.pairs;
    if (A.nodeActive && !A.nodeActive[node]) return;
    {
        const int v = __ldg(&A.pairVar[p]);
        const int2 e = __ldg(&A.adj[p]);
        const TableDev& T = A.tabs[e.x];
        const uint32_t* d = A.dom + __ldg(&A.varOff[v]);
        const int nw = __ldg(&A.varNW[v]);
        if (tid == 0) s_live = 0u;
        uint32_t su = 0;
        for (int q = lane; q < nw; q += 32) su += __popc(d[q]);
        const int s = (int)warp_sum(su);  // the same in every warp
        const int W4 = T.W4;
        for (int c = tid; c < W4; c += kFeatThreads) cur[c] = T.curr[c];
        __syncthreads();
        if (s >= 2) {
            uint32_t lv = 0;
            for (int c = tid; c < W4; c += kFeatThreads) lv += popc4(cur[c]);
            lv = warp_sum(lv);
            if (lane == 0 && lv) atomicAdd(&s_live, lv);
            const uint4* row = T.sup + (size_t)T.varRow0[e.y] * W4;
            const int values = nw * 32;
            for (int a0 = 4 * warp; a0 < values; a0 += 4 * nwarp) {
                const uint32_t word = d[a0 >> 5] >> (a0 & 31);
                if (!(word & 15u)) continue;
                uint32_t n[4] = {0u, 0u, 0u, 0u};
                for (int c = lane; c < W4; c += 32) {
                    const uint4 w = cur[c];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (!((word >> k) & 1u)) continue;
                        const uint4 x = __ldg(row + (size_t)(a0 + k) * W4 + c);
                        n[k] += popc4(make_uint4(x.x & w.x, x.y & w.y, x.z & w.z, x.w & w.w));
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t sum = __reduce_add_sync(0xffffffffu, n[k]);
                    if (lane == 0) counts[a0 + k] = sum;
                }
            }
        }
        __syncthreads();
        if (warp == 0) {
            float4 part = make_float4(0.0f, 0.0f, 0.0f, -1.0f);  // w < 0: the table has no valid tuple
            if (s >= 2 && s_live) {
                const float fl = (float)s_live, ls = log2f((float)s);
                uint32_t cmin = 0xffffffffu, cmax = 0u;
                float hl = 0.0f;
                for (int q = 0; q < nw; ++q) {
                    if (!((d[q] >> lane) & 1u)) continue;
                    const uint32_t c = counts[q * 32 + lane];
                    cmin = min(cmin, c);
                    cmax = max(cmax, c);
                    if (c) {
                        const float pr = (float)c / fl;
                        hl -= pr * log2f(pr);
                    }
                }
                cmin = warp_min(cmin);
                cmax = warp_max(cmax);
                hl = warp_sum_f32(hl);
                part = make_float4((float)cmin / fl, (float)cmax / fl, hl / ls, log2f(1.0f + fl) / 32.0f);
            }
            if (lane == 0) {
                A.pairStat[p] = part;
                __threadfence();
                s_last = atomicAdd(&A.ticket[node], 1u) == (unsigned)A.pairs - 1u;
            }
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid == 0) A.ticket[node] = 0u;
    int mx = 0;
    for (int lx = tid; lx < A.V; lx += kFeatThreads) {
        const int v = node * A.V + lx;
        int s = 0;
        for (int q = 0; q < A.varNW[v]; ++q) s += __popc(A.dom[A.varOff[v] + q]);
        s_size[lx] = s;
        if (s >= 2 && s > mx) mx = s;
    }
    mx = (int)warp_max((uint32_t)mx);
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    int smax = 0;
    for (int k = 0; k < nwarp; ++k) smax = max(smax, red[k]);
    for (int lx = tid; lx < A.V; lx += kFeatThreads) {
        const int v = node * A.V + lx, s = s_size[lx];
        float f[kNF] = {};
        if (s >= 2) {
            const float ls = log2f((float)s);
            float bal = 0.0f, top = 0.0f, ent = 0.0f, liv = 0.0f;
            int cnt = 0;
            for (int j = A.adjBase[v]; j < A.adjBase[v + 1]; ++j) {
                const float4 x = __ldcg(&A.pairStat[j]);
                if (x.w < 0.0f) continue;
                bal += (float)s * x.x;
                top += x.y;
                ent += x.z;
                liv += x.w;
                ++cnt;
            }
            const float inv = cnt ? 1.0f / (float)cnt : 0.0f;
            f[0] = (float)s / (float)A.varD0[v];
            f[1] = ls / 8.0f;
            f[2] = (float)A.deg[v] / (float)A.degmax;
            f[3] = bal * inv;
            f[4] = top * inv;
            f[5] = ent * inv;
            f[6] = liv * inv;
            f[7] = (float)s / (float)smax;
        }
#pragma unroll
        for (int k = 0; k < kNF; ++k) A.feat[(size_t)v * kNF + k] = f[k];
        if (A.publish) {
            float4* out = reinterpret_cast<float4*>(A.publish) + 2 * lx;
            out[0] = make_float4(f[0], f[1], f[2], f[3]);
            out[1] = make_float4(f[4], f[5], f[6], f[7]);
        }
    }
    if (!A.publish) return;
    // every thread's rows before the word the host waits for
    __threadfence_system();
    __syncthreads();
    if (tid == 0)
        asm volatile("st.release.sys.global.s32 [%0], %1;" ::"l"(A.publish + (size_t)A.V * kNF), "r"(1) : "memory");
}

// Offsets of the layers in the flat weight vector.
constexpr int oW1 = 0;
constexpr int oB1 = oW1 + kNH * kNF;
constexpr int oW2 = oB1 + kNH;
constexpr int oB2 = oW2 + kNH * kNH;
constexpr int oW3 = oB2 + kNH;
constexpr int oB3 = oW3 + kNH;

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, const float4& v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ void st2(float* p, const float2& v) { *reinterpret_cast<float2*>(p) = v; }

// acc + a . b over the four components, in order
__device__ __forceinline__ float dot4(const float4& a, const float4& b, float acc) {
    return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}

// Rows of W1 and W2 in shared memory, padded so that 8 lanes' 128-bit reads of
// consecutive rows fall into different banks.
constexpr int kRow = kNH + 4;
constexpr int kRow1 = kNF + 4;

// Scores of n rows of X: a warp takes R rows at a time, lane j holding hidden
// units j and j + 32 of both layers; the rows' layer-1 outputs go through
// shared memory and are read back as broadcast float4. A weight read serves R
// rows: with one row per warp and step the kernel was bound by shared memory
// and shuffles (55 us for 20,000 rows), with eight by the FMAs. Few rows take
// R = 1, so that they spread over more warps. Measured (one row per warp and
// step -> this): 25 rows 7.1 -> 6.2 us, 2,000 rows 10.4 -> 6.3, 20,000 rows
// 55 -> 14, 1,000,000 rows 765 -> 283 us.
template <int R>
__global__ void __launch_bounds__(256) ct_mlp_forward_kernel(const float* __restrict__ w, const float* __restrict__ X,
                                                             int n, float* __restrict__ out) {
    __shared__ __align__(16) float w1[kNH * kRow1];  // [j][i]
    __shared__ __align__(16) float w2[kNH * kRow];   // [j][i]
    __shared__ float bias1[kNH], bias2[kNH], w3[kNH];
    __shared__ __align__(16) float hid[8][R][kNH];
    for (int q = threadIdx.x; q < kNF * kNH; q += blockDim.x) w1[(q / kNF) * kRow1 + q % kNF] = w[oW1 + q];
    for (int q = threadIdx.x; q < kNH * kNH; q += blockDim.x) w2[(q / kNH) * kRow + q % kNH] = w[oW2 + q];
    for (int q = threadIdx.x; q < kNH; q += blockDim.x) {
        bias1[q] = w[oB1 + q];
        bias2[q] = w[oB2 + q];
        w3[q] = w[oW3 + q];
    }
    __syncthreads();
    const float b3 = w[oB3];
    const int lane = threadIdx.x & 31;
    float(*h)[kNH] = hid[threadIdx.x >> 5];
    const int gwarp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    const float4 wa0 = ld4(w1 + lane * kRow1), wa1 = ld4(w1 + lane * kRow1 + 4);
    const float4 wb0 = ld4(w1 + (lane + 32) * kRow1), wb1 = ld4(w1 + (lane + 32) * kRow1 + 4);
    for (long long s0 = (long long)gwarp * R; s0 < n; s0 += (long long)nwarps * R) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long s = min(s0 + r, (long long)n - 1);  // (rows beyond the last one are not stored)
            float x[kNF];
#pragma unroll
            for (int i = 0; i < kNF; ++i) x[i] = __ldg(X + s * kNF + i);
            const float4 x0 = make_float4(x[0], x[1], x[2], x[3]), x1 = make_float4(x[4], x[5], x[6], x[7]);
            h[r][lane] = fmaxf(dot4(wa1, x1, dot4(wa0, x0, bias1[lane])), 0.0f);
            h[r][lane + 32] = fmaxf(dot4(wb1, x1, dot4(wb0, x0, bias1[lane + 32])), 0.0f);
        }
        __syncwarp();
        float za[R], zb[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            za[r] = bias2[lane];
            zb[r] = bias2[lane + 32];
        }
#pragma unroll 4
        for (int i = 0; i < kNH; i += 4) {
            const float4 ua = ld4(w2 + lane * kRow + i), ub = ld4(w2 + (lane + 32) * kRow + i);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float4 hr = ld4(h[r] + i);
                za[r] = dot4(ua, hr, za[r]);
                zb[r] = dot4(ub, hr, zb[r]);
            }
        }
        __syncwarp();
        float o[R];
#pragma unroll
        for (int r = 0; r < R; ++r) o[r] = w3[lane] * fmaxf(za[r], 0.0f) + w3[lane + 32] * fmaxf(zb[r], 0.0f);
#pragma unroll
        for (int k = 16; k > 0; k >>= 1)
#pragma unroll
            for (int r = 0; r < R; ++r) o[r] += __shfl_xor_sync(0xffffffffu, o[r], k);
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (lane == r && s0 + r < n) out[s0 + r] = o[r] + b3;
    }
}

// The scores' launch: eight rows per warp once that still fills the SMs' warps
// (two CTAs of 8 warps per SM), one below.
cudaError_t launch_forward(const float* w, const float* X, int n, float* out, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (n >= 8 * 8 * sms) {
        ct_mlp_forward_kernel<8><<<std::min(n / 64 + 1, 2 * sms), 256, 0, s>>>(w, X, n, out);
    } else {
        ct_mlp_forward_kernel<1><<<std::min(n / 8 + 1, 4 * sms), 256, 0, s>>>(w, X, n, out);
    }
    return cudaGetLastError();
}

struct TrainArgs {
    float* w;             // [kNW] in/out
    float* m;             // [kNW] in/out
    float* v;             // [kNW] in/out
    const float* X;       // [n][kNF]
    const float* y;       // [n]
    const int32_t* order; // [epochs][n]
    float* epochLoss;     // [epochs]
    float* grad;          // grad-only mode: [kNW] gradient of the first batch
    int64_t t0;           // Adam steps before this launch
    int32_t n, epochs, batch;
    float lr;
    int32_t gradOnly;
};

// Training runs on one cluster of kTrainCtas CTAs. The passes over the layers
// are split by samples (CTA r takes the r-th run of the batch, a warp per two
// samples, two units per lane, so that the layers need no CTA barrier: the
// activations a warp reads are the ones it wrote, and a weight read serves both
// samples); the gradients and Adam by units (CTA r owns units 8r .. 8r + 7 of
// both layers: their rows of W1 and W2, their biases and W3 entries, with the
// moments in registers). Each warp stores what the owners need into their
// shared memory, and the owners store the new weights into everybody's: two
// cluster barriers a batch.
// Every sum runs in one thread over its inputs in order (units 0..63, samples
// 0..b-1), whatever the split: Adam divides a gradient by its own size, so one
// that cancels to rounding noise makes a full step, and another order of
// summation would make another network.
// What bounds a batch of 128 samples: the shared memory the products read, the
// chains of 64 and 128 dependent FMAs, the exchange and the barriers. Rows of
// W1 and W2 are padded so that the lanes' 128-bit reads of their units' rows
// (forward) and the consecutive reads of one row (backward) are both free of
// bank conflicts (unpadded, one of them is a 32-way conflict: one CTA took
// 115 us per batch of 128; a half-warp per sample with W2 in both orders, the
// second order's stores scattered over the cluster, 9.9 us).
constexpr int kTrainThreads = 256;
constexpr int kTrainCtas = 8;
constexpr int kTrainSamples = kTrainBatch / kTrainCtas;  // per CTA and batch
constexpr int kOwnU = kNH / kTrainCtas;                  // units a CTA owns
static_assert(kTrainSamples * 16 == kTrainThreads && kNH == 64 && kNF == 8 && kOwnU == 8,
              "a warp per two samples, two units per lane, 8 units per CTA");

struct TrainSmem {
    float w2[kNH * kRow];      // [j][i]: unit j of layer 2, input i
    float w1[kNH * kRow1];     // [j][i]
    float b1[kNH], b2[kNH], w3[kNH];
    // the whole batch, written by the CTAs that hold the samples
    float h1[kTrainBatch * kNH];    // layer-1 activations
    float x[kTrainBatch * kNF];
    float d1o[kTrainBatch * kOwnU], d2o[kTrainBatch * kOwnU], h2o[kTrainBatch * kOwnU];  // of the owned units
    float dout[kTrainBatch], sq[kTrainBatch];
    // the CTA's own samples
    float rx[kTrainSamples * kNF], r1[kTrainSamples * kNH], r2[kTrainSamples * kNH], rd[kTrainSamples * kNH];
    float gw[kOwnU * kNH];  // gradient of the owned W2 rows
    float c[2][2];  // Adam's bias corrections of a batch, by batch parity
    float b3;
};

__device__ __forceinline__ void adam(float& w, float& m, float& v, float g, float lr, float c1, float c2) {
    const float mi = 0.9f * m + 0.1f * g;
    const float vi = 0.999f * v + 0.001f * g * g;
    m = mi;
    v = vi;
    w -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

__global__ void __cluster_dims__(kTrainCtas, 1, 1) __launch_bounds__(kTrainThreads, 1)
ct_mlp_train_kernel(const TrainArgs A) {
    extern __shared__ __align__(16) unsigned char s_train[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(s_train);
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, half = lane >> 4, q = lane & 15;
    const int sl = warp * 2 + half;  // the sample in the CTA a half-warp fetches and sends
    TrainSmem* peer[kTrainCtas];
#pragma unroll
    for (int r = 0; r < kTrainCtas; ++r) peer[r] = cluster.map_shared_rank(&S, r);
    for (int e = tid; e < kNH * kNH; e += kTrainThreads) S.w2[(e / kNH) * kRow + e % kNH] = A.w[oW2 + e];
    for (int e = tid; e < kNH * kNF; e += kTrainThreads) S.w1[(e / kNF) * kRow1 + e % kNF] = A.w[oW1 + e];
    if (tid < kNH) {
        S.b1[tid] = A.w[oB1 + tid];
        S.b2[tid] = A.w[oB2 + tid];
        S.w3[tid] = A.w[oW3 + tid];
    }
    if (tid == 0) {
        S.b3 = A.w[oB3];
        S.c[0][0] = 1.0f - powf(0.9f, (float)(A.t0 + 1));
        S.c[0][1] = 1.0f - powf(0.999f, (float)(A.t0 + 1));
    }
    for (int e = tid; e < kTrainBatch; e += kTrainThreads) S.sq[e] = 0.0f;
    // The entries a thread owns: inputs 2 * lane, 2 * lane + 1 of the W2 row of
    // owned unit `warp` (0, 1), and one more (2) in warps 4, 5 (a W1 entry per
    // lane) and 6 (b1, b2, W3 of the owned units, 8 lanes each; b3 in CTA 0).
    // (All of Adam on the two warps that sum the W2 gradients, 8 entries a
    // thread, made 11,400 of a batch's 20,700 cycles: its divisions follow one
    // another.)
    const int uj = warp < 6 ? (tid & 63) / kNF : lane & 7;  // the extra entry's owned unit and input
    const int unit = rank * kOwnU + uj, ui = lane % kNF;
    const bool extra = warp == 4 || warp == 5 || (warp == 6 && (lane < 24 || (lane == 24 && rank == 0)));
    const int ex = warp < 6 ? oW1 + unit * kNF + ui
                   : lane < 8 ? oB1 + unit
                   : lane < 16 ? oB2 + unit
                   : lane < 24 ? oW3 + unit : oB3;
    auto entry = [&](int k) { return k < 2 ? oW2 + (rank * kOwnU + warp) * kNH + 2 * lane + k : ex; };
    float w[3], m[3], v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const bool own = k < 2 || extra;
        w[k] = own ? A.w[entry(k)] : 0.0f;
        m[k] = own ? A.m[entry(k)] : 0.0f;
        v[k] = own ? A.v[entry(k)] : 0.0f;
    }
    const int epochs = A.gradOnly ? 1 : A.epochs;
    const int nUse = A.gradOnly ? min(A.n, A.batch) : A.n;
    const int nb = (nUse + A.batch - 1) / A.batch;
    const long long total = (long long)nb * epochs;
    // a batch's size, the samples per CTA, and the half-warp's sample (-1: none)
    auto sample_of = [&](int ep, int pos, int& b, int& per) -> int {
        const int s0 = pos * A.batch;
        b = min(A.batch, nUse - s0);
        per = (b + kTrainCtas - 1) / kTrainCtas;
        const int i = rank * per + sl;
        if (sl >= per || i >= b) return -1;
        return __ldg(A.order + (size_t)ep * A.n + s0 + i);
    };
    // the samples are fetched one batch ahead, their indices two
    int b = 0, per = 0, bN = 0, perN = 0, ep2 = 0, pos2 = 0;
    auto advance = [&]() {
        if (++pos2 == nb) {
            pos2 = 0;
            ++ep2;
        }
    };
    float xv = 0.0f, yv = 0.0f;
    bool valid = false;
    int idxN = -1;
    {
        const int i0 = sample_of(0, 0, b, per);
        valid = i0 >= 0;
        if (valid) {
            if (q < kNF) xv = __ldg(A.X + (size_t)i0 * kNF + q);
            yv = __ldg(A.y + i0);
        }
        advance();
        if (total > 1) idxN = sample_of(ep2, pos2, bN, perN);
    }
    cluster.sync();  // every CTA runs: its shared memory may be written
    float lossSum = 0.0f;  // CTA 0, last warp
    int pos = 0, ep = 0;
    for (long long kb = 0; kb < total; ++kb) {
        // next batch's sample, and the one after's index
        float xN = 0.0f, yN = 0.0f;
        const bool validN = kb + 1 < total && idxN >= 0;
        if (validN) {
            if (q < kNF) xN = __ldg(A.X + (size_t)idxN * kNF + q);
            yN = __ldg(A.y + idxN);
        }
        int b2n = 0, per2n = 0, idx2 = -1;
        advance();
        if (kb + 2 < total) idx2 = sample_of(ep2, pos2, b2n, per2n);
        if (warp * 2 < per) {
            const int sg = valid ? rank * per + sl : 0;  // the half-warp's sample in the batch
            float* x0 = S.rx + warp * 2 * kNF;           // the warp's two samples: rows 0 and 1
            float* h0 = S.r1 + warp * 2 * kNH;
            float* z0 = S.r2 + warp * 2 * kNH;
            float* d0 = S.rd + warp * 2 * kNH;
            if (q < kNF) x0[half * kNF + q] = xv;
            __syncwarp();
            // layer 1: units lane and lane + 32 of both samples
            float a[2][2];  // [unit][sample]
            {
                const float4 xa = ld4(x0), xb = ld4(x0 + 4), xc = ld4(x0 + 8), xd = ld4(x0 + 12);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int j = lane + 32 * u;
                    const float4 wa = ld4(S.w1 + j * kRow1), wb = ld4(S.w1 + j * kRow1 + 4);
                    a[u][0] = fmaxf(dot4(wb, xb, dot4(wa, xa, S.b1[j])), 0.0f);
                    a[u][1] = fmaxf(dot4(wb, xd, dot4(wa, xc, S.b1[j])), 0.0f);
                    h0[j] = a[u][0];
                    h0[kNH + j] = a[u][1];
                }
            }
            __syncwarp();
            // layer 2
            float z[2][2];
            z[0][0] = z[0][1] = S.b2[lane];
            z[1][0] = z[1][1] = S.b2[lane + 32];
#pragma unroll 8
            for (int i = 0; i < kNH; i += 4) {
                const float4 ha = ld4(h0 + i), hb = ld4(h0 + kNH + i);
                const float4 wa = ld4(S.w2 + lane * kRow + i), wb = ld4(S.w2 + (lane + 32) * kRow + i);
                z[0][0] = dot4(wa, ha, z[0][0]);
                z[0][1] = dot4(wa, hb, z[0][1]);
                z[1][0] = dot4(wb, ha, z[1][0]);
                z[1][1] = dot4(wb, hb, z[1][1]);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    z[u][t] = fmaxf(z[u][t], 0.0f);
                    z0[t * kNH + lane + 32 * u] = z[u][t];
                }
            __syncwarp();
            // the outputs, units in order: lanes 0 and 16 a sample each
            float o = S.b3;
            if (q == 0) {
#pragma unroll
                for (int j = 0; j < kNH; j += 4) o = dot4(ld4(S.w3 + j), ld4(z0 + half * kNH + j), o);
            }
            const float r = __shfl_sync(0xffffffffu, o, half << 4) - yv, dz = r / (float)b;
            const float dz0 = __shfl_sync(0xffffffffu, dz, 0), dz1 = __shfl_sync(0xffffffffu, dz, 16);
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int j = lane + 32 * u;
                const float c = S.w3[j];
                d0[j] = z[u][0] > 0.0f ? dz0 * c : 0.0f;
                d0[kNH + j] = z[u][1] > 0.0f ? dz1 * c : 0.0f;
            }
            __syncwarp();
            // dL/dz1 of inputs 2 * lane, 2 * lane + 1
            float2 ga = make_float2(0.0f, 0.0f), gb = ga;
#pragma unroll 8
            for (int j = 0; j < kNH; j += 4) {
                const float4 da = ld4(d0 + j), db = ld4(d0 + kNH + j);
                const float fa[4] = {da.x, da.y, da.z, da.w}, fb[4] = {db.x, db.y, db.z, db.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float2 ww = ld2(S.w2 + (j + k) * kRow + 2 * lane);
                    ga.x = fmaf(fa[k], ww.x, ga.x);
                    ga.y = fmaf(fa[k], ww.y, ga.y);
                    gb.x = fmaf(fb[k], ww.x, gb.x);
                    gb.y = fmaf(fb[k], ww.y, gb.y);
                }
            }
            const float4 hs = ld4(h0 + half * kNH + 4 * q), zs = ld4(z0 + half * kNH + 4 * q),
                         ds = ld4(d0 + half * kNH + 4 * q);
            const float2 ha = ld2(h0 + 2 * lane), hb = ld2(h0 + kNH + 2 * lane);
            __syncwarp();  // (dL/dz2 is read: its rows take dL/dz1)
            st2(d0 + 2 * lane, make_float2(ha.x > 0.0f ? ga.x : 0.0f, ha.y > 0.0f ? ga.y : 0.0f));
            st2(d0 + kNH + 2 * lane, make_float2(hb.x > 0.0f ? gb.x : 0.0f, hb.y > 0.0f ? gb.y : 0.0f));
            __syncwarp();
            if (valid) {
                // to every CTA: layer 1, the inputs, dL/dout; to a unit's owner: its activation and gradients
#pragma unroll
                for (int p = 0; p < kTrainCtas; ++p) {
                    st4(peer[p]->h1 + sg * kNH + 4 * q, hs);
                    if (q < kNF) peer[p]->x[sg * kNF + q] = xv;
                    if (q == 0) peer[p]->dout[sg] = dz;
                }
                TrainSmem* own = cluster.map_shared_rank(&S, q >> 1);
                const int at = sg * kOwnU + 4 * (q & 1);
                st4(own->d1o + at, ld4(d0 + half * kNH + 4 * q));
                st4(own->d2o + at, ds);
                st4(own->h2o + at, zs);
                if (q == 0) peer[0]->sq[sg] = r * r;
            }
        }
        cluster.sync();
        // the owned entries: gradient over the batch (samples in order), Adam
        const float c1 = S.c[kb & 1][0], c2 = S.c[kb & 1][1];
        float ge = 0.0f;
        if (warp < 4) {
            // two owned W2 rows, two inputs per lane
            float g[2][2] = {};
#pragma unroll 16
            for (int s = 0; s < b; ++s) {
                const float2 d = ld2(S.d2o + s * kOwnU + 2 * warp);
                const float2 h = ld2(S.h1 + s * kNH + 2 * lane);
                g[0][0] = fmaf(d.x, h.x, g[0][0]);
                g[0][1] = fmaf(d.x, h.y, g[0][1]);
                g[1][0] = fmaf(d.y, h.x, g[1][0]);
                g[1][1] = fmaf(d.y, h.y, g[1][1]);
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) st2(S.gw + (2 * warp + k) * kNH + 2 * lane, make_float2(g[k][0], g[k][1]));
        } else if (warp < 6) {
#pragma unroll 16
            for (int s = 0; s < b; ++s) ge = fmaf(S.d1o[s * kOwnU + uj], S.x[s * kNF + ui], ge);
        } else if (warp == 6) {
            // b1, b2: sums of the units' gradients; W3: of dL/dout times the activation; b3: of dL/dout
            const float* f = lane < 8 ? S.d1o + uj : lane < 16 ? S.d2o + uj : lane < 24 ? S.h2o + uj : S.dout;
            const int step = lane < 24 ? kOwnU : 1;
            const bool times = lane >= 16 && lane < 24;
#pragma unroll 16
            for (int s = 0; s < b; ++s) ge = fmaf(times ? S.dout[s] : 1.0f, f[s * step], ge);
        } else if (warp == kTrainThreads / 32 - 1) {
            // the batch's loss (CTA 0, a binary tree over the samples), the next batch's bias corrections
            if (rank == 0) {
                float l = (S.sq[lane] + S.sq[lane + 64]) + (S.sq[lane + 32] + S.sq[lane + 96]);
                __syncwarp();
                for (int k = 0; k < kTrainBatch; k += 32) S.sq[lane + k] = 0.0f;
#pragma unroll
                for (int k = 16; k > 0; k >>= 1) l += __shfl_down_sync(0xffffffffu, l, k);
                if (lane == 0) {
                    lossSum += l / (2.0f * (float)b);
                    if (pos + 1 == nb) {
                        A.epochLoss[ep] = lossSum / (float)nb;
                        lossSum = 0.0f;
                    }
                }
            }
            if (lane < 2) {
                const float t = (float)(A.t0 + kb + 2);
                S.c[(kb + 1) & 1][lane] = 1.0f - powf(lane == 0 ? 0.9f : 0.999f, t);
            }
        }
        __syncthreads();
        const float2 gw = ld2(S.gw + warp * kNH + 2 * lane);
        if (A.gradOnly) {
            A.grad[entry(0)] = gw.x;
            A.grad[entry(1)] = gw.y;
            if (extra) A.grad[ex] = ge;
        } else {
            adam(w[0], m[0], v[0], gw.x, A.lr, c1, c2);
            adam(w[1], m[1], v[1], gw.y, A.lr, c1, c2);
#pragma unroll
            for (int p = 0; p < kTrainCtas; ++p)
                st2(peer[p]->w2 + (rank * kOwnU + warp) * kRow + 2 * lane, make_float2(w[0], w[1]));
            if (extra) {
                adam(w[2], m[2], v[2], ge, A.lr, c1, c2);
#pragma unroll
                for (int p = 0; p < kTrainCtas; ++p) {
                    TrainSmem* P = peer[p];
                    float* at = warp < 6 ? &P->w1[unit * kRow1 + ui]
                                : lane < 8 ? &P->b1[unit]
                                : lane < 16 ? &P->b2[unit]
                                : lane < 24 ? &P->w3[unit] : &P->b3;
                    *at = w[2];
                }
            }
        }
        cluster.sync();
        xv = xN;
        yv = yN;
        valid = validN;
        idxN = idx2;
        b = bN;
        per = perN;
        bN = b2n;
        perN = per2n;
        if (++pos == nb) {
            pos = 0;
            ++ep;
        }
    }
    if (A.gradOnly) return;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        if (k < 2 || extra) {
            A.w[entry(k)] = w[k];
            A.m[entry(k)] = m[k];
            A.v[entry(k)] = v[k];
        }
    }
}

template <typename T>
int f_alloc(FeatView* f, T** p, size_t n) {
    void* q = nullptr;
    const cudaError_t e = cudaMalloc(&q, std::max<size_t>(n, 1) * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        ct_set_error("features: cudaMalloc: %s", cudaGetErrorString(e));
        return CT_ERR_OOM;
    }
    f->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return CT_OK;
}

template <typename T>
int f_upload(T* dst, const std::vector<T>& src) {
    if (src.empty()) return CT_OK;
    CT_CUDA(cudaMemcpy(dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice));
    return CT_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
// feature view
// ---------------------------------------------------------------------------
int ct_feat_view_build(FeatView* f, int nodes, const std::vector<std::vector<int>>& scopes,
                       const std::vector<int>& tableR, const std::vector<int>& tableSeg,
                       const std::vector<int32_t>& varOff, const std::vector<int32_t>& varNW,
                       const std::vector<int32_t>& varD0, int DWg) {
    const int T = (int)scopes.size();
    const int V = (int)varOff.size();
    const int nt = nodes * T, nv = nodes * V;
    f->nodes = nodes;
    f->T = T;
    f->V = V;
    f->nt = nt;
    f->nv = nv;
    std::vector<int32_t> rowBase(nt + 1, 0), unitBase(nt + 1, 0), scopeBase(nt + 1, 0), scopeOff, vOff(nv), vNW(nv),
        vD0(nv), deg(nv, 0), adjBase(nv + 1, 0);
    std::vector<int2> adj;
    std::vector<std::vector<int2>> perVar(V);
    for (int k = 0; k < T; ++k)
        for (int i = 0; i < (int)scopes[k].size(); ++i) perVar[scopes[k][i]].push_back(make_int2(k, i));
    int degmax = 1;
    for (int v = 0; v < V; ++v) degmax = std::max(degmax, (int)perVar[v].size());
    for (int n = 0; n < nodes; ++n) {
        for (int k = 0; k < T; ++k) {
            const int t = n * T + k;
            rowBase[t + 1] = rowBase[t] + tableR[k];
            int sw = 0;
            for (int v : scopes[k]) sw += varNW[v];
            unitBase[t + 1] = unitBase[t] + tableSeg[k] * sw;
            scopeBase[t + 1] = scopeBase[t] + (int)scopes[k].size();
            for (int v : scopes[k]) scopeOff.push_back(varOff[v] + n * DWg);
        }
        for (int v = 0; v < V; ++v) {
            const int g = n * V + v;
            vOff[g] = varOff[v] + n * DWg;
            vNW[g] = varNW[v];
            vD0[g] = varD0[v];
            deg[g] = (int)perVar[v].size();
            for (const int2& e : perVar[v]) adj.push_back(make_int2(n * T + e.x, e.y));
            adjBase[g + 1] = (int)adj.size();
        }
    }
    f->pairs = nodes > 0 ? (int)adj.size() / nodes : 0;
    f->small = f->pairs > 0 && V <= kFeatVars;
    for (int k = 0; k < T; ++k) {
        const int chunks = tableSeg[k] * 32;
        for (int v : scopes[k])
            f->small = f->small && chunks <= kFeatChunks && varNW[v] <= kFeatValues / 32 &&
                       varNW[v] * 32 * chunks <= kFeatTests;
    }
    std::vector<int32_t> pairVar(adj.size());
    for (int v = 0; v < nv; ++v) std::fill(pairVar.begin() + adjBase[v], pairVar.begin() + adjBase[v + 1], v);
    f->degmax = degmax;
    f->totalUnits = unitBase[nt];
    const int64_t entries = (int64_t)nodes * f->pairs;
    f->small = f->small && (nodes == 1 || V <= kFeatNodeVars || entries <= kFeatEntries || f->totalUnits >= 3 * entries);
    f->totalRows = rowBase[nt];
    int st;
    if ((st = f_alloc(f, &f->rowBase, nt + 1)) != CT_OK || (st = f_alloc(f, &f->unitBase, nt + 1)) != CT_OK ||
        (st = f_alloc(f, &f->scopeBase, nt + 1)) != CT_OK || (st = f_alloc(f, &f->scopeOff, scopeOff.size())) != CT_OK ||
        (st = f_alloc(f, &f->adjBase, nv + 1)) != CT_OK || (st = f_alloc(f, &f->adj, adj.size())) != CT_OK ||
        (st = f_alloc(f, &f->varOff, nv)) != CT_OK || (st = f_alloc(f, &f->varNW, nv)) != CT_OK ||
        (st = f_alloc(f, &f->varD0, nv)) != CT_OK || (st = f_alloc(f, &f->deg, nv)) != CT_OK ||
        (st = f_alloc(f, &f->pairVar, pairVar.size())) != CT_OK ||
        (st = f_alloc(f, &f->pairStat, pairVar.size())) != CT_OK || (st = f_alloc(f, &f->ticket, nodes)) != CT_OK ||
        (st = f_alloc(f, &f->counts, rowBase[nt])) != CT_OK || (st = f_alloc(f, &f->live, nt)) != CT_OK ||
        (st = f_alloc(f, &f->feat, (size_t)nv * kNF)) != CT_OK || (st = f_alloc(f, &f->scores, nv)) != CT_OK)
        return st;
    if ((st = f_upload(f->rowBase, rowBase)) != CT_OK || (st = f_upload(f->unitBase, unitBase)) != CT_OK ||
        (st = f_upload(f->scopeBase, scopeBase)) != CT_OK || (st = f_upload(f->scopeOff, scopeOff)) != CT_OK ||
        (st = f_upload(f->adjBase, adjBase)) != CT_OK || (st = f_upload(f->adj, adj)) != CT_OK ||
        (st = f_upload(f->varOff, vOff)) != CT_OK || (st = f_upload(f->varNW, vNW)) != CT_OK ||
        (st = f_upload(f->varD0, vD0)) != CT_OK || (st = f_upload(f->deg, deg)) != CT_OK ||
        (st = f_upload(f->pairVar, pairVar)) != CT_OK)
        return st;
    CT_CUDA(cudaMemset(f->ticket, 0, (size_t)std::max(nodes, 1) * sizeof(unsigned)));
    const size_t nscores = (size_t)(std::max(nv, 1) + 3) & ~(size_t)3;  // (the features on a 16-byte boundary)
    const bool publish = f->small && nodes == 1;
    if (cudaHostAlloc((void**)&f->h_scores, (nscores + (publish ? (size_t)nv * kNF + 1 : 0)) * sizeof(float),
                      publish ? cudaHostAllocMapped : cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        f->h_scores = nullptr;
        ct_set_error("features: pinned scores");
        return CT_ERR_OOM;
    }
    if (publish) {
        f->h_feat = f->h_scores + nscores;
        CT_CUDA(cudaHostGetDevicePointer((void**)&f->d_hfeat, f->h_feat, 0));
    }
    return CT_OK;
}

void ct_feat_view_free(FeatView* f) {
    if (!f) return;
    for (void* p : f->allocs) cudaFree(p);
    f->allocs.clear();
    if (f->h_scores) cudaFreeHost(f->h_scores);
    f->h_scores = f->h_feat = f->d_hfeat = nullptr;
    cudaGetLastError();
}

int ct_feat_compute(FeatView* f, const TableDev* d_tabs, const uint32_t* dom, const uint8_t* nodeActive,
                    cudaStream_t s, bool publish) {
    if (!f->counts) {
        ct_set_error("features: view not built");
        return CT_ERR_STATE;
    }
    FeatArgs A;
    A.tabs = d_tabs;
    A.dom = dom;
    A.nodeActive = nodeActive;
    A.rowBase = f->rowBase;
    A.unitBase = f->unitBase;
    A.scopeBase = f->scopeBase;
    A.scopeOff = f->scopeOff;
    A.adjBase = f->adjBase;
    A.adj = f->adj;
    A.varOff = f->varOff;
    A.varNW = f->varNW;
    A.varD0 = f->varD0;
    A.deg = f->deg;
    A.counts = f->counts;
    A.live = f->live;
    A.feat = f->feat;
    A.nt = f->nt;
    A.nv = f->nv;
    A.T = f->T;
    A.V = f->V;
    A.degmax = f->degmax;
    A.totalUnits = f->totalUnits;
    A.pairVar = f->pairVar;
    A.pairStat = f->pairStat;
    A.ticket = f->ticket;
    A.pairs = f->pairs;
    A.publish = publish ? f->d_hfeat : nullptr;
    if (f->small) {
        ct_features_small_kernel<<<f->nodes * f->pairs, kFeatThreads, 0, s>>>(A);
        CT_CUDA(cudaGetLastError());
        return CT_OK;
    }
    CT_CUDA(cudaMemsetAsync(f->counts, 0, sizeof(uint32_t) * (size_t)std::max(f->totalRows, 1), s));
    CT_CUDA(cudaMemsetAsync(f->live, 0, sizeof(uint32_t) * (size_t)std::max(f->nt, 1), s));
    int sms = 0, dev = 0;
    CT_CUDA(cudaGetDevice(&dev));
    CT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const int warps = std::max(1, f->totalUnits);
    const int grid = std::max(1, std::min((warps + 7) / 8, sms * 8));
    if (f->totalUnits > 0) {
        ct_counts_kernel<<<grid, 256, 0, s>>>(A);
        CT_CUDA(cudaGetLastError());
    }
    const int perNode = (f->V + 7) / 8;
    ct_features_kernel<<<f->nodes * std::max(perNode, 1), 256, 0, s>>>(A, std::max(perNode, 1));
    CT_CUDA(cudaGetLastError());
    return CT_OK;
}

int ct_feat_scores(FeatView* f, const ct_mlp* mlp, cudaStream_t s) {
    const int n = f->nv;
    CT_CUDA(launch_forward(mlp->d_w, f->feat, n, f->scores, s));
    CT_CUDA(cudaMemcpyAsync(f->h_scores, f->scores, (size_t)n * sizeof(float), cudaMemcpyDeviceToHost, s));
    CT_CUDA(cudaStreamSynchronize(s));
    return CT_OK;
}

// ---------------------------------------------------------------------------
// C ABI: the scoring network
// ---------------------------------------------------------------------------
namespace {

int mlp_reset(ct_mlp* m, const float* w_host) {
    CT_CUDA(cudaMemcpyAsync(m->d_w, w_host, kNW * sizeof(float), cudaMemcpyHostToDevice, m->stream));
    CT_CUDA(cudaMemsetAsync(m->d_m, 0, kNW * sizeof(float), m->stream));
    CT_CUDA(cudaMemsetAsync(m->d_v, 0, kNW * sizeof(float), m->stream));
    CT_CUDA(cudaStreamSynchronize(m->stream));
    m->t = 0;
    return CT_OK;
}

// Device copies of a host array (freed by the caller with cudaFree).
template <typename T>
int to_device(const T* h, size_t n, T** d, cudaStream_t s) {
    *d = nullptr;
    cudaError_t e = cudaMalloc((void**)d, std::max<size_t>(n, 1) * sizeof(T));
    if (e == cudaSuccess && n) e = cudaMemcpyAsync(*d, h, n * sizeof(T), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
        if (*d) cudaFree(*d);
        *d = nullptr;
        return ct_cuda_fail(e, "training data upload");
    }
    return CT_OK;
}

int run_train(ct_mlp* m, const float* x_host, const float* y_host, int64_t n, const int32_t* orders, int epochs,
              int batch, float lr, bool gradOnly, float* loss_out, float* grad_host) {
    float *dX = nullptr, *dY = nullptr, *dLoss = nullptr, *dGrad = nullptr;
    int32_t* dOrd = nullptr;
    std::vector<int32_t> ident;
    if (gradOnly) {
        ident.resize((size_t)n);
        for (int64_t i = 0; i < n; ++i) ident[(size_t)i] = (int32_t)i;
        orders = ident.data();
    }
    int st = to_device(x_host, (size_t)n * kNF, &dX, m->stream);
    if (st == CT_OK) st = to_device(y_host, (size_t)n, &dY, m->stream);
    if (st == CT_OK) st = to_device(orders, (size_t)n * (gradOnly ? 1 : epochs), &dOrd, m->stream);
    cudaError_t e = cudaSuccess;
    if (st == CT_OK) {
        e = cudaMalloc((void**)&dLoss, sizeof(float) * (size_t)std::max(epochs, 1));
        if (e == cudaSuccess) e = cudaMalloc((void**)&dGrad, sizeof(float) * kNW);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(ct_mlp_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
        if (e == cudaSuccess) {
            TrainArgs A;
            A.w = m->d_w;
            A.m = m->d_m;
            A.v = m->d_v;
            A.X = dX;
            A.y = dY;
            A.order = dOrd;
            A.epochLoss = dLoss;
            A.grad = dGrad;
            A.t0 = m->t;
            A.n = (int32_t)n;
            A.epochs = gradOnly ? 1 : epochs;
            A.batch = batch;
            A.lr = lr;
            A.gradOnly = gradOnly ? 1 : 0;
            ct_mlp_train_kernel<<<kTrainCtas, kTrainThreads, sizeof(TrainSmem), m->stream>>>(A);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess && loss_out)
            e = cudaMemcpyAsync(loss_out, dLoss, sizeof(float) * (size_t)(gradOnly ? 1 : epochs), cudaMemcpyDeviceToHost,
                                m->stream);
        if (e == cudaSuccess && gradOnly && grad_host)
            e = cudaMemcpyAsync(grad_host, dGrad, sizeof(float) * kNW, cudaMemcpyDeviceToHost, m->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
        if (e != cudaSuccess) st = ct_cuda_fail(e, "ct_mlp training kernel");
    }
    if (dX) cudaFree(dX);
    if (dY) cudaFree(dY);
    if (dOrd) cudaFree(dOrd);
    if (dLoss) cudaFree(dLoss);
    if (dGrad) cudaFree(dGrad);
    if (st == CT_OK && !gradOnly) {
        const int64_t per = (n + batch - 1) / batch;
        m->t += per * epochs;
    }
    return st;
}

}  // namespace

extern "C" int ct_mlp_create(const float* weights_host, void* cuda_stream, ct_mlp** out) {
    if (!out || !weights_host) {
        ct_set_error("ct_mlp_create: null argument");
        return CT_ERR_ARG;
    }
    *out = nullptr;
    ct_mlp* m = new (std::nothrow) ct_mlp();
    if (!m) return CT_ERR_OOM;
    cudaError_t e = cudaSuccess;
    if (cuda_stream) {
        m->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        e = cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking);
        m->ownStream = e == cudaSuccess;
    }
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->d_w, kNW * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->d_m, kNW * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc((void**)&m->d_v, kNW * sizeof(float));
    int st = e == cudaSuccess ? mlp_reset(m, weights_host) : ct_cuda_fail(e, "ct_mlp_create");
    if (st != CT_OK) {
        ct_mlp_destroy(m);
        return st;
    }
    *out = m;
    return CT_OK;
}

extern "C" int ct_mlp_set_weights(ct_mlp* m, const float* weights_host) {
    if (!m || !weights_host) {
        ct_set_error("ct_mlp_set_weights: null argument");
        return CT_ERR_ARG;
    }
    return mlp_reset(m, weights_host);
}

extern "C" int ct_mlp_get_weights(ct_mlp* m, float* weights_host) {
    if (!m || !weights_host) {
        ct_set_error("ct_mlp_get_weights: null argument");
        return CT_ERR_ARG;
    }
    CT_CUDA(cudaMemcpyAsync(weights_host, m->d_w, kNW * sizeof(float), cudaMemcpyDeviceToHost, m->stream));
    CT_CUDA(cudaStreamSynchronize(m->stream));
    return CT_OK;
}

extern "C" int ct_mlp_forward(ct_mlp* m, const float* x_dev, int64_t n, float* scores_dev) {
    if (!m || (n > 0 && (!x_dev || !scores_dev)) || n < 0 || n > 0x7fffffffLL) {
        ct_set_error("ct_mlp_forward: bad argument");
        return CT_ERR_ARG;
    }
    if (n == 0) return CT_OK;
    CT_CUDA(launch_forward(m->d_w, x_dev, (int)n, scores_dev, m->stream));
    return CT_OK;
}

extern "C" int ct_mlp_grad(ct_mlp* m, const float* x_host, const float* y_host, int n, float* loss_out,
                           float* grad_host) {
    if (!m || !x_host || !y_host || !grad_host || n < 1 || n > kTrainBatch) {
        ct_set_error("ct_mlp_grad: bad argument (1 <= n <= %d)", kTrainBatch);
        return CT_ERR_ARG;
    }
    return run_train(m, x_host, y_host, n, nullptr, 1, n, 0.0f, true, loss_out, grad_host);
}

extern "C" int ct_mlp_train(ct_mlp* m, const float* x_host, const float* y_host, int64_t n, const int32_t* orders_host,
                            int epochs, int batch, float lr, float* epoch_loss_host) {
    if (!m || !x_host || !y_host || !orders_host || n < 1 || n > 0x7fffffffLL || epochs < 1 || batch < 1 ||
        batch > kTrainBatch || !(lr > 0.0f)) {
        ct_set_error("ct_mlp_train: bad argument (1 <= batch <= %d, epochs >= 1, lr > 0)", kTrainBatch);
        return CT_ERR_ARG;
    }
    for (int64_t i = 0; i < n * epochs; ++i) {
        if (orders_host[i] < 0 || orders_host[i] >= n) {
            ct_set_error("ct_mlp_train: order entry %lld out of range", (long long)i);
            return CT_ERR_ARG;
        }
    }
    return run_train(m, x_host, y_host, n, orders_host, epochs, batch, lr, false, epoch_loss_host, nullptr);
}

extern "C" int ct_mlp_destroy(ct_mlp* m) {
    if (!m) return CT_OK;
    if (m->stream) cudaStreamSynchronize(m->stream);
    if (m->d_w) cudaFree(m->d_w);
    if (m->d_m) cudaFree(m->d_m);
    if (m->d_v) cudaFree(m->d_v);
    if (m->ownStream && m->stream) cudaStreamDestroy(m->stream);
    cudaGetLastError();
    delete m;
    return CT_OK;
}
