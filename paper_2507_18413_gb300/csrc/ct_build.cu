// ct_build.cu -- kernels that build a table's device state from its tuple list
// (the constructor of class Table, Sec. 3): the check of the tuples against
// the initial domains, the supports rows (Sec. 2, Table 1(b)), currTable with
// its non-zero index, and each row's first residue.
//
// What bounds it: the rows are written once (R * t / 8 bytes) and the tuple
// list is read from device memory. A block holds a tile of 1,024 tuples (32
// words, one 128-byte line per row) of one variable in shared memory, sets a
// bit per tuple there and writes whole lines, zeros included, so no row is
// cleared first and no global atomic is used. (On the host, a word at a time
// through rows of t / 8 bytes, the construction of 1,000,000 tuples over six
// variables of 32 values took 13 ms with its upload of 24 MB of rows; the
// kernels and the tuples' copy take 0.3 ms.)
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "ct_internal.cuh"

namespace ctk {
namespace {

constexpr int kTileWords = 32;               // words per tile: one 128-byte line of a row
constexpr int kTileRow = kTileWords + 1;     // padded: the rows of one word fall into different banks
constexpr int kTileRows = 360;               // rows of a variable held at once (47.5 KB)

// Tuples with a component outside its initial domain (counts[0]), and of the
// others those with a wildcard (counts[1]).
__global__ void ct_check_tuples_kernel(const int32_t* __restrict__ tup, long long t, int n,
                                       const int32_t* __restrict__ lo, const int32_t* __restrict__ row0,
                                       unsigned long long* counts) {
    const long long nth = (long long)gridDim.x * blockDim.x;
    unsigned bad = 0u, shortTup = 0u;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < t; j += nth) {
        bool ok = true, star = false;
        for (int i = 0; i < n; ++i) {
            const int32_t v = tup[j * n + i];
            if (v == CT_STAR) {
                star = true;
                continue;
            }
            const long long off = (long long)v - lo[i];
            ok = ok && off >= 0 && off < row0[i + 1] - row0[i];
        }
        bad += !ok;
        shortTup += ok && star;
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    shortTup = __reduce_add_sync(0xffffffffu, shortTup);
    if ((threadIdx.x & 31) == 0) {
        if (bad) atomicAdd(&counts[0], (unsigned long long)bad);
        if (shortTup) atomicAdd(&counts[1], (unsigned long long)shortTup);
    }
}

// Rows of the variables blockIdx.y, blockIdx.y + gridDim.y, ... on the tile of
// words [word0 + 32 * blockIdx.x, + 32): bit j of row (i, v) is set for tuple
// tupleBase + j with value v, or a wildcard (sup only; del, when given, holds the
// tuples with the value itself). tup holds the tuples from tupleBase on.
__global__ void __launch_bounds__(256) ct_build_rows_kernel(const int32_t* __restrict__ tup, long long tuples, int n,
                                                            const int32_t* __restrict__ lo,
                                                            const int32_t* __restrict__ row0, uint32_t* sup,
                                                            uint32_t* del, long long rowWords, long long word0) {
    __shared__ uint32_t tile[kTileRows * kTileRow];
    __shared__ uint32_t star[kTileWords];
    const int tid = threadIdx.x;
    const long long j0 = (long long)blockIdx.x * (kTileWords * 32);
    const long long w0 = word0 + (long long)blockIdx.x * kTileWords;
    for (int i = blockIdx.y; i < n; i += gridDim.y) {
        const int r0 = row0[i], d = row0[i + 1] - r0;
        const int32_t base = lo[i];
        for (int p0 = 0; p0 < d; p0 += kTileRows) {
            const int rows = min(kTileRows, d - p0);
            for (int q = tid; q < rows * kTileRow; q += 256) tile[q] = 0u;
            if (tid < kTileWords) star[tid] = 0u;
            __syncthreads();
#pragma unroll
            for (int k = tid; k < kTileWords * 32; k += 256) {
                if (j0 + k < tuples) {
                    const int32_t v = tup[(j0 + k) * n + i];
                    const uint32_t bit = 1u << (k & 31);
                    const long long a = (long long)v - base - p0;
                    if (v == CT_STAR) atomicOr(&star[k >> 5], bit);
                    else if (a >= 0 && a < rows) atomicOr(&tile[(int)a * kTileRow + (k >> 5)], bit);
                }
            }
            __syncthreads();
            const int w = tid & (kTileWords - 1);
            if (w0 + w < rowWords) {
                for (int r = tid / kTileWords; r < rows; r += 256 / kTileWords) {
                    const uint32_t v = tile[r * kTileRow + w];
                    const size_t at = (size_t)(r0 + p0 + r) * rowWords + w0 + w;
                    sup[at] = v | star[w];
                    if (del) del[at] = v;
                }
            }
            __syncthreads();
        }
    }
}

// currTable with every retained tuple valid, padded to whole segments, the
// empty trail links, and the non-zero index (every chunk below W4 holds a tuple).
__global__ void ct_build_state_kernel(const TableDev T, long long t) {
    const long long nth = (long long)gridDim.x * blockDim.x, id = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    for (long long c = id; c < (long long)T.nseg * 32; c += nth) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const long long left = t - (c * 4 + k) * 32;
            w[k] = left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u;
        }
        T.curr[c] = make_uint4(w[0], w[1], w[2], w[3]);
        T.lastpos[c] = -1;
    }
    for (long long s = id; s < T.nseg; s += nth) {
        const long long left = T.W4 - s * 32;
        T.segMask[s] = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
    }
}

// First chunk of each row that holds a tuple (0 for a row without one), a warp per row.
__global__ void ct_build_residue_kernel(const TableDev T) {
    const int lane = threadIdx.x & 31;
    const int nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int r = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); r < T.R; r += nwarps) {
        const uint4* row = T.sup + (size_t)r * T.W4;
        int found = 0;
        for (int c0 = 0; c0 < T.W4; c0 += 128) {
            unsigned any[4];
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 32 * u + lane;
                v[u] = c < T.W4 ? row[c] : make_uint4(0u, 0u, 0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) any[u] = __ballot_sync(0xffffffffu, (v[u].x | v[u].y | v[u].z | v[u].w) != 0u);
            int at = -1;
#pragma unroll
            for (int u = 3; u >= 0; --u)
                if (any[u]) at = c0 + 32 * u + __ffs(any[u]) - 1;
            if (at >= 0) {
                found = at;
                break;
            }
        }
        if (lane == 0) T.residue[r] = found;
    }
}

int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
        return 1;
    return sms;
}

}  // namespace

cudaError_t launch_check_tuples(const int32_t* tup, int64_t t, int n, const int32_t* lo, const int32_t* row0,
                                unsigned long long* counts, cudaStream_t s) {
    const int grid = (int)std::min<int64_t>((t + 255) / 256, 8LL * sm_count());
    ct_check_tuples_kernel<<<std::max(grid, 1), 256, 0, s>>>(tup, t, n, lo, row0, counts);
    return cudaGetLastError();
}

cudaError_t launch_build_rows(const int32_t* tup, int64_t tuples, int n, const int32_t* lo, const int32_t* row0,
                              uint4* sup, uint4* del, int64_t W4, int64_t tupleBase, bool last, cudaStream_t s) {
    // the tiles of these tuples; the last call also writes the padding words of the rows
    const int64_t word0 = tupleBase / 32, rowWords = W4 * 4;
    const int64_t words = last ? rowWords - word0 : tuples / 32;
    const int64_t tiles = (words + kTileWords - 1) / kTileWords;
    if (tiles <= 0) return cudaSuccess;
    // variables over blocks until the grid has a few blocks per SM, then in turns
    // within a block (whose tuples then come from L1)
    const int64_t y = std::max<int64_t>(1, std::min<int64_t>(n, 8LL * sm_count() / tiles));
    ct_build_rows_kernel<<<dim3((unsigned)tiles, (unsigned)y), 256, 0, s>>>(
        tup, tuples, n, lo, row0, reinterpret_cast<uint32_t*>(sup), reinterpret_cast<uint32_t*>(del), rowWords, word0);
    return cudaGetLastError();
}

cudaError_t launch_build_state(const TableDev& T, int64_t t, cudaStream_t s) {
    const int64_t chunks = (int64_t)T.nseg * 32;
    ct_build_state_kernel<<<(unsigned)std::min<int64_t>((chunks + 255) / 256, 4LL * sm_count()), 256, 0, s>>>(T, t);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    ct_build_residue_kernel<<<(unsigned)std::min<int64_t>(((int64_t)T.R + 7) / 8, 8LL * sm_count()), 256, 0, s>>>(T);
    return cudaGetLastError();
}

}  // namespace ctk
