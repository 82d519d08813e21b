// ct_small.cu -- one propagation of a small table (Algorithm 1, enforceGAC) by
// one CTA: tables of at most 128 chunks (16,384 tuples), a value per thread.
//
// On such a table a call moves a few kilobytes; what it costs is the launch,
// the host's wait and the chain of round trips inside the kernel. The general
// kernel (ct_kernels.cu) spends most of its 8 us there on what several CTAs
// need of one another: counters flushed and read back through L2, a trail
// reservation, one or two grid barriers. Here currTable, the index, the plan
// and every counter live in shared memory, the trail position comes with the
// call, and the chain is: domains, residues and currTable; the call's rows
// beside the supports chunks at the residues; the rows of the values that
// missed; publication. The windows after a residue cover the table (4 at
// most), so no value is left for a full scan.
#include <cstdint>
#include <cuda_runtime.h>

#include "ct_device.cuh"

namespace ctk {
namespace {

constexpr int kPer = kSmallRows / kThreads;  // values per thread

struct SmallSmem {
    uint4 cur[kSmallChunks];
    int32_t lp[kSmallChunks];
    uint32_t mask[kSmallChunks / 32];
    int32_t codes[kSmallRows];
    uint32_t dom[kParamArity * kWarpPlanWords];      // the call's domains (packed)
    uint32_t removed[kParamArity * kWarpPlanWords];  // values to take off them
    unsigned long long other[kParamArity];  // negative tables: product of the other domain sizes (saturated)
    int32_t sup[kParamArity];               // |dom| > 1
    uint32_t cnt[12];
    int32_t nrows, nval, ndelta, nreset, nsup, status, trail, changed;
};

__global__ void __launch_bounds__(kThreads) ct_small_kernel(const __grid_constant__ TableDev T, uint32_t* dom,
                                                            const __grid_constant__ CallParams P) {
    __shared__ SmallSmem sm;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    SliceSmem& parts = *reinterpret_cast<SliceSmem*>(s_dyn);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned FULL = 0xffffffffu;
    uint64_t t0 = 0, t1 = 0, t2 = 0, t3 = 0;
    if (tid == 0) t0 = gtimer();
    const uint32_t* domIn = P.domInParams ? P.domWords : dom;
    const int W4 = T.W4, nseg = T.nseg;
    // currTable, trail links and index; every value's variable and residue
    if (tid < nseg * 32) {
        const bool in = tid < W4;
        sm.cur[tid] = in ? T.curr[tid] : make_uint4(0u, 0u, 0u, 0u);
        sm.lp[tid] = (in && P.mark >= 0) ? T.lastpos[tid] : 0x7fffffff;
    }
    if (tid < nseg) {
        const uint32_t m = T.segMask[tid];
        sm.mask[tid] = m;
        for (int l = P.snapFrom; l < P.snapTo; ++l) T.levelSeg[(size_t)l * nseg + tid] = m;
    }
    // a lane's values: consecutive ones in different warps, so that the few
    // values of a small scope (and their searches) spread over the CTA
    auto value_of = [&](int l, int k) { return l * kWarps + warp + k * kThreads; };
    int var[kPer], bit[kPer], res[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int r = value_of(lane, k);
        var[k] = 0;
        bit[k] = res[k] = 0;
        if (r < T.R) {
            for (int i = 1; i < T.arity; ++i) var[k] = r >= T.pRow0[i] ? i : var[k];
            bit[k] = r - T.pRow0[var[k]];
            if (!T.negative) res[k] = T.residue[r];
        }
    }
    if (tid < 12) sm.cnt[tid] = 0u;
    if (tid < T.DW) sm.removed[tid] = 0u;
    // plan (Algorithm 1 lines 1-3, the rows of Algorithm 2): warp 0, lane i holds variable i
    if (warp == 0) {
        const bool own = lane < T.arity;
        uint32_t d[kWarpPlanWords], l[kWarpPlanWords];
        int nw = 0, ld = 0, nd = 0, ndel = 0;
        uint32_t grow = 0u;
        if (own) {
            nw = T.pNW[lane];
            ld = T.pLD[lane];
            const uint32_t* dp = domIn + P.domOff[lane];
#pragma unroll
            for (int q = 0; q < kWarpPlanWords; ++q) {
                d[q] = q < nw ? dp[q] : 0u;
                l[q] = q < nw ? T.lastDom[ld + q] : 0u;
            }
#pragma unroll
            for (int q = 0; q < kWarpPlanWords; ++q) {
                grow |= d[q] & ~l[q];
                nd += __popc(d[q]);
                ndel += __popc(l[q] & ~d[q]);
                if (q < nw) {
                    sm.dom[ld + q] = d[q];
                    for (int v = P.snapFrom; v < P.snapTo; ++v) T.levelDom[(size_t)v * T.DW + ld + q] = l[q];
                }
            }
            sm.sup[lane] = nd > 1;
        }
        // Algorithm 2, line 3: the delta mask when |Delta| < |dom| (strict)
        const bool delta = ndel > 0 && ndel < nd;
        const bool bad = __ballot_sync(FULL, grow != 0u) != 0u;
        const bool empty = __ballot_sync(FULL, own && nd == 0) != 0u;
        const int nval = __popc(__ballot_sync(FULL, ndel > 0)), ndelta = __popc(__ballot_sync(FULL, delta));
        const int nsup = __popc(__ballot_sync(FULL, nd > 1));
        const int rows = (bad || empty || ndel == 0) ? 0 : delta ? ndel : nd;
        int incl = rows;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += a;
        }
        if (rows > 0) {
            int out = incl - rows;
            const int last = incl - 1;
#pragma unroll
            for (int q = 0; q < kWarpPlanWords; ++q) {
                uint32_t bits = delta ? (l[q] & ~d[q]) : d[q];
                while (bits) {
                    const int b = __ffs(bits) - 1;
                    bits &= bits - 1u;
                    int code = T.pRow0[lane] + q * 32 + b;
                    if (delta) code |= kCodeDelta;
                    if (out == last) code |= kCodeLast;
                    sm.codes[out++] = code;
                }
            }
        }
        if (T.negative) {
            // every value of x_i is excluded when all prod_{j != i} |D_j| combinations with it are forbidden
            unsigned long long prod = 1ull;
            for (int j = 0; j < T.arity; ++j) {
                const int s = __shfl_sync(FULL, nd, j);
                if (j != lane) prod = sat_mul(prod, (unsigned long long)s);
            }
            if (own) sm.other[lane] = prod;
        }
        if (lane == 31) {
            sm.nrows = incl;
            sm.nval = nval;
            sm.ndelta = ndelta;
            sm.nreset = nval - ndelta;
            sm.nsup = nsup;
            sm.status = bad ? CT_ERR_STATE : empty ? CT_INFEASIBLE : CT_OK;
            sm.trail = 0;
            sm.changed = 0;
        }
    }
    __syncthreads();
    if (tid == 0) t1 = gtimer();
    const int nrows = sm.nrows;
    int st = sm.status;
    const bool update = st == CT_OK && (nrows > 0 || T.negative);
    // the supports chunks at the residues of the values to test, beside the update's rows
    bool need[kPer];
    uint4 sr[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int r = value_of(lane, k);
        need[k] = r < T.R && st == CT_OK && ((sm.dom[T.pLD[var[k]] + (bit[k] >> 5)] >> (bit[k] & 31)) & 1u) &&
                  (T.negative || sm.sup[var[k]]);
        sr[k] = make_uint4(0u, 0u, 0u, 0u);
        if (need[k] && !T.negative) sr[k] = ld_sup_pred(T.sup + (size_t)r * W4 + res[k], true);
    }
    if (update) {
        // updateTable (Algorithm 2): the row list of a segment cut over up to
        // 8 / nseg warps, one batch of 16 loads each where that is enough
        int G = 1, lg = 0;
        const int want = (nrows + 15) / 16;
        while (G < want && (nseg << (lg + 1)) <= kWarps) {
            G <<= 1;
            ++lg;
        }
        const int per = (nrows + G - 1) >> lg, seg = warp >> lg, slice = warp & (G - 1);
        const bool unit = seg < nseg;
        SegState S;
        S.mask = unit ? sm.mask[seg] : 0u;
        S.cur = unit ? sm.cur[seg * 32 + lane] : make_uint4(0u, 0u, 0u, 0u);
        S.lp = unit ? sm.lp[seg * 32 + lane] : 0x7fffffff;
        uint4 acc = make_uint4(~0u, ~0u, ~0u, ~0u);
        if (G == 1) {
            if (S.mask != 0u)
                acc = slice_rows<16, false, false, 4>(T, seg, (S.mask >> lane) & 1u, S.cur, 0, nrows, sm.codes, nullptr, 0);
        } else {
            if (S.mask != 0u) {
                const int qa = min(nrows, slice * per);
                slice_rows<16, false, true, 4>(T, seg, (S.mask >> lane) & 1u, S.cur, qa, min(nrows, qa + per), sm.codes,
                                            &parts, warp);
            }
            __syncthreads();
            if (S.mask != 0u && slice == 0) acc = combine_slices(parts, warp, G);
        }
        if (S.mask != 0u && slice == 0) {
            TrailItem it;
            finish_segment(T, P.mark, seg, S, acc, sm.cnt, &sm.cnt[kCntTuples], it);
            sm.cur[seg * 32 + lane] = and4(S.cur, acc);
            // (trail positions from the call's on: this CTA is the only writer)
            const unsigned nb = __ballot_sync(FULL, it.need);
            int base = 0;
            if (lane == 0 && nb) base = atomicAdd(&sm.trail, __popc(nb));
            base = P.trailTop + __shfl_sync(FULL, base, 0);
            if (it.need) {
                const int p = base + __popc(nb & lanemask_lt());
                T.trailKey[p] = make_int2(it.w, it.lp);
                T.trailOld[p] = it.cur;
                T.lastpos[it.w] = p;
            }
        }
        __syncthreads();
        // Algorithm 1 line 5 (a negative table with no valid forbidden tuple forbids nothing)
        if (!T.negative && sm.cnt[kCntLive] == 0u) st = CT_INFEASIBLE;
    }
    if (tid == 0) t2 = gtimer();
    // filterDomains (Algorithm 3)
    if (st == CT_OK && T.negative) {
        // a value loses its support when the valid forbidden tuples carrying it
        // are all the combinations of the other domains: counted, a value per
        // warp, for those whose combinations do not exceed the valid tuples
        const unsigned long long liveT = sm.cnt[kCntTuples];
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            unsigned todo = __ballot_sync(FULL, need[k] && sm.other[var[k]] <= liveT);
            if (lane == 0 && todo) atomicAdd(&sm.cnt[kCntHard], (uint32_t)__popc(todo));
            while (todo) {
                constexpr int U = 4;  // values at a time
                int ln[U];
                uint32_t c[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    ln[u] = todo ? __ffs(todo) - 1 : -1;
                    todo &= todo - 1u;
                    c[u] = 0u;
                }
                for (int w = lane; w < W4; w += 32) {
                    const uint4 cw = sm.cur[w];
                    uint4 v[U];
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        v[u] = ld_sup_pred(T.sup + (size_t)value_of(max(ln[u], 0), k) * W4 + w,
                                           ln[u] >= 0 && nz(cw));
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        v[u] = and4(v[u], cw);
                        c[u] += __popc(v[u].x) + __popc(v[u].y) + __popc(v[u].z) + __popc(v[u].w);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t sum = __reduce_add_sync(FULL, c[u]);
                    if (lane == ln[u] && (unsigned long long)sum >= sm.other[var[k]])
                        atomicOr(&sm.removed[T.pLD[var[k]] + (bit[k] >> 5)], 1u << (bit[k] & 31));
                }
            }
        }
    } else if (st == CT_OK) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const bool hit = need[k] && nz(and4(sr[k], sm.cur[res[k]]));
            const int nhit = __popc(__ballot_sync(FULL, hit));
            unsigned miss = __ballot_sync(FULL, need[k] && !hit);
            if (lane == 0 && nhit) atomicAdd(&sm.cnt[kCntHits], (uint32_t)nhit);
            bool gone = need[k] && !hit;
            while (miss) {
                // four values at a time over the windows after their residues
                constexpr int U = 4;
                int ln[U], c[U];
                unsigned open = 0u;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    ln[u] = miss ? __ffs(miss) - 1 : 0;
                    if (miss) open |= 1u << u;
                    miss &= miss - 1u;
                    c[u] = wrap_chunk(__shfl_sync(FULL, res[k], ln[u]) + 1 + lane, W4);
                }
                for (int b = 0; b < nseg && open; ++b) {
                    if (lane == 0) atomicAdd(&sm.cnt[kCntWin], (uint32_t)__popc(open));
                    uint4 s[U];
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        s[u] = ld_sup_pred(T.sup + (size_t)value_of(ln[u], k) * W4 + c[u],
                                           ((open >> u) & 1u) && nz(sm.cur[c[u]]));
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        if (!((open >> u) & 1u)) continue;
                        const unsigned bal = __ballot_sync(FULL, nz(and4(s[u], sm.cur[c[u]])));
                        if (bal) {
                            const int cf = __shfl_sync(FULL, c[u], __ffs(bal) - 1);
                            if (lane == ln[u]) {
                                T.residue[value_of(lane, k)] = cf;
                                gone = false;
                            }
                            if (lane == 0) atomicAdd(&sm.cnt[kCntLocal], 1u);
                            open &= ~(1u << u);
                        }
                        c[u] = wrap_chunk(c[u] + 32, W4);
                    }
                }
            }
            const int ngone = __popc(__ballot_sync(FULL, gone));
            if (lane == 0 && ngone) atomicAdd(&sm.cnt[kCntHard], (uint32_t)ngone);
            if (gone) atomicOr(&sm.removed[T.pLD[var[k]] + (bit[k] >> 5)], 1u << (bit[k] & 31));
        }
    }
    __syncthreads();
    if (tid == 0) t3 = gtimer();
    // publication: removals, lastDom (a negative table's removed value still has
    // valid forbidden tuples, which the next call removes as Delta), the status block
    int32_t* H = T.statusBlk;
    if (st == CT_OK && tid < T.DW) {
        const uint32_t d = sm.dom[tid], r = sm.removed[tid], nd = d & ~r;
        T.lastDom[tid] = T.negative ? d : nd;
        reinterpret_cast<uint32_t*>(H + kStatusHdr + T.nChangedWords)[tid] = nd;
        if (r) {
            int i = 0;
            for (int j = 1; j < T.arity; ++j) i = tid >= T.pLD[j] ? j : i;
            if (!P.domInParams) dom[P.domOff[i] + tid - T.pLD[i]] = nd;
            atomicOr(&sm.changed, 1 << i);
            atomicAdd(&sm.cnt[kCntPruned], (uint32_t)__popc(r));
        }
    }
    __syncthreads();
    if (tid == 0) {
        H[kStatusHdr] = sm.changed;
        const int live = update ? (int)sm.cnt[kCntLive] : P.prevLive;
        H[kSlotLiveOut] = live;
        H[kSlotWordsIn] = (int)sm.cnt[kCntWords];
        H[kSlotTrailTop] = P.trailTop + sm.trail;
        H[kSlotMisses] = 0;
        H[kSlotPruned] = (int)sm.cnt[kCntPruned];
        H[kSlotHits] = (int)sm.cnt[kCntHits];
        H[kSlotRowsOred] = nrows;
        H[kSlotNval] = sm.nval;
        H[kSlotNsup] = sm.nsup;
        H[kSlotNdelta] = sm.ndelta;
        H[kSlotNreset] = sm.nreset;
        H[kSlotTrailAdded] = sm.trail;
        H[kSlotLiveIn] = update ? (int)sm.cnt[kCntLiveIn] : P.prevLive;
        H[kSlotLocal] = (int)sm.cnt[kCntLocal];
        H[kSlotHard] = (int)sm.cnt[kCntHard];
        H[kSlotWindows] = (int)sm.cnt[kCntWin];
        H[kSlotT1] = (int32_t)(t1 - t0);
        H[kSlotT2] = (int32_t)((update ? t2 : t1) - t0);
        H[kSlotT3] = (int32_t)(t3 - t0);
        H[kSlotT4] = (int32_t)(gtimer() - t0);
        H[kSlotScan] = T.negative ? (int)sm.cnt[kCntHard] : 0;
        H[kSlotEarly] = 0;
        if (sm.trail) T.ctrl->trail_top = P.trailTop + sm.trail;
        st_release_sys(&H[kSlotStatus], st);
    }
}

}  // namespace

bool small_table(const TableDev& T) {
    bool narrow = T.arity <= kParamArity;
    for (int i = 0; narrow && i < T.arity; ++i) narrow = T.pNW[i] <= kWarpPlanWords;
    return narrow && T.W4 <= kSmallChunks && T.R <= kSmallRows && T.useResidues && !T.shard;
}

cudaError_t launch_small(const TableDev& T, uint32_t* dom, const CallParams& P, cudaStream_t s) {
    ct_small_kernel<<<1, kThreads, sizeof(SliceSmem), s>>>(T, dom, P);
    return cudaGetLastError();
}

}  // namespace ctk
