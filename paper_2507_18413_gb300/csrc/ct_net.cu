// ct_net.cu -- the fixpoint of one small network in one cooperative launch with
// two grid barriers per round (ct_model_kernel, for networks of any size and
// for many nodes at once, has five).
//
// Rounds are the Jacobi steps of ct_model_kernel. What bounds them on a small
// network is the chain of dependent round trips to L2 and the barriers, not
// bytes: a node of the 20-variable, 8-table search (200 segments, 1,536 rows)
// took 24 us a round, of which 6 us in barriers. So work that every warp can do
// for itself is not handed over:
//   update   a warp plans the table of its (table, segment) unit itself (lane i
//            holds variable i), row codes in its own shared memory, while the
//            segment's state is loading; the warp of segment 0 stores what the
//            filter needs (row count, |dom| > 1, the domains as they were).
//   -- grid barrier --
//   filter   failure test; the residue of every (table, row), a row per lane,
//            residue and supports chunk loaded before the barrier; the warp
//            searches its own misses (few rows per warp) or, in a crowded
//            round, they are queued for the grid as in ct_model_kernel.
//   -- grid barrier --
//   next     every CTA finds the next round's tables for itself from the
//            variables' marks: the same list everywhere, no barrier.
// Nothing is reset where another CTA may still read it: marks, queue lengths
// and the tables' counters alternate by round parity, and a table's last-seen
// domains alternate between two buffers (lastDom and the unused code buffer),
// the update writing the one the plan does not read. Presence of a value in the
// filter is taken from the table's own copy of the domains, so that removals of
// other tables in the same round do not change what it tests (the same rounds
// and propagations as ct_model_kernel).
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

#include "ct_device.cuh"

namespace ctk {
namespace {

// The block of a launch in the kernel's parameters.
struct NetCall {
    int32_t words;
    alignas(16) int32_t w[kNetCallWords];
};

constexpr int kDirectRows = 4;  // rows per warp up to which a warp searches its own misses

// Dynamic shared memory, in words: per-warp row codes, the round's work list
// with its prefixes, per-table and per-scope tables, the variables' marks, and
// the table descriptors (small networks).
struct NetLayout {
    int codes, work, preU, preR, nseg, rows, mark, snap, base, var, off, prune, flip, done, tabs, words;
};

__host__ __device__ inline NetLayout net_layout(const ModelDev& M) {
    NetLayout L{};
    int at = 0;
    auto take = [&](int n) {
        const int a = at;
        at += (n + 3) & ~3;
        return a;
    };
    const int n = M.ntables, bits = (n + 31) / 32;
    L.codes = take(kWarps * M.netCodes);
    L.work = take(n);
    L.preU = take(n + 1);
    L.preR = take(n + 1);
    L.nseg = take(n);
    L.rows = take(n);
    L.mark = take(n);
    L.snap = take(n);
    L.base = take(n + 1);
    L.var = take(M.nscope);
    L.off = take(M.nscope);
    L.prune = take(M.nvars);
    L.flip = take(bits);
    L.done = take(bits);
    L.tabs = n <= kNetTabSmem ? take(n * (int)(sizeof(TableDev) / 4)) : -1;
    L.words = at;
    return L;
}

struct NetPlan {
    int nrows;
    bool bad;    // a domain grew since the table's last propagation
    bool empty;  // a domain is empty
};

// Algorithm 1 lines 1-3 and the row list of Algorithm 2 for one table by one
// warp (lane i holds variable i; plan_warp of ct_model_kernel): row codes into
// the warp's shared memory. off: the scope's domain offsets. The warp of
// segment 0 (store) also writes the row count, s_sup, the domains as the
// table's next last-seen ones and, into level `snap` (>= 0), the ones before.
__device__ __forceinline__ NetPlan net_plan(const TableDev& T, const int32_t* off, const uint32_t* dom,
                                            const uint32_t* last, uint32_t* next, int32_t* codes, bool store,
                                            int snap) {
    const int lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu;
    const bool own = lane < T.arity;
    uint32_t d[kWarpPlanWords], l[kWarpPlanWords];
    int nw = 0, ld = 0, nd = 0, ndel = 0;
    uint32_t grow = 0u;
    const VarLayout V(T, nullptr, off);
    if (own) {
        nw = V.nw(lane);
        ld = V.ld(lane);
        const uint32_t* dp = dom + off[lane];  // (parameters or global memory)
        const uint32_t* lp = last + ld;
#pragma unroll
        for (int q = 0; q < kWarpPlanWords; ++q) {
            d[q] = q < nw ? *reinterpret_cast<const volatile uint32_t*>(dp + q) : 0u;
            l[q] = q < nw ? __ldcg(lp + q) : 0u;
        }
#pragma unroll
        for (int q = 0; q < kWarpPlanWords; ++q) {
            grow |= d[q] & ~l[q];
            nd += __popc(d[q]);
            ndel += __popc(l[q] & ~d[q]);
        }
    }
    // Algorithm 2, line 3: the delta mask when |Delta| < |dom| (strict)
    const bool delta = ndel > 0 && ndel < nd;
    NetPlan P;
    P.bad = __ballot_sync(FULL, grow != 0u) != 0u;
    P.empty = __ballot_sync(FULL, own && nd == 0) != 0u;
    const int rows = (P.bad || P.empty || ndel == 0) ? 0 : delta ? ndel : nd;
    int incl = rows;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += a;
    }
    P.nrows = __shfl_sync(FULL, incl, 31);
    __syncwarp();  // (the codes of the warp's previous table have been read)
    if (rows > 0) {
        const int row0 = V.row0(lane);
        int out = incl - rows;
        const int lastAt = incl - 1;
#pragma unroll
        for (int q = 0; q < kWarpPlanWords; ++q) {
            uint32_t bits = delta ? (l[q] & ~d[q]) : d[q];
            while (bits) {
                const int b = __ffs(bits) - 1;
                bits &= bits - 1u;
                int code = row0 + q * 32 + b;
                if (delta) code |= kCodeDelta;
                if (out == lastAt) code |= kCodeLast;
                codes[out++] = code;
            }
        }
    }
    __syncwarp();
    if (store) {
        if (own) {
            T.varSup[lane] = nd > 1;
#pragma unroll
            for (int q = 0; q < kWarpPlanWords; ++q) {
                if (q < nw) {
                    next[ld + q] = d[q];
                    if (snap >= 0) T.levelDom[(size_t)snap * T.DW + ld + q] = l[q];
                }
            }
        }
        if (lane == 0) T.ctrl->nrows = P.nrows;
    }
    return P;
}

// in.words > 0: the launch's block (count, calls, domains, first work list) in
// the parameters; round 0 plans from those domains while they are stored.
// One CTA per SM, so that it has the 195 registers it takes: at 128 (two CTAs) the
// batches of rows spilled, 53.2 us a search node (8 tables of 100,000 tuples) and
// 51.1 without.
__global__ void __launch_bounds__(kThreads, 1)
ct_net_kernel(const __grid_constant__ ModelDev M, const __grid_constant__ NetCall in) {
    extern __shared__ __align__(16) int32_t dyn[];
    __shared__ uint32_t s_cnt[12];
    __shared__ int s_flag, s_sum[2 * kWarps];
    __shared__ unsigned long long s_bytes[2];
    const NetLayout L = net_layout(M);
    int32_t *work = dyn + L.work, *preU = dyn + L.preU, *preR = dyn + L.preR;
    const int32_t *s_nseg = dyn + L.nseg, *s_rows = dyn + L.rows, *s_mark = dyn + L.mark, *s_snap = dyn + L.snap;
    const int32_t *s_base = dyn + L.base, *s_var = dyn + L.var, *s_off = dyn + L.off;
    uint32_t *flip = reinterpret_cast<uint32_t*>(dyn + L.flip), *done = reinterpret_cast<uint32_t*>(dyn + L.done);
    const TableDev* tabs = L.tabs >= 0 ? reinterpret_cast<const TableDev*>(dyn + L.tabs) : M.tabs;
    ModelCtrl* C = M.ctrl;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int gwarp = blockIdx.x * kWarps + warp, nwarps = gridDim.x * kWarps;
    const int gtid = blockIdx.x * kThreads + tid, gth = gridDim.x * kThreads;
    const int n = M.ntables;
    int32_t* codes = dyn + L.codes + warp * M.netCodes;
    GridBarrier bar;
    bar_init(bar, &C->bar_count, &C->bar_base, &C->status, M.spinLimit ? M.spinLimit : kBarrierSpinLimit);
    auto sync = [&]() { return bar_sync(bar, &s_flag) != 0; };
    uint64_t tmark = (M.phaseNs && gtid == 0) ? gtimer() : 0ull;
    auto phase = [&](int p) {
        if (M.phaseNs && gtid == 0) {
            const uint64_t now = gtimer();
            M.phaseNs[p] += now - tmark;
            tmark = now;
        }
    };
    // the launch's constants, the first work list, and the marks of round 0
    const bool inl = in.words > 0;
    const uint32_t* dom0 = inl ? reinterpret_cast<const uint32_t*>(in.w) + 4 + 4 * n : M.dom;
    for (int t = tid; t < n; t += kThreads) {
        dyn[L.nseg + t] = __ldg(&M.tabs[t].nseg);
        dyn[L.rows + t] = __ldg(&M.tabs[t].R);
        const ModelTabCall cl = inl ? reinterpret_cast<const ModelTabCall*>(in.w + 4)[t] : M.calls[t];
        dyn[L.mark + t] = cl.mark;
        dyn[L.snap + t] = cl.snapFrom < cl.snapTo ? cl.snapFrom : -1;
    }
    if (inl)
        for (int q = gtid; q < M.DWg; q += gth) M.dom[q] = dom0[q];
    for (int t = tid; t <= n; t += kThreads) dyn[L.base + t] = __ldg(&M.scopeBase[t]);
    for (int q = tid; q < M.nscope; q += kThreads) {
        dyn[L.var + q] = __ldg(&M.scopeVar[q]);
        dyn[L.off + q] = __ldg(&M.scopeOff[q]);
    }
    if (L.tabs >= 0) {
        const int32_t* src = reinterpret_cast<const int32_t*>(M.tabs);
        for (int q = tid; q < n * (int)(sizeof(TableDev) / 4); q += kThreads) dyn[L.tabs + q] = __ldcg(src + q);
    }
    for (int q = tid; q < (n + 31) / 32; q += kThreads) flip[q] = done[q] = 0u;
    for (int v = gtid; v < M.nvars; v += gth) M.prunedBy[v] = -1;
    if (tid < 12) s_cnt[tid] = 0u;
    if (tid < 2) s_bytes[tid] = 0ull;
    int nwork = inl ? in.w[0] : __ldcg(M.nworkIn);
    for (int k = tid; k < nwork; k += kThreads) work[k] = inl ? in.w[4 + 4 * n + M.DWg + k] : __ldcg(&M.work[k]);
    __syncthreads();
    auto bit_of = [&](const uint32_t* bits, int t) { return (bits[t >> 5] >> (t & 31)) & 1u; };
    // a table's last-seen domains, and where the round's domains go
    auto last_of = [&](const TableDev& T, int t, bool next) {
        return (bit_of(flip, t) != (next ? 1u : 0u)) ? reinterpret_cast<uint32_t*>(T.codes) : T.lastDom;
    };
    int round = 0, props = 0;
    bool failed = false;
    for (;; ++round) {
        phase(round == 0 ? 0 : 6);
        const int par = round & 1;
        int32_t* pruned = M.prunedBy + (size_t)par * M.nvars;
        props += nwork;
        // prefixes of the work list's segments and rows (each thread a run of entries)
        {
            const int per = (nwork + kThreads - 1) / kThreads, b0 = tid * per, b1 = min(nwork, b0 + per);
            int su = 0, sr = 0;
            for (int k = b0; k < b1; ++k) {
                su += s_nseg[work[k]];
                sr += s_rows[work[k]];
            }
            int iu = su, ir = sr;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int a = __shfl_up_sync(0xffffffffu, iu, o), c = __shfl_up_sync(0xffffffffu, ir, o);
                if (lane >= o) {
                    iu += a;
                    ir += c;
                }
            }
            if (lane == 31) {
                s_sum[warp] = iu;
                s_sum[kWarps + warp] = ir;
            }
            __syncthreads();
            int ru = iu - su, rr = ir - sr;
            for (int w = 0; w < warp; ++w) {
                ru += s_sum[w];
                rr += s_sum[kWarps + w];
            }
            for (int k = b0; k < b1; ++k) {
                preU[k] = ru;
                preR[k] = rr;
                ru += s_nseg[work[k]];
                rr += s_rows[work[k]];
            }
            if (tid == kThreads - 1) {
                preU[nwork] = ru;
                preR[nwork] = rr;
            }
            __syncthreads();
        }
        const int totalUnits = preU[nwork], totalRows = preR[nwork];

        // the first row of the warp's lanes, what does not depend on the update:
        // its residue is on the way while the warp updates, then the supports chunk
        const int rpw = min(32, max(1, (totalRows + nwarps - 1) / nwarps));
        const bool direct = totalRows <= kDirectRows * nwarps;
        struct RowRef {
            int t, r, res, word, bit, var;
            uint4 sup;
        };
        auto row_ref = [&](int u) {
            RowRef R;
            const int k = lane_find_prefix(preR, nwork, u, false);
            R.t = work[k];
            R.r = u - preR[k];
            const TableDev& T = tabs[R.t];
            R.res = T.useResidues ? __ldcg(&T.residue[R.r]) : 0;
            R.var = __ldg(&T.rowVar[R.r]);
            return R;
        };
        auto row_sup = [&](RowRef& R) {
            const TableDev& T = tabs[R.t];
            R.sup = ld_sup(T.sup + (size_t)R.r * T.W4 + R.res);
            const VarLayout V(T, nullptr, nullptr);
            const int a = R.r - V.row0(R.var);
            R.word = V.ld(R.var) + (a >> 5);
            R.bit = a & 31;
        };
        RowRef R0{};
        const int u00 = gwarp * rpw;
        const bool row0 = lane < rpw && u00 + lane < totalRows;
        if (row0) R0 = row_ref(u00 + lane);

        // update: unit u to warp u % nwarps
        int planned = -1;
        NetPlan P{};
        for (int u = gwarp; u < totalUnits; u += nwarps) {
            const int k = find_prefix(preU, nwork, u, false);
            const int t = work[k], seg = u - preU[k];
            const TableDev& T = tabs[t];
            const int mark = s_mark[t];
            const SegState S = load_segment(T, seg, mark);
            const int cap = __ldcg(&T.ctrl->trail_cap);
            const bool first = seg == 0;
            const int snap = s_snap[t] >= 0 && !bit_of(done, t) ? s_snap[t] : -1;
            if (t != planned || first) {
                P = net_plan(T, s_off + s_base[t], round == 0 ? dom0 : M.dom, last_of(T, t, false), last_of(T, t, true), codes, first,
                             first ? snap : -1);
                planned = t;
                if (first && lane == 0) {
                    if (P.bad) atomicCAS(&C->status, CT_OK, CT_ERR_STATE);
                    else if (P.empty) M.nodeStatus[0] = CT_INFEASIBLE;
                }
            }
            if (snap >= 0 && lane == 0) T.levelSeg[(size_t)snap * T.nseg + seg] = S.mask;
            if (P.nrows > 0) {
                TrailItem it;
                it.need = false;
                if (S.mask != 0u) {
                    const uint4 acc = slice_rows<16, false, false, 4>(T, seg, (S.mask >> lane) & 1u, S.cur, 0, P.nrows,
                                                                   codes, nullptr, 0);
                    finish_segment(T, mark, seg, S, acc, T.ctrl->bank[par], &T.ctrl->tuples, it);
                }
                trail_warp(T, it, cap, &C->status);
            }
        }
        if (row0) row_sup(R0);
        if (!sync()) return;
        phase(2);

        // failure test (Algorithm 1 line 5) beside the first rows' loads (all of
        // them: read where they are used, each waited for the one before, 1.3 us a node)
        uint4 cur0 = make_uint4(0u, 0u, 0u, 0u);
        int32_t in0 = 0;
        uint32_t last0 = 0u;
        if (row0) {
            const TableDev& T = tabs[R0.t];
            cur0 = __ldcg(T.curr + R0.res);
            in0 = __ldcg(&T.varSup[R0.var]);
            last0 = __ldcg(last_of(T, R0.t, true) + R0.word);
        }
        bool stop = false;
        for (int k = tid; k < nwork; k += kThreads) {
            Ctrl* Tc = tabs[work[k]].ctrl;
            const int nr = __ldcg(&Tc->nrows);
            const uint32_t live = __ldcg(&Tc->bank[par][kCntLive]);
            stop |= nr > 0 && live == 0u;
            if (blockIdx.x == 0 && nr > 0) {
                Tc->live_state = (int32_t)live;
                atomicAdd(&s_bytes[0], 4ull * __ldcg(&Tc->bank[par][kCntWords]) * (unsigned long long)(nr + 2));
            }
        }
        if (tid == 0) stop |= __ldcg(&C->status) != CT_OK || __ldcg(&M.nodeStatus[0]) != CT_OK;
        failed = __syncthreads_or(stop) != 0;
        if (failed) {
            // (nothing below is reset before every CTA has read it)
            for (int k = tid; k < nwork; k += kThreads) atomicOr(&done[work[k] >> 5], 1u << (work[k] & 31));
            if (!sync()) return;
            break;
        }
        // the next round's marks, counters and queue lengths
        for (int v = gtid; v < M.nvars; v += gth) M.prunedBy[(size_t)(par ^ 1) * M.nvars + v] = -1;
        for (int t = gtid; t < n; t += gth) {
            uint32_t* b = tabs[t].ctrl->bank[par ^ 1];
            b[0] = b[1] = b[2] = 0u;
        }
        if (gtid == 0) {
            C->nmiss[par ^ 1] = 0;
            C->nscanAll[par ^ 1] = 0;
        }
        // Value r of table t has no support: off the shared domains and the
        // table's own copy; its variable is marked as pruned by t (-2: several)
        auto remove = [&](const TableDev& T, int t, int r) {
            const VarLayout V(T, nullptr, s_off + s_base[t]);
            const int i = T.rowVar[r], a = r - V.row0(i), v = s_var[s_base[t] + i];
            atomicAnd(&M.dom[V.off(i) + (a >> 5)], ~(1u << (a & 31)));
            atomicAnd(&last_of(T, t, true)[V.ld(i) + (a >> 5)], ~(1u << (a & 31)));
            const int old = atomicCAS(&pruned[v], -1, t);
            if (old != -1 && old != t) atomicExch(&pruned[v], -2);
        };
        auto undecided = [&](const TableDev& T, int r) {
            const unsigned m = atomicAdd(&T.ctrl->nhard, 1u);
            T.hardRow[m] = r;
            T.foundChunk[m] = kNoChunk;
            atomicAdd(&s_cnt[kCntMiss], 1u);
            atomicAdd(&C->nscanAll[par], 1);
        };
        // filterDomains (Algorithm 3)
        for (int u0 = u00; u0 < totalRows; u0 += nwarps * rpw) {
            const int u = u0 + lane;
            bool need = false, hit = false;
            RowRef R = R0;
            if (lane < rpw && u < totalRows) {
                uint4 cur = cur0;
                int32_t in = in0;
                uint32_t last = last0;
                if (u0 != u00) {
                    R = row_ref(u);
                    row_sup(R);
                    const TableDev& T = tabs[R.t];
                    cur = __ldcg(T.curr + R.res);
                    in = __ldcg(&T.varSup[R.var]);
                    last = __ldcg(last_of(T, R.t, true) + R.word);
                }
                const TableDev& T = tabs[R.t];
                const bool present = in != 0 && ((last >> R.bit) & 1u);
                hit = present && T.useResidues && nz(and4(R.sup, cur));
                need = present && !hit;
            }
            unsigned miss = __ballot_sync(0xffffffffu, need);
            const int nhit = __popc(__ballot_sync(0xffffffffu, hit));
            if (lane == 0 && nhit) atomicAdd(&s_cnt[kCntHits], (unsigned)nhit);
            if (direct) {
                while (miss) {
                    const int l = __ffs(miss) - 1;
                    miss &= miss - 1u;
                    const int t = __shfl_sync(0xffffffffu, R.t, l), r = __shfl_sync(0xffffffffu, R.r, l);
                    const TableDev& T = tabs[t];
                    const int o = probe_network(T, r, __shfl_sync(0xffffffffu, R.res, l), s_cnt);
                    if (lane == 0 && o == kProbeGone) remove(T, t, r);
                    else if (lane == 0 && o != kProbeFound) undecided(T, r);
                }
            } else if (miss) {
                int base = 0;
                if (lane == 0) base = atomicAdd(&C->nmiss[par], __popc(miss));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (need) M.missQ[base + __popc(miss & lanemask_lt())] = make_int4(R.t, R.r, R.res, 0);
            }
        }
        if (!direct) {
            if (!sync()) return;
            const int nm = __ldcg(&C->nmiss[par]);
            for (int q = gwarp; q < nm; q += nwarps) {
                const int4 e = __ldcg(&M.missQ[q]);
                const TableDev& T = tabs[e.x];
                const int o = probe_network(T, e.y, e.z, s_cnt);
                if (lane == 0 && o == kProbeGone) remove(T, e.x, e.y);
                else if (lane == 0 && o != kProbeFound) undecided(T, e.y);
            }
        }
        __syncthreads();
        if (tid == 0) {
            if (s_cnt[kCntHits]) atomicAdd(&C->hits, s_cnt[kCntHits]);
            if (s_cnt[kCntLocal]) atomicAdd(&C->local, s_cnt[kCntLocal]);
            if (s_cnt[kCntMiss]) atomicAdd(&C->hard, s_cnt[kCntMiss]);
            if (s_cnt[kCntWin]) atomicAdd(&C->windows, s_cnt[kCntWin]);
            s_cnt[kCntHits] = s_cnt[kCntLocal] = s_cnt[kCntMiss] = s_cnt[kCntWin] = 0u;
        }
        if (!sync()) return;
        phase(3);
        if (__ldcg(&C->nscanAll[par]) > 0) {
            // full scans of the values whose residues and windows missed
            for (int u = gwarp; u < totalUnits; u += nwarps) {
                const int k = find_prefix(preU, nwork, u, false);
                const TableDev& T = tabs[work[k]];
                const int nh = (int)__ldcg(&T.ctrl->nhard);
                if (nh > 0) scan_segment<16, true>(T, u - preU[k], 0, nh, nullptr);
            }
            if (!sync()) return;
            phase(4);
            // Algorithm 3 line 4: remove the values no live tuple carries
            for (int k = blockIdx.x; k < nwork; k += gridDim.x) {
                const int t = work[k];
                const TableDev& T = tabs[t];
                const int nh = (int)__ldcg(&T.ctrl->nhard);
                for (int m = tid; m < nh; m += kThreads) {
                    const int r = __ldcg(&T.hardRow[m]), fc = __ldcg(&T.foundChunk[m]);
                    if (fc != kNoChunk) T.residue[r] = fc;
                    else remove(T, t, r);
                }
                __syncthreads();
                if (tid == 0 && nh > 0) {
                    // (a table's live count is final since the update)
                    const int nr = __ldcg(&T.ctrl->nrows);
                    const unsigned long long live = nr > 0 ? __ldcg(&T.ctrl->bank[par][kCntLive])
                                                           : (unsigned long long)__ldcg(&T.ctrl->live_state);
                    atomicAdd(&C->bytesFilter, 16ull * (unsigned)nh * live);
                    T.ctrl->nhard = 0u;
                }
            }
            if (!sync()) return;
            phase(5);
        }
        // next round: the tables that share a variable another table pruned,
        // ascending (every CTA the same list)
        for (int v = tid; v < M.nvars; v += kThreads) dyn[L.prune + v] = __ldcg(&pruned[v]);
        for (int k = tid; k < nwork; k += kThreads) {
            const int t = work[k];
            atomicXor(&flip[t >> 5], 1u << (t & 31));
            atomicOr(&done[t >> 5], 1u << (t & 31));
        }
        __syncthreads();
        int nnext = 0;
        for (int t0 = 0; t0 < n; t0 += kThreads) {
            const int t = t0 + tid;
            bool dirty = false;
            if (t < n)
                for (int j = s_base[t]; j < s_base[t + 1]; ++j) {
                    const int p = dyn[L.prune + s_var[j]];
                    dirty |= p != -1 && p != t;
                }
            const unsigned bal = __ballot_sync(0xffffffffu, dirty);
            if (lane == 0) s_sum[warp] = __popc(bal);
            __syncthreads();
            int at = nnext + __popc(bal & lanemask_lt());
            for (int w = 0; w < kWarps; ++w) {
                if (w < warp) at += s_sum[w];
                nnext += s_sum[w];
            }
            if (dirty) work[at] = t;
            __syncthreads();
        }
        nwork = nnext;
        if (nwork == 0) {
            ++round;
            break;
        }
        if (round + 1 >= M.maxRounds) {
            if (gtid == 0) atomicCAS(&C->status, CT_OK, CT_ERR_TIMEOUT);
            ++round;
            break;
        }
    }
    if (failed) ++round;
    phase(6);

    // The tables' state as other kernels expect it: last-seen domains in lastDom,
    // counters clear (every CTA is past its last read of them). The host may
    // start anything once it has the status word, so all of it is done before:
    // by the CTAs that do not publish, beside the publication, which waits for
    // them before its last store; of few tables by CTA 0 itself, which saves the
    // wait (200 search nodes of 8 tables 10.04 and 9.88 ms, 9.79 with the clean-up
    // behind the publication; 40 and 64 tables no different).
    const bool alone = gridDim.x == 1 || n <= 2 * kWarps;
    if (alone && blockIdx.x != 0) return;
    const int idle = alone ? 0 : kWarps;  // warps of CTA 0, which publishes
    for (int t = gwarp - idle; t >= 0 && t < n; t += alone ? kWarps : nwarps - idle) {
        const TableDev& T = tabs[t];
        if (bit_of(flip, t))
            for (int q = lane; q < T.DW; q += 32) T.lastDom[q] = __ldcg(reinterpret_cast<uint32_t*>(T.codes) + q);
        if (lane < 8) (&T.ctrl->bank[0][0])[lane] = 0u;
        if (lane == 8) T.ctrl->nrows = 0;
    }
    if (blockIdx.x != 0) {
        __syncthreads();
        if (tid == 0) bar_signal(bar);
        return;
    }
    // publish: CTA 0, the status word last
    // (of the tables, those that ran: bit t of the words after the node status; a
    // table's two words and the host's bookkeeping for them cost 2-5 us a call on 512 tables)
    int32_t* H = M.statusBlk;
    int st = CT_OK;
    if (tid == 0) {
        st = __ldcg(&C->status);
        const uint32_t hits = __ldcg(&C->hits), local = __ldcg(&C->local), hard = __ldcg(&C->hard);
        const uint32_t windows = __ldcg(&C->windows);
        const unsigned long long bf = __ldcg(&C->bytesFilter) + 4ull * hits + 512ull * windows, bu = s_bytes[0];
        C->hits = C->local = C->hard = C->windows = 0u;
        C->bytesFilter = 0ull;
        C->nmiss[0] = C->nmiss[1] = 0;
        C->nscanAll[0] = C->nscanAll[1] = 0;
        C->status = CT_OK;
        C->nwork = 0;
        M.nodeStatus[0] = CT_OK;
        H[kModelHdr + 2 * n + M.DWg] = failed && st == CT_OK ? CT_INFEASIBLE : CT_OK;
        H[1] = round;
        H[2] = props;
        H[3] = (int32_t)hits;
        H[4] = (int32_t)local;
        H[5] = (int32_t)hard;
        H[6] = (int32_t)windows;
        H[8] = (int32_t)(bu & 0xffffffffull);
        H[9] = (int32_t)(bu >> 32);
        H[10] = (int32_t)(bf & 0xffffffffull);
        H[11] = (int32_t)(bf >> 32);
    }
    uint32_t* outDom = reinterpret_cast<uint32_t*>(H + kModelHdr + 2 * n);
    for (int q0 = tid; q0 < M.DWg; q0 += 8 * kThreads) {
        uint32_t w[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (q0 + u * kThreads < M.DWg) w[u] = __ldcg(&M.dom[q0 + u * kThreads]);
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (q0 + u * kThreads < M.DWg) outDom[q0 + u * kThreads] = w[u];
    }
    for (int t = tid; t < n; t += kThreads) {
        if (!bit_of(done, t)) continue;
        const Ctrl* Tc = tabs[t].ctrl;
        const int top = __ldcg(&Tc->trail_top), live = __ldcg(&Tc->live_state);
        H[kModelHdr + 2 * t] = top;
        H[kModelHdr + 2 * t + 1] = live;
    }
    int32_t* outRan = H + kModelHdr + 2 * n + M.DWg + 1;
    for (int q = tid; q < (n + 31) / 32; q += kThreads) outRan[q] = (int32_t)done[q];
    __syncthreads();
    if (tid == 0 && (alone || bar_collect(bar))) {
        phase(7);
        st_release_sys(&H[0], st);
    }
}

}  // namespace

int net_smem_bytes(const ModelDev& M) { return net_layout(M).words * (int)sizeof(int32_t); }

int max_coresident_net_blocks(const ModelDev& M) {
    int dev = 0, sms = 0, per = 0;
    const int bytes = net_smem_bytes(M);
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(ct_net_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kNetSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, ct_net_kernel, kThreads, bytes) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return per * sms;
}

cudaError_t launch_net(const ModelDev& M, const int32_t* block, int words, int grid, cudaStream_t s) {
    ModelDev m = M;
    NetCall in;
    in.words = block && words <= kNetCallWords ? words : 0;
    if (in.words > 0) std::memcpy(in.w, block, (size_t)words * sizeof(int32_t));
    void* args[] = {&m, &in};
    return cudaLaunchCooperativeKernel((const void*)ct_net_kernel, dim3(grid), dim3(kThreads), args,
                                       (size_t)net_smem_bytes(M), s);
}

}  // namespace ctk
