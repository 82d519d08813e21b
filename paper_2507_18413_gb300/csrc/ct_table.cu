// ct_table.cu -- host side of one table constraint: construction of the
// device layout (Sec. 3 constructor, Sec. 4 device copies), propagation calls,
// backtrack levels and inspection.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "ct_table.cuh"

using namespace ctk;

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
static thread_local std::string g_err;

void ct_set_error(const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
}

int ct_cuda_fail(cudaError_t e, const char* what) {
    ct_set_error("%s: %s", what, cudaGetErrorString(e));
    return CT_ERR_CUDA;
}

extern "C" const char* ct_last_error(void) { return g_err.c_str(); }

extern "C" const char* ct_status_string(int s) {
    switch (s) {
        case CT_OK: return "CT_OK";
        case CT_INFEASIBLE: return "CT_INFEASIBLE";
        case CT_ERR_ARG: return "CT_ERR_ARG";
        case CT_ERR_OOM: return "CT_ERR_OOM";
        case CT_ERR_CUDA: return "CT_ERR_CUDA";
        case CT_ERR_STATE: return "CT_ERR_STATE";
        case CT_ERR_TIMEOUT: return "CT_ERR_TIMEOUT";
        case CT_ERR_LEVEL: return "CT_ERR_LEVEL";
        default: return "CT_UNKNOWN";
    }
}

extern "C" int ct_version(void) { return 10000; }

extern "C" int ct_read_ceiling(const void* dev_buf, int64_t bytes, void* cuda_stream, float* ms_out) {
    if (!dev_buf || bytes <= 0 || (bytes & 15) || (reinterpret_cast<uintptr_t>(dev_buf) & 15)) {
        ct_set_error("ct_read_ceiling: a 16-byte aligned buffer and a positive multiple of 16 bytes");
        return CT_ERR_ARG;
    }
    const cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    cudaEvent_t ev[2] = {nullptr, nullptr};
    cudaError_t e = cudaSuccess;
    if (ms_out) {
        e = cudaEventCreate(&ev[0]);
        if (e == cudaSuccess) e = cudaEventCreate(&ev[1]);
        if (e == cudaSuccess) e = cudaEventRecord(ev[0], s);
    }
    if (e == cudaSuccess) e = ctk::launch_read_ceiling(static_cast<const uint4*>(dev_buf), (size_t)(bytes / 16), s);
    if (ms_out && e == cudaSuccess) {
        e = cudaEventRecord(ev[1], s);
        if (e == cudaSuccess) e = cudaEventSynchronize(ev[1]);
        if (e == cudaSuccess) e = cudaEventElapsedTime(ms_out, ev[0], ev[1]);
    }
    for (cudaEvent_t x : ev)
        if (x) cudaEventDestroy(x);
    if (e != cudaSuccess) {
        ct_set_error("ct_read_ceiling: %s", cudaGetErrorString(e));
        return CT_ERR_CUDA;
    }
    return CT_OK;
}


namespace {

// ---------------------------------------------------------------------------
// device buffers of tables: every buffer a table owns (ct_create's buffers,
// the trail and the level stack) is allocated and freed here, with the test
// hooks ct_debug_*: guard regions around each buffer, a countdown that makes
// one allocation fail, and the bytes held, counted by the allocator itself
// ---------------------------------------------------------------------------
constexpr size_t kGuardBytes = 256;       // before and after a guarded buffer (keeps its 256-byte alignment)
constexpr unsigned char kGuardFill = 0xA5;
// One device allocation holding the buffers that were asked for together
// (cudaMalloc takes about 33 us and cudaFree 28 us here, whatever the size: a
// table's 25 buffers one by one made most of its construction); freed with the
// last of them.
struct DevBlock {
    char* base;
    int used;  // buffers still held
};
struct DevBuf {
    size_t bytes;
    bool guarded;
    DevBlock* block;
};
std::mutex g_bufMu;
std::unordered_map<void*, DevBuf> g_bufs;  // buffer as the table sees it -> size
int64_t g_bufBytes = 0;
int64_t g_stageBytes = 0;                  // device scratch of constructions under way
int64_t g_limitBytes = -1;                 // ct_debug_limit_bytes: a device of this many bytes (-1: the real one)
bool g_guardNew = false;                   // ct_debug_guard_buffers
long long g_failAfter = -1;                // ct_debug_fail_alloc: allocations left before one fails

struct BufAsk {
    void** p;
    size_t bytes;
};

// Whether n more device bytes are beyond the test hook's limit (under g_bufMu).
bool beyond_limit(int64_t n) { return g_limitBytes >= 0 && g_bufBytes + g_stageBytes + n > g_limitBytes; }

// The buffers of `ask` in one allocation, all or none (each counts as one
// allocation of the failure countdown; *injected: it was the countdown that failed it).
cudaError_t table_malloc_all(const std::vector<BufAsk>& ask, bool* injected = nullptr) {
    std::lock_guard<std::mutex> lk(g_bufMu);
    for (const BufAsk& a : ask) *a.p = nullptr;
    if (g_failAfter >= 0) {
        if (g_failAfter < (long long)ask.size()) {
            g_failAfter = -1;
            if (injected) *injected = true;
            return cudaErrorMemoryAllocation;
        }
        g_failAfter -= (long long)ask.size();
    }
    const bool guarded = g_guardNew;
    const size_t guard = guarded ? kGuardBytes : 0;
    auto room = [&](size_t bytes) { return ((bytes + 255) & ~size_t(255)) + 2 * guard; };
    size_t total = 0, sum = 0;
    for (const BufAsk& a : ask) {
        total += room(a.bytes);
        sum += a.bytes;
    }
    if (beyond_limit((int64_t)sum)) return cudaErrorMemoryAllocation;
    char* base = nullptr;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&base), total);
    if (e != cudaSuccess) return e;
    if (guarded) {
        // (the guard behind a buffer begins at its last byte; the rounding behind
        // it is filled too, as nobody writes there)
        e = cudaMemset(base, kGuardFill, total);
        if (e == cudaSuccess) e = cudaDeviceSynchronize();  // the guards are set before any use
        if (e != cudaSuccess) {
            cudaFree(base);
            return e;
        }
    }
    DevBlock* block = new DevBlock{base, (int)ask.size()};
    size_t at = 0;
    for (const BufAsk& a : ask) {
        void* user = base + at + guard;
        g_bufs[user] = DevBuf{a.bytes, guarded, block};
        g_bufBytes += (int64_t)a.bytes;
        *a.p = user;
        at += room(a.bytes);
    }
    return cudaSuccess;
}

void table_free(void* p) {
    if (!p) return;
    std::lock_guard<std::mutex> lk(g_bufMu);
    const auto it = g_bufs.find(p);
    if (it == g_bufs.end()) {
        cudaFree(p);
        return;
    }
    g_bufBytes -= (int64_t)it->second.bytes;
    DevBlock* block = it->second.block;
    g_bufs.erase(it);
    if (--block->used == 0) {
        cudaFree(block->base);
        delete block;
    }
}

// A table's buffers, asked for one by one and allocated together by take().
struct TableBufs {
    ct_table* ct;
    std::vector<BufAsk> ask;
    bool injected = false;  // the last take() failed by the test hook's countdown
    template <typename T>
    void want(T** p, size_t count) {
        ask.push_back({reinterpret_cast<void**>(const_cast<std::remove_const_t<T>**>(p)), std::max<size_t>(count, 1) * sizeof(T)});
    }
    int take() {
        size_t bytes = 0;
        for (const BufAsk& a : ask) bytes += a.bytes;
        const cudaError_t e = table_malloc_all(ask, &injected);
        if (e != cudaSuccess) {
            cudaGetLastError();
            ct_set_error("device buffers of a table (%zu bytes): %s", bytes, cudaGetErrorString(e));
            return CT_ERR_OOM;
        }
        for (const BufAsk& a : ask) ct->allocs.push_back(*a.p);
        ct->deviceBytes += (int64_t)bytes;
        return CT_OK;
    }
};

// ---------------------------------------------------------------------------
// status blocks: mapped host memory, in slabs shared by the tables of the
// process (cudaHostAlloc and cudaFreeHost take 110-250 us and 160 us here).
// Blocks of up to kSlabBytes / 4 come from a slab of kSlabUnit units; a slab is
// given back with its last block, but for one empty slab that is kept for the
// next table. Larger blocks are allocations of their own.
// ---------------------------------------------------------------------------
constexpr size_t kSlabBytes = 64 << 10, kSlabUnit = 256;
constexpr int kSlabUnits = (int)(kSlabBytes / kSlabUnit);
struct Slab {
    char* base = nullptr;
    std::vector<bool> taken = std::vector<bool>(kSlabUnits, false);
    int blocks = 0;
};
std::mutex g_slabMu;
std::vector<Slab*> g_slabs;
std::unordered_map<void*, std::pair<Slab*, int>> g_statusBlocks;  // block -> (slab, units); slab null: its own

cudaError_t status_alloc(void** p, size_t bytes) {
    std::lock_guard<std::mutex> lk(g_slabMu);
    *p = nullptr;
    if (bytes > kSlabBytes / 4) {
        const cudaError_t e = cudaHostAlloc(p, bytes, cudaHostAllocMapped | cudaHostAllocPortable);
        if (e == cudaSuccess) g_statusBlocks[*p] = {nullptr, 0};
        return e;
    }
    const int units = (int)((bytes + kSlabUnit - 1) / kSlabUnit);
    for (size_t k = 0; k <= g_slabs.size(); ++k) {
        if (k == g_slabs.size()) {
            Slab* s = new Slab();
            const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&s->base), kSlabBytes,
                                                cudaHostAllocMapped | cudaHostAllocPortable);
            if (e != cudaSuccess) {
                delete s;
                return e;
            }
            g_slabs.push_back(s);
        }
        Slab* s = g_slabs[k];
        for (int u = 0, run = 0; u < kSlabUnits; ++u) {
            run = s->taken[u] ? 0 : run + 1;
            if (run < units) continue;
            const int first = u + 1 - units;
            std::fill(s->taken.begin() + first, s->taken.begin() + u + 1, true);
            s->blocks += 1;
            *p = s->base + (size_t)first * kSlabUnit;
            g_statusBlocks[*p] = {s, units};
            return cudaSuccess;
        }
    }
    return cudaErrorMemoryAllocation;  // (a new slab has room for any block)
}

void status_free(void* p) {
    if (!p) return;
    std::lock_guard<std::mutex> lk(g_slabMu);
    const auto it = g_statusBlocks.find(p);
    if (it == g_statusBlocks.end()) return;
    Slab* s = it->second.first;
    const int units = it->second.second;
    g_statusBlocks.erase(it);
    if (!s) {
        cudaFreeHost(p);
        return;
    }
    const int first = (int)((static_cast<char*>(p) - s->base) / kSlabUnit);
    std::fill(s->taken.begin() + first, s->taken.begin() + first + units, false);
    if (--s->blocks > 0) return;
    int empty = 0;
    for (const Slab* o : g_slabs) empty += o->blocks == 0;
    if (empty < 2) return;  // the one empty slab that is kept
    g_slabs.erase(std::find(g_slabs.begin(), g_slabs.end(), s));
    cudaFreeHost(s->base);
    delete s;
}

template <typename T>
int upload(ct_table* ct, T* dst, const std::vector<T>& src) {
    if (src.empty()) return CT_OK;
    CT_CUDA(cudaMemcpyAsync(dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, ct->stream));
    return CT_OK;
}

int sync(ct_table* ct) {
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    return CT_OK;
}

// Grow the trail so that `need` entries fit.
// The event ring of ct_options.profile (created once, on first use).
int create_events(ct_table* ct) {
    ct->ev.assign(2 * ct_table::kEvRing, nullptr);
    for (auto& e : ct->ev) CT_CUDA(cudaEventCreate(&e));
    return CT_OK;
}

int ensure_trail(ct_table* ct, int64_t need) {
    if (need <= ct->trailCap) return CT_OK;
    if (need > 0x7fffffffLL) {
        ct_set_error("trail would exceed 2^31 entries");
        return CT_ERR_OOM;
    }
    int64_t cap = std::max<int64_t>(need, 2LL * ct->trailCap);
    if (cap > 0x7fffffffLL) cap = 0x7fffffffLL;
    int2* nk = nullptr;
    uint4* no = nullptr;
    const cudaError_t e = table_malloc_all({{reinterpret_cast<void**>(&nk), (size_t)cap * sizeof(int2)},
                                            {reinterpret_cast<void**>(&no), (size_t)cap * sizeof(uint4)}});
    if (e != cudaSuccess) {
        cudaGetLastError();
        ct_set_error("trail growth to %lld entries: %s", (long long)cap, cudaGetErrorString(e));
        return CT_ERR_OOM;
    }
    if (ct->trailTop > 0) {
        CT_CUDA(cudaMemcpyAsync(nk, ct->dev.trailKey, (size_t)ct->trailTop * sizeof(int2), cudaMemcpyDeviceToDevice,
                                ct->stream));
        CT_CUDA(cudaMemcpyAsync(no, ct->dev.trailOld, (size_t)ct->trailTop * sizeof(uint4),
                                cudaMemcpyDeviceToDevice, ct->stream));
    }
    int32_t capi = (int32_t)cap;
    CT_CUDA(cudaMemcpyAsync(&ct->dev.ctrl->trail_cap, &capi, sizeof(int32_t), cudaMemcpyHostToDevice, ct->stream));
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    if (!ct->trailInArena) {
        table_free(ct->dev.trailKey);
        table_free(ct->dev.trailOld);
    }
    ct->trailInArena = false;
    ct->deviceBytes += (cap - ct->trailCap) * (int64_t)(sizeof(int2) + sizeof(uint4));
    ct->dev.trailKey = nk;
    ct->dev.trailOld = no;
    ct->trailCap = (int)cap;
    ct->version++;
    return CT_OK;
}

int ensure_levels(ct_table* ct, int need) {
    if (need <= ct->levelCap) return CT_OK;
    const int cap = std::max(need, 2 * ct->levelCap);
    uint32_t* ns = nullptr;
    uint32_t* nd = nullptr;
    const cudaError_t e =
        table_malloc_all({{reinterpret_cast<void**>(&ns), (size_t)cap * std::max(ct->nseg, 1) * sizeof(uint32_t)},
                          {reinterpret_cast<void**>(&nd), (size_t)cap * std::max(ct->DW, 1) * sizeof(uint32_t)}});
    if (e != cudaSuccess) {
        cudaGetLastError();
        ct_set_error("level stack growth: %s", cudaGetErrorString(e));
        return CT_ERR_OOM;
    }
    const int used = (int)ct->levels.size();
    if (used > 0) {
        CT_CUDA(cudaMemcpyAsync(ns, ct->dev.levelSeg, (size_t)used * ct->nseg * sizeof(uint32_t),
                                cudaMemcpyDeviceToDevice, ct->stream));
        CT_CUDA(cudaMemcpyAsync(nd, ct->dev.levelDom, (size_t)used * ct->DW * sizeof(uint32_t),
                                cudaMemcpyDeviceToDevice, ct->stream));
    }
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    if (!ct->levelsInArena) {
        table_free(ct->dev.levelSeg);
        table_free(ct->dev.levelDom);
    }
    ct->levelsInArena = false;
    ct->deviceBytes += (int64_t)(cap - ct->levelCap) * (ct->nseg * 4 + ct->DW * 4);
    ct->dev.levelSeg = ns;
    ct->dev.levelDom = nd;
    ct->levelCap = cap;
    ct->version++;
    return CT_OK;
}

void free_table(ct_table* ct) {
    if (!ct) return;
    if (ct->stream) cudaStreamSynchronize(ct->stream);
    for (void* p : ct->allocs) table_free(p);
    if (!ct->trailInArena) {
        table_free(ct->dev.trailKey);
        table_free(ct->dev.trailOld);
    }
    if (!ct->levelsInArena) {
        table_free(ct->dev.levelSeg);
        table_free(ct->dev.levelDom);
    }
    status_free(ct->h_status);
    if (ct->h_curr) cudaFreeHost(ct->h_curr);
    for (auto& e : ct->ev)
        if (e) cudaEventDestroy(e);
    if (ct->ownStream && ct->stream) cudaStreamDestroy(ct->stream);
    cudaGetLastError();
    delete ct;
}

// The tuple list while a table is built, with the layout its kernels need: a
// bounded scratch buffer on the device (kStageInts components; lists beyond it go
// through in chunks), given back when the rows are built. Not one of the table's
// buffers, and never the reason that a table does not fit: it gets smaller where
// memory is short, steps aside for the table's buffers (close, then open again),
// and where the device has no room for 1,024 tuples it is mapped host memory,
// which the kernels read.
struct TupleStage {
    static constexpr int64_t kStageInts = 1LL << 26;  // 256 MB
    char* base = nullptr;  // as the kernels address it
    char* host = nullptr;  // ... and the host, when it is mapped host memory
    int64_t bytes = 0;     // device bytes held
    cudaStream_t stream = nullptr;
    int32_t* lo = nullptr;
    int32_t* row0 = nullptr;
    unsigned long long* counts = nullptr;
    int32_t* tup = nullptr;
    int64_t cap = 0;              // tuples per chunk (a multiple of 1,024)
    const int32_t* held = nullptr;  // host list whose chunk at heldAt is in the stage
    int64_t heldAt = 0;
    std::vector<int32_t> meta;  // what lo and row0 are copied from (kept until the copy is done)
    ~TupleStage() { close(); }
    void close() {
        if (host) {
            cudaStreamSynchronize(stream);  // (a kernel may still read it)
            cudaFreeHost(host);
        } else if (base) {
            cudaFree(base);
        }
        if (bytes > 0) {
            std::lock_guard<std::mutex> lk(g_bufMu);
            g_stageBytes -= bytes;
        }
        base = host = nullptr;
        held = nullptr;
        bytes = 0;
    }
    cudaError_t take_device(size_t n) {
        {
            std::lock_guard<std::mutex> lk(g_bufMu);
            if (beyond_limit((int64_t)n)) return cudaErrorMemoryAllocation;
            g_stageBytes += (int64_t)n;
        }
        bytes = (int64_t)n;
        const cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&base), n);
        if (e != cudaSuccess) {
            cudaGetLastError();
            base = nullptr;
            close();
        }
        return e;
    }
    // Room for t tuples of n components, or as many as memory allows.
    int open(const ct_table* ct, int64_t t) {
        const int n = ct->arity;
        stream = ct->stream;
        const int64_t whole = (t + 1023) / 1024 * 1024;
        cap = std::max<int64_t>(1024, std::min(whole, kStageInts / n / 1024 * 1024));
        const size_t head = ((size_t)(2 * n + 1) * sizeof(int32_t) + 2 * sizeof(unsigned long long) + 511) & ~size_t(255);
        while (take_device(head + (size_t)cap * n * sizeof(int32_t)) != cudaSuccess) {
            if (cap == 1024) {
                const cudaError_t e = cudaHostAlloc(reinterpret_cast<void**>(&host), head + (size_t)cap * n * sizeof(int32_t),
                                                    cudaHostAllocMapped);
                if (e != cudaSuccess) {
                    cudaGetLastError();
                    host = nullptr;
                    ct_set_error("ct_create: scratch for the tuples: %s", cudaGetErrorString(e));
                    return CT_ERR_OOM;
                }
                CT_CUDA(cudaHostGetDevicePointer(reinterpret_cast<void**>(&base), host, 0));
                break;
            }
            cap = std::max<int64_t>(1024, cap / 2 / 1024 * 1024);
        }
        counts = reinterpret_cast<unsigned long long*>(base);
        lo = reinterpret_cast<int32_t*>(base + 2 * sizeof(unsigned long long));
        row0 = lo + n;
        tup = reinterpret_cast<int32_t*>(base + head);
        meta.assign(2 * sizeof(unsigned long long) / sizeof(int32_t), 0);  // the counts start at zero
        meta.insert(meta.end(), ct->lo.begin(), ct->lo.end());
        meta.insert(meta.end(), ct->row0.begin(), ct->row0.end());
        return put(ct, base, meta.data(), meta.size() * sizeof(int32_t));
    }
    int put(const ct_table* ct, void* dst, const void* src, size_t n) {
        if (!host) {
            CT_CUDA(cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, ct->stream));
            return CT_OK;
        }
        CT_CUDA(cudaStreamSynchronize(ct->stream));  // the kernels before have read what is overwritten
        std::memcpy(host + (static_cast<char*>(dst) - base), src, n);
        return CT_OK;
    }
    // The counts of launch_check_tuples (waits for them).
    int counted(const ct_table* ct, unsigned long long (&c)[2]) {
        if (!host) CT_CUDA(cudaMemcpyAsync(c, counts, sizeof(c), cudaMemcpyDeviceToHost, ct->stream));
        CT_CUDA(cudaStreamSynchronize(ct->stream));
        if (host) std::memcpy(c, host, sizeof(c));
        return CT_OK;
    }
    // The chunk of `tuples` that starts at tuple j0 (nothing to do if it is there).
    int load(const ct_table* ct, const int32_t* tuples, int64_t t, int64_t j0) {
        if (held == tuples && heldAt == j0) return CT_OK;
        const int64_t m = std::min(cap, t - j0);
        const int st = put(ct, tup, tuples + j0 * ct->arity, (size_t)m * ct->arity * sizeof(int32_t));
        if (st != CT_OK) return st;
        held = tuples;
        heldAt = j0;
        return CT_OK;
    }
};

int build(ct_table* ct, const int32_t* dom_lo, const int32_t* dom_size, const int32_t* tuples, int64_t t,
          const ct_options* opt, bool negative) {
    const int n = ct->arity;
    ct->lo.assign(dom_lo, dom_lo + n);
    ct->size.assign(dom_size, dom_size + n);
    ct->nw.resize(n);
    ct->ld.resize(n);
    ct->row0.resize(n + 1);
    int DW = 0, R = 0;
    for (int i = 0; i < n; ++i) {
        ct->nw[i] = (ct->size[i] + 31) / 32;
        ct->ld[i] = DW;
        DW += ct->nw[i];
        ct->row0[i] = R;
        R += ct->size[i];
    }
    ct->row0[n] = R;
    ct->DW = DW;
    ct->R = R;
    ct->nChW = (n + 31) / 32;
    ct->rowVar.resize(R);
    for (int i = 0; i < n; ++i)
        for (int a = 0; a < ct->size[i]; ++a) ct->rowVar[ct->row0[i] + a] = i;

    // Retained tuples: every value inside its initial domain or a wildcard
    // (input order kept). A positive table's list is checked on the device, a
    // short one (kHostCheck components: less time than the device's answer
    // takes, about 20 us) here; a list that keeps all its tuples is used as it is.
    constexpr int64_t kHostCheck = 8192;
    ct->profile = opt && opt->profile;
    ct->copyState = opt && opt->copy_state;
    int st;
    int64_t nShort = 0;
    TupleStage stage;
    bool all = false;
    if (!negative && t * n > kHostCheck) {
        if ((st = stage.open(ct, t)) != CT_OK) return st;
        for (int64_t j0 = 0; j0 < t; j0 += stage.cap) {
            if ((st = stage.load(ct, tuples, t, j0)) != CT_OK) return st;
            CT_CUDA(launch_check_tuples(stage.tup, std::min(stage.cap, t - j0), n, stage.lo, stage.row0, stage.counts,
                                        ct->stream));
        }
        unsigned long long c[2] = {0, 0};
        if ((st = stage.counted(ct, c)) != CT_OK) return st;
        all = c[0] == 0;
        nShort = (int64_t)c[1];
    }
    std::vector<int64_t> keep;
    if (!all) {
        keep.reserve((size_t)t);
        nShort = 0;  // (counted again, over the retained tuples)
        for (int64_t j = 0; j < t; ++j) {
            const int32_t* tu = tuples + j * n;
            bool ok = true, star = false;
            for (int i = 0; i < n && ok; ++i) {
                if (tu[i] == CT_STAR) {
                    star = true;
                    continue;
                }
                const int64_t off = (int64_t)tu[i] - ct->lo[i];
                ok = off >= 0 && off < ct->size[i];
            }
            if (ok) {
                keep.push_back(j);
                nShort += star;
            }
        }
    }
    ct->shortTuples = nShort;
    if (negative) {
        // forbidden tuples: no wildcard, each counted once (the filter compares counts)
        if (nShort > 0) {
            ct_set_error("ct_create_negative: wildcards are not allowed in a negative table");
            return CT_ERR_ARG;
        }
        std::vector<std::pair<std::vector<int32_t>, int64_t>> keyed;
        keyed.reserve(keep.size());
        for (int64_t j : keep) keyed.push_back({std::vector<int32_t>(tuples + j * n, tuples + j * n + n), j});
        std::stable_sort(keyed.begin(), keyed.end(),
                         [](const auto& a, const auto& b) { return a.first < b.first; });
        for (size_t q = 1; q < keyed.size(); ++q)
            if (keyed[q].first == keyed[q - 1].first) keyed[q].second = -1 - keyed[q].second;
        std::vector<int64_t> drop;
        for (const auto& kv : keyed)
            if (kv.second < 0) drop.push_back(-1 - kv.second);
        std::sort(drop.begin(), drop.end());
        std::vector<int64_t> kept2;
        kept2.reserve(keep.size());
        for (int64_t j : keep)
            if (!std::binary_search(drop.begin(), drop.end(), j)) kept2.push_back(j);
        keep.swap(kept2);
        if (keep.empty()) {
            ct_set_error("ct_create_negative: a negative table needs at least one tuple inside the domains");
            return CT_ERR_ARG;
        }
        if (!(n <= kLocalMaxArity && ct->DW <= kLocalMaxDW && ct->R <= kCodeCap)) {
            ct_set_error("ct_create_negative: arity <= %d, <= %d domain words and <= %d values", kLocalMaxArity,
                         kLocalMaxDW, kCodeCap);
            return CT_ERR_ARG;
        }
        ct->negative = true;
    }
    std::vector<int32_t> packed;  // the retained tuples of a list that loses some
    all = all || (int64_t)keep.size() == t;
    if (!all) {
        packed.reserve(keep.size() * (size_t)n);
        for (int64_t j : keep) packed.insert(packed.end(), tuples + j * n, tuples + (j + 1) * n);
        tuples = packed.data();
    }
    ct->t = all ? t : (int64_t)keep.size();
    ct->W = (ct->t + 31) / 32;
    ct->W4 = (ct->W + 3) / 4;
    if (ct->t == 0) {
        ct->empty = true;
        return CT_INFEASIBLE;
    }
    if (ct->W4 > 0x3fffffffLL) {
        ct_set_error("too many tuples");
        return CT_ERR_ARG;
    }
    const int64_t W4 = ct->W4;
    ct->S = 32;
    ct->nseg = (int)((W4 + 31) / 32);
    ct->localPlan = n <= kLocalMaxArity && DW <= kLocalMaxDW && R <= kCodeCap;

    std::vector<uint32_t> hdom(DW, 0u);
    for (int i = 0; i < n; ++i)
        for (int a = 0; a < ct->size[i]; ++a) hdom[ct->ld[i] + a / 32] |= 1u << (a % 32);

    TableDev& d = ct->dev;
    uint4* sup = nullptr;
    int32_t *wordVar = nullptr, *rowVar = nullptr, *varRow0 = nullptr, *varNW = nullptr, *varLD = nullptr;
    uint4* supDel = nullptr;
    // currTable and lastpos are padded to whole 32-chunk segments.
    const size_t padChunks = (size_t)ct->nseg * 32;
    TableBufs bufs{ct, {}};
    bufs.want(&sup, (size_t)R * W4);
    if (nShort > 0) bufs.want(&supDel, (size_t)R * W4);
    bufs.want(&d.curr, padChunks);
    bufs.want(&d.segMask, (size_t)ct->nseg);
    bufs.want(&d.lastpos, padChunks);
    bufs.want(&d.residue, (size_t)R);
    bufs.want(&d.lastDom, (size_t)DW);
    bufs.want(&d.ctrl, 1);
    bufs.want(&d.codes, (size_t)R);
    bufs.want(&d.planK, (size_t)n);
    bufs.want(&d.planRowOff, (size_t)n);
    bufs.want(&d.varSup, (size_t)n);
    bufs.want(&d.other, (size_t)n);
    bufs.want(&d.hardRow, (size_t)R);
    bufs.want(&d.foundChunk, (size_t)R);
    bufs.want(&d.removed, (size_t)DW);
    bufs.want(&wordVar, (size_t)DW);
    bufs.want(&rowVar, (size_t)R);
    bufs.want(&varRow0, (size_t)n + 1);
    bufs.want(&varNW, (size_t)n);
    bufs.want(&varLD, (size_t)n);
    bufs.want(&ct->d_domScratch, (size_t)DW);
    st = bufs.take();
    if (st == CT_ERR_OOM && stage.base && !bufs.injected) {
        // the stage may be what is in the way: it comes back with what is left
        stage.close();
        st = bufs.take();
    }
    if (st != CT_OK) return st;
    if (nShort == 0) supDel = sup;
    ct->statusInts = (size_t)kStatusHdr + ct->nChW + DW;
    d.sup = sup;
    d.supDelta = supDel;
    d.negative = ct->negative ? 1 : 0;
    d.shard = (opt && opt->shard) ? 1 : 0;
    d.wordVar = wordVar;
    d.rowVar = rowVar;
    d.varRow0 = varRow0;
    d.varNW = varNW;
    d.varLD = varLD;
    d.arity = n;
    d.R = R;
    d.W4 = (int32_t)W4;
    d.nseg = ct->nseg;
    d.S = ct->S;
    d.DW = DW;
    d.nChangedWords = ct->nChW;
    d.useResidues = (opt && opt->no_residues) ? 0 : 1;
    const int maxNW = *std::max_element(ct->nw.begin(), ct->nw.end());
    while (maxNW > 2 && d.wordLanesLog < 5 && (1 << d.wordLanesLog) < maxNW) ++d.wordLanesLog;
    d.warpPlan = (!ct->negative && n <= 32) ? 1 : 0;
    for (int i = 0; i < n; ++i)
        if (ct->nw[i] > kWarpPlanWords) d.warpPlan = 0;
    for (int i = 0; i < n && i < kParamArity; ++i) {
        d.pNW[i] = ct->nw[i];
        d.pLD[i] = ct->ld[i];
        d.pRow0[i] = ct->row0[i];
    }
    ct->live = (int)W4;

    // The status block lives in mapped host memory: the kernel's last CTA writes
    // it directly and the host reads it after the stream synchronises.
    if (status_alloc((void**)&ct->h_status, ct->statusInts * sizeof(int32_t)) != cudaSuccess) {
        cudaGetLastError();
        ct->h_status = nullptr;
        ct_set_error("cudaHostAlloc of the status block failed");
        return CT_ERR_OOM;
    }
    std::memset(ct->h_status, 0, ct->statusInts * sizeof(int32_t));
    CT_CUDA(cudaHostGetDevicePointer((void**)&d.statusBlk, ct->h_status, 0));
    {
        // 16 loads in flight per lane at 2 CTAs per SM. With the row list of a
        // segment cut over up to kMaxSplit warps of a CTA, every segment can
        // keep a whole CTA busy: one CTA per segment (a long row list then
        // spreads over the whole grid), capped at residency, and at least one
        // warp per two values for the probes.
        ct->maxSplit = (opt && opt->no_split) ? 1 : kMaxSplit;
        ct->early = !(opt && opt->no_early_filter);
        const int narrow = (ct->localPlan ? 1 : 0);
        // more segments than one wave of warps at 2 CTAs per SM: 8 loads at 3 CTAs per SM
        const int maxNarrow = max_coresident_blocks(narrow);
        ct->variant = (ct->nseg > maxNarrow * kWarps) ? (narrow | 2) : narrow;
        // A warp per segment and one per value at one CTA per SM: the second CTA's
        // warps find nothing to do, and its registers are better used (32 calls,
        // one and two CTAs per SM: 25 segments of 192 values 671 and 686 us, 245
        // 701 and 735, 611 715 and 761, 977 725 and 768; a warp short of that, two
        // are better again: 1,197 segments 779 and 774, 1,465 818 and 773).
        if (ct->localPlan && !(opt && opt->grid_blocks > 0) &&
            ct->nseg + R <= max_coresident_blocks(kLoneVariant) * kWarps)
            ct->variant = kLoneVariant;
        const int maxCo = max_coresident_blocks(ct->variant);
        if (maxCo <= 0) {
            ct_set_error("ct_create: the propagation kernel cannot be made resident on this device");
            return CT_ERR_CUDA;
        }
        int want = (ct->nseg * ct->maxSplit + kWarps - 1) / kWarps;
        want = std::max(want, (R + 2 * kWarps - 1) / (2 * kWarps));
        // (a warp per value beside a warp per segment, up to 64 CTAs: 24 values
        // and 1 segment 575 -> 543 us per 32 calls, 192 values and 25 segments
        // 724 -> 691)
        want = std::max(want, std::min((ct->nseg + R + kWarps - 1) / kWarps, 64));
        if (opt && opt->grid_blocks > 0) want = opt->grid_blocks;
        ct->grid = std::max(1, std::min(want, maxCo));
        // (a launch shape that was asked for, or is to be tuned, is the general kernel's)
        ct->small = small_table(d) && !(opt && (opt->grid_blocks > 0 || opt->autotune));
        if (ct->small) ct->grid = 1;
    }

    // supports rows (Sec. 2), value-major, 16-byte aligned rows of W4 chunks (a
    // short tuple is in every row of its wildcard positions; the delta rows hold
    // only the tuples whose component equals the row's value)
    if (!stage.base && (st = stage.open(ct, ct->t)) != CT_OK) return st;
    for (int64_t j0 = 0; j0 < ct->t; j0 += stage.cap) {
        const int64_t m = std::min(stage.cap, ct->t - j0);
        if ((st = stage.load(ct, tuples, ct->t, j0)) != CT_OK) return st;
        CT_CUDA(launch_build_rows(stage.tup, m, n, stage.lo, stage.row0, sup, nShort > 0 ? supDel : nullptr, W4, j0,
                                  j0 + m == ct->t, ct->stream));
    }
    CT_CUDA(launch_build_state(d, ct->t, ct->stream));
    if ((st = upload(ct, d.lastDom, hdom)) != CT_OK) return st;
    std::vector<int32_t> hWordVar;
    hWordVar.reserve(DW);
    for (int i = 0; i < n; ++i) hWordVar.insert(hWordVar.end(), ct->nw[i], i);
    if ((st = upload(ct, wordVar, hWordVar)) != CT_OK) return st;
    if ((st = upload(ct, rowVar, ct->rowVar)) != CT_OK) return st;
    if ((st = upload(ct, varRow0, ct->row0)) != CT_OK) return st;
    if ((st = upload(ct, varNW, ct->nw)) != CT_OK) return st;
    if ((st = upload(ct, varLD, ct->ld)) != CT_OK) return st;
    CT_CUDA(cudaMemsetAsync(d.removed, 0, (size_t)DW * sizeof(uint32_t), ct->stream));
    CT_CUDA(cudaMemsetAsync(d.other, 0, (size_t)n * sizeof(unsigned long long), ct->stream));

    Ctrl c{};
    c.status = CT_OK;
    c.trail_top = 0;
    c.cur_mark = -1;
    c.trail_cap = 0;
    CT_CUDA(cudaMemcpyAsync(d.ctrl, &c, sizeof(Ctrl), cudaMemcpyHostToDevice, ct->stream));
    if ((st = sync(ct)) != CT_OK) return st;
    stage.close();
    if ((st = ensure_levels(ct, 8)) != CT_OK) return st;
    if (ct->profile) {
        if ((st = create_events(ct)) != CT_OK) return st;
    }
    return sync(ct);
}

void fill_stats(ct_table* ct) {
    const int32_t* h = ct->h_status;
    ct_call_stats& s = ct->last;
    s.status = h[kSlotStatus];
    s.changed_vars = h[kSlotNval];
    s.delta_vars = h[kSlotNdelta];
    s.reset_vars = h[kSlotNreset];
    s.rows_ored = h[kSlotRowsOred];
    s.sup_vars = h[kSlotNsup];
    s.residue_hits = h[kSlotHits];
    s.local_found = h[kSlotLocal];
    s.hard = h[kSlotHard];
    s.windows = h[kSlotWindows];
    s.pruned = h[kSlotPruned];
    s.trail_added = h[kSlotTrailAdded];
    s.live_chunks_in = (uint32_t)h[kSlotLiveIn];
    s.live_chunks_out = (uint32_t)h[kSlotLiveOut];
    s.live_words_in = (uint32_t)h[kSlotWordsIn];
    // Algorithmic bytes (what CT itself must move, 4-byte words): updateTable
    // reads k rows and currTable and writes currTable over the N live words;
    // filterDomains reads one word per residue hit, the windows it probes and
    // the whole live table for every value scanned (a negative table's: counted)
    // in full; a value that its windows decide costs no more than they do.
    s.update_bytes = s.rows_ored > 0 ? 4LL * s.live_words_in * (s.rows_ored + 2) : 0;
    s.filter_bytes = 4LL * s.residue_hits + 4LL * 128 * s.windows + 16LL * h[kSlotScan] * s.live_chunks_out;
    s.phase_ns[0] = h[kSlotT1];
    s.phase_ns[1] = h[kSlotT2];
    s.phase_ns[2] = h[kSlotT3];
    s.phase_ns[3] = h[kSlotT4];
    s.early_filter = h[kSlotEarly];
}

}  // namespace

// ---------------------------------------------------------------------------
// internal entry points for the model
// ---------------------------------------------------------------------------
namespace {

// Read the oldest pending event pair into the profile (waits for it).
int drain_event(ct_table* ct) {
    if (ct->evPending == 0) return CT_OK;
    const int slot = (ct->evNext - ct->evPending + ct_table::kEvRing) % ct_table::kEvRing;
    float a = 0.f;
    CT_CUDA(cudaEventSynchronize(ct->ev[2 * slot + 1]));
    CT_CUDA(cudaEventElapsedTime(&a, ct->ev[2 * slot], ct->ev[2 * slot + 1]));
    ct->prof.kernel_ms += a;
    ct->evPending -= 1;
    return CT_OK;
}

// copy_state ablation: the host copy of currTable, (re)read from the device.
int fetch_host_curr(ct_table* ct) {
    const size_t bytes = (size_t)ct->W4 * sizeof(uint4);
    if (!ct->h_curr && cudaHostAlloc((void**)&ct->h_curr, bytes, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        ct->h_curr = nullptr;
        ct_set_error("copy_state: pinned host copy of currTable");
        return CT_ERR_OOM;
    }
    CT_CUDA(cudaMemcpyAsync(ct->h_curr, ct->dev.curr, bytes, cudaMemcpyDeviceToHost, ct->stream));
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    return CT_OK;
}

int drain_events(ct_table* ct) {
    int st = CT_OK;
    while (ct->evPending > 0 && (st = drain_event(ct)) == CT_OK) {
    }
    return st;
}

}  // namespace

// domHost (host memory, the table's packed layout; local-plan tables with at
// most kParamDomWords domain words): the domains travel in the kernel
// parameters instead of `dom`, which may then be null; the filtered domains
// are in the status block when the call returns.
int ct_table_propagate_on(ct_table* ct, uint32_t* dom, const int32_t* domOffDev, const int32_t* domOffHost,
                          uint32_t* changed, const uint32_t* domHost) {
    if (!ct || (!dom && !domHost)) {
        ct_set_error("ct_propagate: null argument");
        return CT_ERR_ARG;
    }
    if (ct->empty) {
        ct->last = ct_call_stats{};
        ct->last.status = CT_INFEASIBLE;
        ct->failed = true;
        return CT_INFEASIBLE;
    }
    if (ct->broken) {
        ct_set_error("ct_propagate: the table is unusable after a device-side timeout");
        return CT_ERR_TIMEOUT;
    }
    if (ct->failed) {
        ct_set_error("ct_propagate: the previous call failed; restore a level first");
        return CT_ERR_STATE;
    }
    int st;
    if (!ct->levels.empty() && (st = ensure_trail(ct, (int64_t)ct->trailTop + ct->W4)) != CT_OK) return st;
    cudaStream_t s = ct->stream;
    int32_t* h = ct->h_status;
    volatile int32_t* hv = h;
    const auto t0 = std::chrono::steady_clock::now();
    CallParams P{};
    P.mark = ct->levels.empty() ? -1 : ct->levels.back().mark;
    P.snapFrom = ct->pendingFrom;
    P.snapTo = (int)ct->levels.size();
    P.prevLive = ct->live;
    P.spinLimit = kBarrierSpinLimit;
    P.maxSplit = ct->maxSplit;
    P.packed = domOffHost == ct->ld.data() ? 1 : 0;
    P.early = ct->early ? 16 : 0;
    for (int i = 0; i < ct->arity && i < kParamArity; ++i) P.domOff[i] = domOffHost[i];
    if (domHost) {
        if (!ct->localPlan || ct->DW > kParamDomWords) {
            ct_set_error("ct_propagate: domains in parameters need a local plan and <= %d words", kParamDomWords);
            return CT_ERR_ARG;
        }
        P.domInParams = 1;
        std::memcpy(P.domWords, domHost, (size_t)ct->DW * sizeof(uint32_t));
    }
    hv[kSlotStatus] = kNoChunk;  // overwritten by the kernel's last CTA
    P.trailTop = ct->trailTop;
    const bool small = ct->small && !ct->armPolls;  // (the hook is for the general kernel's barriers)
    if (ct->armPolls) {
        // Test hook (ct_arm_wait_timeout): an arrival count 2^30 behind every
        // target of this call (base 0), so no barrier completes and every wait
        // runs out after armPolls polls.
        const uint32_t unreachable[2] = {0xC0000000u, 0u};  // bar_count, bar_base
        static_assert(offsetof(Ctrl, bar_base) == offsetof(Ctrl, bar_count) + sizeof(uint32_t), "adjacent words");
        CT_CUDA(cudaMemcpyAsync(&ct->dev.ctrl->bar_count, unreachable, sizeof(unreachable), cudaMemcpyHostToDevice, s));
        P.spinLimit = ct->armPolls;
        ct->armPolls = 0;
    }
    if (ct->copyState) {
        // the paper's propagators copy currTable to the device before each call
        if (!ct->h_curr && (st = fetch_host_curr(ct)) != CT_OK) return st;
        CT_CUDA(cudaMemcpyAsync(ct->dev.curr, ct->h_curr, (size_t)ct->W4 * sizeof(uint4), cudaMemcpyHostToDevice, s));
    }
    int evSlot = 0;
    if (ct->profile) {
        if (ct->evPending == ct_table::kEvRing && (st = drain_event(ct)) != CT_OK) return st;
        evSlot = ct->evNext;
        CT_CUDA(cudaEventRecord(ct->ev[2 * evSlot], s));
    }
    CT_CUDA(small ? launch_small(ct->dev, dom, P, s)
                  : launch_propagate(ct->dev, ct->variant, ct->grid, dom, domOffDev, P, s));
    if (ct->profile) {
        CT_CUDA(cudaEventRecord(ct->ev[2 * evSlot + 1], s));
        ct->evNext = (ct->evNext + 1) % ct_table::kEvRing;
        ct->evPending += 1;
    }
    const auto t1 = std::chrono::steady_clock::now();
    ct->pendingFrom = (int)ct->levels.size();
    // Wait for the status word the kernel publishes last (bounded), then fall
    // back to a stream synchronisation to collect any CUDA error.
    // A kernel that returned without publishing (a barrier wait ran out) is
    // noticed when the stream has gone idle.
    bool seen = false;
    for (uint64_t it = 0;; ++it) {
        if (hv[kSlotStatus] != kNoChunk) {
            seen = true;
            break;
        }
        if ((it & 1023u) == 1023u) {
            if (cudaStreamQuery(s) == cudaSuccess) {
                seen = hv[kSlotStatus] != kNoChunk;
                break;
            }
            if (std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(kHostWaitMs)) break;
        }
    }
    if (!seen) CT_CUDA(cudaStreamSynchronize(s));
    std::atomic_thread_fence(std::memory_order_acquire);  // the results after the word that publishes them
    if (ct->copyState) {
        // ... and back to the host after it
        CT_CUDA(cudaMemcpyAsync(ct->h_curr, ct->dev.curr, (size_t)ct->W4 * sizeof(uint4), cudaMemcpyDeviceToHost, s));
        CT_CUDA(cudaStreamSynchronize(s));
    }
    const auto t2 = std::chrono::steady_clock::now();
    int status = hv[kSlotStatus];
    if (status == kNoChunk) {
        // The kernel returned before publishing: a grid barrier timed out.
        Ctrl c{};
        CT_CUDA(cudaMemcpy(&c, ct->dev.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost));
        status = c.status == CT_OK ? CT_ERR_TIMEOUT : c.status;
        c.bar_count = c.bar_base = 0;
        c.status = CT_OK;
        c.live = c.live_in = c.words_in = c.nhard = c.done = c.tuples = 0u;
        c.nscan = 0;
        c.upd_done = 0u;
        CT_CUDA(cudaMemcpy(ct->dev.ctrl, &c, sizeof(Ctrl), cudaMemcpyHostToDevice));
        ct->failed = true;
        ct->broken = true;
        ct->last = ct_call_stats{};
        ct->last.status = status;
        ct_set_error("ct_propagate: a device-side wait ran out (status %d)", status);
        return status;
    }
    fill_stats(ct);
    ct->trailTop = h[kSlotTrailTop];
    if (status == CT_OK) ct->live = h[kSlotLiveOut];
    if (ct->profile) {
        ct->prof.host_ms +=
            std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
        ct->prof.launch_ms += std::chrono::duration<double, std::milli>(t1 - t0).count();
        ct->prof.wait_ms += std::chrono::duration<double, std::milli>(t2 - t1).count();
        ct->prof.calls += 1;
        ct->prof.update_bytes += ct->last.update_bytes;
        ct->prof.filter_bytes += ct->last.filter_bytes;
        ct->prof.device_ms += ct->last.phase_ns[3] * 1e-6;
    }
    if (status == CT_INFEASIBLE) {
        ct->failed = true;
    } else if (status == CT_ERR_STATE) {
        ct_set_error("ct_propagate: a domain grew since the last call without a restore");
    } else if (status == CT_ERR_OOM) {
        ct->failed = true;
        ct_set_error("ct_propagate: trail overflow");
    } else if (status != CT_OK) {
        ct->failed = true;
        ct_set_error("ct_propagate: device status %d", status);
    }
    if (changed) {
        // The changed mask is only written when a value was pruned.
        if (status == CT_OK && h[kSlotPruned] > 0)
            std::memcpy(changed, h + kStatusHdr, (size_t)ct->nChW * sizeof(uint32_t));
        else
            std::memset(changed, 0, (size_t)ct->nChW * sizeof(uint32_t));
    }
    return status;
}

const int32_t* ct_table_status_host(const ct_table* ct) { return ct->h_status; }

// --- the batched network path (ct_model.cu) ---
int ct_table_is_empty(const ct_table* ct) { return ct->empty ? 1 : 0; }

int ct_table_grow_trail(ct_table* ct, int64_t need) { return ensure_trail(ct, need); }


namespace {

constexpr int kCloneLevels = 8;

int64_t clone_trail_entries(const ct_table* src) { return 2 * src->W4 + 64; }

size_t rnd256(size_t b) { return (std::max<size_t>(b, 1) + 255) & ~size_t(255); }

// Bytes of every dynamic buffer of a clone, in allocation order.
std::vector<size_t> clone_pieces(const ct_table* src) {
    const size_t padChunks = (size_t)src->nseg * 32;
    const size_t R = (size_t)src->R, n = (size_t)src->arity;
    const size_t tr = (size_t)clone_trail_entries(src);
    return {padChunks * sizeof(uint4), (size_t)src->nseg * 4, padChunks * 4, R * 4, (size_t)src->DW * 4, R * 4,
            n * 4, n * 4, n * 4, n * 8, R * 4, R * 4,
            (size_t)kCloneLevels * std::max(src->nseg, 1) * 4, (size_t)kCloneLevels * std::max(src->DW, 1) * 4,
            tr * sizeof(int2), tr * sizeof(uint4)};
}

}  // namespace

size_t ct_table_clone_bytes(const ct_table* src) {
    size_t b = 0;
    for (size_t p : clone_pieces(src)) b += rnd256(p);
    return b + 256;
}

// A table that shares `src`'s static buffers (supports rows and the layout
// tables, which stay owned by src) with dynamic buffers of its own (currTable,
// index, lastDom, residues, trail, levels), filled by launch_clone_state. Used
// for the independent search nodes of a batched search. The dynamic buffers, 8
// levels and a first trail come out of the arena in one piece; a trail or level
// stack that outgrows them moves to its own allocation.
ct_table* ct_table_clone(const ct_table* src, cudaStream_t stream, DeviceArena& arena, Ctrl* ctrl, int* status) {
    *status = CT_ERR_ARG;
    if (!src || src->empty) return nullptr;
    ct_table* ct = new (std::nothrow) ct_table();
    if (!ct) {
        *status = CT_ERR_OOM;
        return nullptr;
    }
    ct->arity = src->arity;
    ct->lo = src->lo;
    ct->size = src->size;
    ct->nw = src->nw;
    ct->ld = src->ld;
    ct->row0 = src->row0;
    ct->rowVar = src->rowVar;
    ct->R = src->R;
    ct->t = src->t;
    ct->W = src->W;
    ct->W4 = src->W4;
    ct->nseg = src->nseg;
    ct->S = src->S;
    ct->grid = src->grid;
    ct->DW = src->DW;
    ct->nChW = src->nChW;
    ct->localPlan = src->localPlan;
    ct->variant = src->variant;
    ct->maxSplit = src->maxSplit;
    ct->early = src->early;
    ct->live = src->live;
    ct->stream = stream;
    ct->dev = src->dev;  // static pointers shared; dynamic ones replaced below
    TableDev& d = ct->dev;
    d.trailKey = nullptr;
    d.trailOld = nullptr;
    d.levelSeg = nullptr;
    d.levelDom = nullptr;
    d.statusBlk = src->dev.statusBlk;  // never written by the batched path; kept valid
    const std::vector<size_t> pc = clone_pieces(src);
    void* p[16];
    for (int i = 0; i < 16; ++i) {
        p[i] = arena.take(pc[i]);
        if (!p[i]) {
            free_table(ct);
            ct_set_error("clone arena exhausted");
            *status = CT_ERR_OOM;
            return nullptr;
        }
    }
    d.curr = static_cast<uint4*>(p[0]);
    d.segMask = static_cast<uint32_t*>(p[1]);
    d.lastpos = static_cast<int32_t*>(p[2]);
    d.residue = static_cast<int32_t*>(p[3]);
    d.lastDom = static_cast<uint32_t*>(p[4]);
    d.codes = static_cast<int32_t*>(p[5]);
    d.planK = static_cast<int32_t*>(p[6]);
    d.planRowOff = static_cast<int32_t*>(p[7]);
    d.varSup = static_cast<int32_t*>(p[8]);
    d.other = static_cast<unsigned long long*>(p[9]);
    d.hardRow = static_cast<int32_t*>(p[10]);
    d.foundChunk = static_cast<int32_t*>(p[11]);
    d.levelSeg = static_cast<uint32_t*>(p[12]);
    d.levelDom = static_cast<uint32_t*>(p[13]);
    d.trailKey = static_cast<int2*>(p[14]);
    d.trailOld = static_cast<uint4*>(p[15]);
    ct->levelCap = kCloneLevels;
    ct->levelsInArena = true;
    ct->trailCap = (int)clone_trail_entries(src);
    ct->trailInArena = true;
    d.ctrl = ctrl;
    *status = CT_OK;
    return ct;
}

int ct_table_trail_cap(const ct_table* ct) { return ct->trailCap; }

// Host side of a clone taking its source's state (the device side is
// launch_clone_state): empty trail, no levels, the source's live count.
void ct_table_adopt_state(ct_table* dst, const ct_table* src) {
    dst->live = src->live;
    dst->trailTop = 0;
    dst->levels.clear();
    dst->pendingFrom = 0;
    dst->failed = false;
}

int ct_table_live(const ct_table* ct) { return ct->live; }

void ct_table_free(ct_table* ct) { free_table(ct); }


int ct_table_depth(const ct_table* ct) { return (int)ct->levels.size(); }

int ct_table_restore_device(ct_table* ct, const RestoreDesc& d) {
    CT_CUDA(launch_restore(ct->dev, d.level, d.mark, d.top, -1, ct->stream));
    return CT_OK;
}

int ct_table_dom_words(const ct_table* ct) { return ct->DW; }
const int32_t* ct_table_var_ld(const ct_table* ct) { return ct->ld.data(); }
int ct_table_changed_words(const ct_table* ct) { return ct->nChW; }

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
namespace {

// Launch-shape autotuner: time trial propagations of every candidate shape
// (row loads in flight x CTA count) between a save and a restore, keep the
// fastest. Trials: a delta call (one value of the largest domain removed) and
// a reset call (every domain cut to a quarter); the score is the sum of their
// best-of-3 host-observed latencies (launch to published result).
int autotune(ct_table* ct) {
    if (ct->empty || ct->R < 1) return CT_OK;
    const int narrow = ct->localPlan ? 1 : 0;
    const int base = std::max((ct->nseg * ct->maxSplit + kWarps - 1) / kWarps, (ct->R + 2 * kWarps - 1) / (2 * kWarps));
    std::vector<std::pair<int, int>> cands;
    for (int wide = 0; wide < 2; ++wide) {
        const int var = wide ? narrow | 2 : ct->variant == kLoneVariant ? kLoneVariant : narrow;
        const int maxCo = max_coresident_blocks(var);
        if (maxCo <= 0) continue;
        for (int g : {base / 4, base / 2, base, 2 * base, maxCo / 2, maxCo}) {
            g = std::max(1, std::min(g, maxCo));
            if (std::find(cands.begin(), cands.end(), std::make_pair(var, g)) == cands.end()) cands.push_back({var, g});
        }
    }
    if (cands.empty()) return CT_OK;
    // trial domains in the table's packed layout
    std::vector<uint32_t> full((size_t)ct->DW, 0u), delta, reset;
    int big = 0;
    for (int i = 0; i < ct->arity; ++i) {
        for (int a = 0; a < ct->size[i]; ++a) full[(size_t)ct->ld[i] + a / 32] |= 1u << (a % 32);
        if (ct->size[i] > ct->size[big]) big = i;
    }
    delta = full;
    reset = full;
    if (ct->size[big] > 1) delta[(size_t)ct->ld[big]] &= ~1u;
    for (int i = 0; i < ct->arity; ++i) {
        const int keep = std::max(1, ct->size[i] / 4);
        for (int a = keep; a < ct->size[i]; ++a) reset[(size_t)ct->ld[i] + a / 32] &= ~(1u << (a % 32));
    }
    const int saveVar = ct->variant, saveGrid = ct->grid;
    const bool saveProfile = ct->profile;
    ct->profile = false;
    int L = 0;
    int st = ct_save(ct, &L);
    if (st != CT_OK) return st;
    double best = 1e30;
    int bestVar = saveVar, bestGrid = saveGrid;
    for (const auto& c : cands) {
        ct->variant = c.first;
        ct->grid = c.second;
        double score = 0.0;
        for (const std::vector<uint32_t>* trial : {&delta, &reset}) {
            double tmin = 1e30;
            for (int rep = 0; rep < 3 && st == CT_OK; ++rep) {
                CT_CUDA(cudaMemcpyAsync(ct->d_domScratch, trial->data(), trial->size() * sizeof(uint32_t),
                                        cudaMemcpyHostToDevice, ct->stream));
                CT_CUDA(cudaStreamSynchronize(ct->stream));
                const auto t0 = std::chrono::steady_clock::now();
                const int r = ct_table_propagate_on(ct, ct->d_domScratch, ct->dev.varLD, ct->ld.data(), nullptr);
                const double dt = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
                if (r < 0) st = r;
                tmin = std::min(tmin, dt);
                if (st == CT_OK && (st = ct_restore(ct, L)) == CT_OK) st = ct_save(ct, &L);
            }
            score += tmin;
        }
        if (st != CT_OK) break;
        if (score < best) {
            best = score;
            bestVar = c.first;
            bestGrid = c.second;
        }
    }
    const int rs = ct_restore(ct, L);
    ct->variant = st == CT_OK ? bestVar : saveVar;
    ct->grid = st == CT_OK ? bestGrid : saveGrid;
    ct->profile = saveProfile;
    ct->prof = ct_profile{};
    ct->autotuned = st == CT_OK;
    return st != CT_OK ? st : rs;
}

}  // namespace

namespace {
int create_impl(int arity, const int32_t* dom_lo, const int32_t* dom_size, const int32_t* tuples, int64_t t,
                const ct_options* opt, void* cuda_stream, ct_table** out, bool negative);
}  // namespace

extern "C" int ct_debug_guard_buffers(int on) {
    std::lock_guard<std::mutex> lk(g_bufMu);
    g_guardNew = on != 0;
    return CT_OK;
}

extern "C" int ct_debug_fail_alloc(int n) {
    std::lock_guard<std::mutex> lk(g_bufMu);
    g_failAfter = n < 0 ? -1 : n;
    return CT_OK;
}

extern "C" int ct_debug_limit_bytes(int64_t bytes) {
    std::lock_guard<std::mutex> lk(g_bufMu);
    g_limitBytes = bytes < 0 ? -1 : bytes;
    return CT_OK;
}

extern "C" int ct_debug_device_bytes(int64_t* bytes_out) {
    if (!bytes_out) {
        ct_set_error("ct_debug_device_bytes: bytes_out is null");
        return CT_ERR_ARG;
    }
    std::lock_guard<std::mutex> lk(g_bufMu);
    *bytes_out = g_bufBytes;
    return CT_OK;
}

extern "C" int ct_debug_check_guards(ct_table* ct, int poke, int64_t* changed_out) {
    if (!ct || !changed_out || poke < 0 || poke > (int)kGuardBytes) {
        ct_set_error("ct_debug_check_guards: a table, changed_out, and 0 <= poke <= %d", (int)kGuardBytes);
        return CT_ERR_ARG;
    }
    if (ct->stream) CT_CUDA(cudaStreamSynchronize(ct->stream));
    std::vector<void*> bufs(ct->allocs.begin(), ct->allocs.end());
    if (!ct->trailInArena) {
        bufs.push_back(ct->dev.trailKey);
        bufs.push_back(ct->dev.trailOld);
    }
    if (!ct->levelsInArena) {
        bufs.push_back(ct->dev.levelSeg);
        bufs.push_back(ct->dev.levelDom);
    }
    std::vector<std::pair<char*, size_t>> guarded;
    {
        std::lock_guard<std::mutex> lk(g_bufMu);
        for (void* b : bufs) {
            const auto it = b ? g_bufs.find(b) : g_bufs.end();
            if (it != g_bufs.end() && it->second.guarded) guarded.emplace_back(static_cast<char*>(b), it->second.bytes);
        }
    }
    if (poke > 0 && !guarded.empty())
        CT_CUDA(cudaMemset(guarded[0].first - kGuardBytes, 0, (size_t)poke));  // from the host: no kernel writes it
    CT_CUDA(cudaDeviceSynchronize());
    int64_t changed = 0;
    std::vector<unsigned char> h(kGuardBytes);
    for (const auto& g : guarded) {
        for (int side = 0; side < 2; ++side) {
            const char* at = side == 0 ? g.first - kGuardBytes : g.first + g.second;
            CT_CUDA(cudaMemcpy(h.data(), at, kGuardBytes, cudaMemcpyDeviceToHost));
            for (unsigned char c : h) changed += c != kGuardFill;
        }
    }
    *changed_out = changed;
    return CT_OK;
}

extern "C" int ct_create(int arity, const int32_t* dom_lo, const int32_t* dom_size, const int32_t* tuples,
                         int64_t t, const ct_options* opt, void* cuda_stream, ct_table** out) {
    return create_impl(arity, dom_lo, dom_size, tuples, t, opt, cuda_stream, out, false);
}

extern "C" int ct_create_negative(int arity, const int32_t* dom_lo, const int32_t* dom_size, const int32_t* tuples,
                                  int64_t t, const ct_options* opt, void* cuda_stream, ct_table** out) {
    return create_impl(arity, dom_lo, dom_size, tuples, t, opt, cuda_stream, out, true);
}

int ct_table_is_negative(const ct_table* ct) { return ct->negative ? 1 : 0; }

namespace {
int create_impl(int arity, const int32_t* dom_lo, const int32_t* dom_size, const int32_t* tuples, int64_t t,
                const ct_options* opt, void* cuda_stream, ct_table** out, bool negative) {
    if (!out) {
        ct_set_error("ct_create: out is null");
        return CT_ERR_ARG;
    }
    *out = nullptr;
    if (arity < 1 || arity > kMaxArity || !dom_lo || !dom_size || t < 0 || (t > 0 && !tuples)) {
        ct_set_error("ct_create: invalid arity/domains/tuples (arity %d, t %lld)", arity, (long long)t);
        return CT_ERR_ARG;
    }
    for (int i = 0; i < arity; ++i) {
        if (dom_size[i] < 1 || dom_size[i] > kMaxDomSize) {
            ct_set_error("ct_create: dom_size[%d] = %d out of [1, %d]", i, dom_size[i], kMaxDomSize);
            return CT_ERR_ARG;
        }
    }
    if (negative && opt && opt->shard) {
        ct_set_error("ct_create_negative: negative tables cannot be shards");
        return CT_ERR_ARG;
    }
    ct_table* ct = new (std::nothrow) ct_table();
    if (!ct) return CT_ERR_OOM;
    ct->arity = arity;
    if (cuda_stream) {
        ct->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        const cudaError_t e = cudaStreamCreateWithFlags(&ct->stream, cudaStreamNonBlocking);
        if (e != cudaSuccess) {
            delete ct;
            return ct_cuda_fail(e, "cudaStreamCreateWithFlags");
        }
        ct->ownStream = true;
    }
    const int st = build(ct, dom_lo, dom_size, tuples, t, opt, negative);
    if (st < 0) {
        free_table(ct);
        return st;
    }
    if (st == CT_OK && opt && opt->autotune && opt->grid_blocks <= 0) {
        const int at = autotune(ct);
        if (at < 0) {
            free_table(ct);
            return at;
        }
    }
    *out = ct;
    return st;
}
}  // namespace

extern "C" int ct_propagate(ct_table* ct, uint32_t* dom_bits, uint32_t* changed_vars) {
    if (!ct) {
        ct_set_error("ct_propagate: null handle");
        return CT_ERR_ARG;
    }
    return ct_table_propagate_on(ct, dom_bits, ct->dev.varLD, ct->ld.data(), changed_vars);
}

extern "C" int ct_arm_wait_timeout(ct_table* ct, uint32_t polls) {
    if (polls == 0) {
        ct_set_error("ct_arm_wait_timeout: polls must be positive");
        return CT_ERR_ARG;
    }
    if (!ct) return ct_noalloc_arm_wait_timeout(polls);
    ct->armPolls = polls;
    return CT_OK;
}

extern "C" int ct_propagate_host(ct_table* ct, uint32_t* dom_bits_host, uint32_t* changed_vars) {
    if (!ct || !dom_bits_host) {
        ct_set_error("ct_propagate_host: null argument");
        return CT_ERR_ARG;
    }
    if (ct->empty) return ct_table_propagate_on(ct, dom_bits_host, nullptr, nullptr, changed_vars);
    int st;
    if (ct->localPlan && ct->DW <= kParamDomWords && !ct->copyState) {
        // a few domain words: they go to the device with the launch itself
        st = ct_table_propagate_on(ct, nullptr, ct->dev.varLD, ct->ld.data(), changed_vars, dom_bits_host);
    } else {
        CT_CUDA(cudaMemcpyAsync(ct->d_domScratch, dom_bits_host, (size_t)ct->DW * sizeof(uint32_t),
                                cudaMemcpyHostToDevice, ct->stream));
        st = ct_table_propagate_on(ct, ct->d_domScratch, ct->dev.varLD, ct->ld.data(), changed_vars);
    }
    if (st == CT_OK && ct->h_status[kSlotPruned] > 0) {
        // Only the variables that lost values differ from the input.
        const int32_t* h = ct->h_status;
        const uint32_t* outDom = reinterpret_cast<const uint32_t*>(h + kStatusHdr + ct->nChW);
        for (int i = 0; i < ct->arity; ++i) {
            if (!(((uint32_t)h[kStatusHdr + (i >> 5)] >> (i & 31)) & 1u)) continue;
            std::memcpy(dom_bits_host + ct->ld[i], outDom + ct->ld[i], (size_t)ct->nw[i] * sizeof(uint32_t));
        }
    }
    return st;
}

extern "C" int ct_save(ct_table* ct, int* level_out) {
    if (!ct) {
        ct_set_error("ct_save: null handle");
        return CT_ERR_ARG;
    }
    if (ct->failed) {
        ct_set_error("ct_save: the previous call failed; restore a level first");
        return CT_ERR_STATE;
    }
    const int L = (int)ct->levels.size();
    if (!ct->empty) {
        int st;
        if ((st = ensure_levels(ct, L + 1)) != CT_OK) return st;
    }
    // The snapshot itself is taken by the next propagation (or never, if the
    // level is restored before any propagation changed the state).
    ct->levels.push_back(ct_table::Level{ct->trailTop, ct->live, L});
    if (level_out) *level_out = L;
    return CT_OK;
}

extern "C" int ct_restore(ct_table* ct, int level) {
    if (!ct) {
        ct_set_error("ct_restore: null handle");
        return CT_ERR_ARG;
    }
    if (level < 0 || level >= (int)ct->levels.size()) {
        ct_set_error("ct_restore: level %d not in [0, %d)", level, (int)ct->levels.size());
        return CT_ERR_LEVEL;
    }
    if (ct->broken) {
        ct_set_error("ct_restore: the table is unusable after a device-side timeout");
        return CT_ERR_TIMEOUT;
    }
    const int mark = ct->levels[level].mark;
    if (!ct->empty && level < ct->pendingFrom) {
        CT_CUDA(launch_restore(ct->dev, ct->levels[level].snap, mark, ct->trailTop, -1, ct->stream));
        ct->trailTop = mark;
        if (ct->copyState && ct->h_curr) {
            const int st = fetch_host_curr(ct);
            if (st != CT_OK) return st;
        }
    }
    // A level saved after the last propagation still equals the current state.
    ct->failed = false;
    ct->live = ct->levels[level].live;
    ct->levels.resize(level);
    ct->pendingFrom = std::min(ct->pendingFrom, level);
    return CT_OK;
}

extern "C" int ct_get_currtable(ct_table* ct, uint32_t* words_host, int64_t* nonzero_words_out) {
    if (!ct) {
        ct_set_error("ct_get_currtable: null handle");
        return CT_ERR_ARG;
    }
    if (ct->empty) {
        if (nonzero_words_out) *nonzero_words_out = 0;
        return CT_OK;
    }
    // straight into the caller's words; the non-zero ones are counted there, or
    // from 24,576 words on by a kernel before the copy (the loop takes 0.32 ns a
    // word, 7.9 us there and 101 us for 312,500, where the kernel adds 7.7)
    const bool onDevice = nonzero_words_out && ct->W >= 24576;
    std::vector<uint32_t> buf;
    if (!words_host && nonzero_words_out && !onDevice) {
        buf.resize((size_t)ct->W);
        words_host = buf.data();
    }
    if (onDevice) CT_CUDA(launch_count_words(ct->dev, ct->stream));
    if (words_host)
        CT_CUDA(cudaMemcpyAsync(words_host, ct->dev.curr, (size_t)ct->W * sizeof(uint32_t), cudaMemcpyDeviceToHost,
                                ct->stream));
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    if (onDevice) {
        *nonzero_words_out = (uint32_t)ct->h_status[kSlotWords];
    } else if (nonzero_words_out) {
        int64_t nz = 0;
        for (int64_t w = 0; w < ct->W; ++w) nz += words_host[w] != 0u;
        *nonzero_words_out = nz;
    }
    return CT_OK;
}

extern "C" int ct_get_support_row(ct_table* ct, int row, uint32_t* words_host) {
    if (!ct || !words_host || row < 0 || row >= ct->R) {
        ct_set_error("ct_get_support_row: bad argument");
        return CT_ERR_ARG;
    }
    if (ct->empty) return CT_OK;
    CT_CUDA(cudaMemcpyAsync(words_host, ct->dev.sup + (size_t)row * ct->W4, (size_t)ct->W * sizeof(uint32_t),
                            cudaMemcpyDeviceToHost, ct->stream));
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    return CT_OK;
}

extern "C" int ct_get_index(ct_table* ct, int32_t* index_host, int64_t* count_out) {
    if (!ct) {
        ct_set_error("ct_get_index: null handle");
        return CT_ERR_ARG;
    }
    if (ct->empty) {
        if (count_out) *count_out = 0;
        return CT_OK;
    }
    std::vector<uint32_t> mask(ct->nseg);
    CT_CUDA(cudaMemcpyAsync(mask.data(), ct->dev.segMask, mask.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost,
                            ct->stream));
    CT_CUDA(cudaStreamSynchronize(ct->stream));
    int64_t n = 0;
    for (int s = 0; s < ct->nseg; ++s) {
        for (int j = 0; j < 32; ++j) {
            if (!((mask[s] >> j) & 1u)) continue;
            if (index_host) index_host[n] = s * 32 + j;
            ++n;
        }
    }
    if (count_out) *count_out = n;
    return CT_OK;
}

extern "C" int ct_get_info(ct_table* ct, ct_table_info* info) {
    if (!ct || !info) {
        ct_set_error("ct_get_info: null argument");
        return CT_ERR_ARG;
    }
    ct_table_info r{};
    r.arity = ct->arity;
    r.rows = ct->R;
    r.tuples = ct->t;
    r.words = ct->W;
    r.chunks = ct->W4;
    r.segments = ct->nseg;
    r.seg_capacity = ct->S;
    r.trail_size = ct->trailTop;
    r.depth = (int)ct->levels.size();
    r.local_plan = ct->localPlan ? 1 : 0;
    r.grid_blocks = ct->grid;
    r.short_tuples = (int32_t)std::min<int64_t>(ct->shortTuples, 0x7fffffff);
    r.loads_in_flight = (ct->variant & 2) ? 8 : 16;
    r.autotuned = ct->autotuned ? 1 : 0;
    r.device_bytes = ct->deviceBytes;
    int64_t live = 0;
    const int st = ct_get_index(ct, nullptr, &live);
    if (st != CT_OK) return st;
    r.live_chunks = live;
    *info = r;
    return CT_OK;
}

extern "C" int ct_get_call_stats(ct_table* ct, ct_call_stats* stats) {
    if (!ct || !stats) {
        ct_set_error("ct_get_call_stats: null argument");
        return CT_ERR_ARG;
    }
    *stats = ct->last;
    return CT_OK;
}

extern "C" int ct_get_profile(ct_table* ct, ct_profile* prof) {
    if (!ct || !prof) {
        ct_set_error("ct_get_profile: null argument");
        return CT_ERR_ARG;
    }
    const int st = drain_events(ct);
    if (st != CT_OK) return st;
    *prof = ct->prof;
    return CT_OK;
}

extern "C" int ct_set_profile(ct_table* ct, int on) {
    if (!ct) {
        ct_set_error("ct_set_profile: null handle");
        return CT_ERR_ARG;
    }
    if (on && ct->ev.empty()) {
        const int st = create_events(ct);
        if (st != CT_OK) return st;
    }
    if (!on) {
        const int st = drain_events(ct);
        if (st != CT_OK) return st;
    }
    ct->profile = on != 0;
    return CT_OK;
}

extern "C" int ct_reset_profile(ct_table* ct) {
    if (!ct) return CT_ERR_ARG;
    const int st = drain_events(ct);
    ct->prof = ct_profile{};
    return st;
}

extern "C" int ct_destroy(ct_table* ct) {
    free_table(ct);
    return CT_OK;
}
