// Host side of the kvsched C-ABI (see include/kvsched.h for the contract of every entry point).
// All scheduling arithmetic runs in the kernels of k1_* .. k7_*; this
// file validates arguments, owns device memory and enqueues launches.  There is no CPU fallback.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <mutex>
#include <new>
#include <type_traits>
#include <unordered_map>
#include <vector>

#include "common.cuh"
#include "k1_sort.cuh"
#include "k2_fmetric.cuh"
#include "k2_local_swap.cuh"
#include "k2_dp.cuh"
#include "k2_quantile.cuh"
#include "k3_eval.cuh"
#include "k3_lanes.cuh"
#include "k3_policy.cuh"
#include "k5_argmin.cuh"
#include "k6_online.cuh"
#include "k7_amin.cuh"

thread_local char g_last_cuda_error[256] = "";

int kv_cuda_fail(cudaError_t e, const char* what) {
    snprintf(g_last_cuda_error, sizeof(g_last_cuda_error), "%s: %s", what, cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? SCHED_E_NOMEM : SCHED_E_CUDA;
}

namespace {

const i64 kSweepChunk = 1ll << 22;          // candidates per launch inside a sweep
const int kResultBad = 9;                   // word of d_result: the candidates of a host call are not what they should be
const int kDeviceCheckMax = 1 << 20;        // requests whose bits fit a CTA's shared memory
const i64 kHostCheckMax = 1 << 13;          // ids or starts checked by the host: 8 us, a launch and a read-back 13
const i64 kAcceptSmall = 16384;              // sweep results that one CTA reduces (4 us against a launch of its own)
const int kSnapshots = 256;                 // states of the base run kept for the sweeps (chunked simulator)
const int kLeadingFrom = 2048;              // requests from which the quantile solver's keys are made beforehand: 2 and more per thread
const size_t kLeadingBytes = 64ull << 20;   // of them, at most; without them where that is not all batches there may well be
const int kSnapStrideHyb = 8;               // positions per state (hybrid simulator)
const size_t kSnapBudget = 512ull << 20;    // bytes of snapshot memory

// Runs CALL(SIM) with SIM = the simulator class of the handle: the chunked one (NM far registers per
// lane for decodes up to 1,025 / 2,049 / 4,097 / 8,193 rounds), beyond that the hybrid one, whose
// per-lane state does not grow with the longest decode.
#define KV_DISPATCH_SIM(h, CALL)                               \
    switch ((h)->nm) {                                          \
        case 1: CALL(ChunkSim<1>); break;                       \
        case 2: CALL(ChunkSim<2>); break;                       \
        case 4: CALL(ChunkSim<4>); break;                       \
        case 8: CALL(ChunkSim<8>); break;                       \
        default: CALL(HybSim); break;                           \
    }

int bits_of(u64 v) { int b = 0; while (v) { ++b; v >>= 1; } return b; }

// ------------------------------------------------------------------------------------------------
// Device-memory cache.  Creating and destroying a handle allocates and frees a few hundred MB (base
// run snapshots, staging, per-candidate scratch); cudaFree of such blocks was seen to take from 2 ms
// to more than half a second on a busy machine.  Blocks of at least 1 MiB therefore go back to a
// process-wide per-device free list (at most KVSCHED_POOL_MB MiB in total, default 1024, 0 turns the
// cache off) and are handed out again to later requests of similar size.  kv_free() waits for the
// device first, exactly as cudaFree does, so a cached block is never still in use.
// sched_release_cached_memory() returns everything to the driver.
// ------------------------------------------------------------------------------------------------
struct PoolBlock { void* p; size_t bytes; int device; };
std::mutex g_pool_mu;
std::vector<PoolBlock> g_pool_free;
std::unordered_map<void*, PoolBlock> g_pool_live;
size_t g_pool_cached = 0;
const size_t kPoolMinBlock = 1ull << 20;

size_t pool_cap_bytes() {
    static const size_t cap = [] {
        const char* e = getenv("KVSCHED_POOL_MB");
        const long long mb = e ? atoll(e) : 1024;
        return (size_t)(mb < 0 ? 0 : mb) << 20;
    }();
    return cap;
}

void pool_trim_locked(int device) {             // device < 0: every device
    for (size_t k = 0; k < g_pool_free.size();) {
        if (device < 0 || g_pool_free[k].device == device) {
            cudaFree(g_pool_free[k].p);
            g_pool_cached -= g_pool_free[k].bytes;
            g_pool_free[k] = g_pool_free.back();
            g_pool_free.pop_back();
        } else {
            ++k;
        }
    }
}

cudaError_t kv_malloc(void** out, size_t bytes) {
    *out = nullptr;
    if (const char* least = getenv("KVSCHED_REFUSE_MB"))        // testing knob: there is no memory for blocks of this size and more
        if (bytes >= (size_t)atoll(least) << 20) return cudaErrorMemoryAllocation;
    if (bytes < kPoolMinBlock || pool_cap_bytes() == 0) return cudaMalloc(out, bytes);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const size_t want = (bytes + (kPoolMinBlock - 1)) & ~(kPoolMinBlock - 1);
    std::lock_guard<std::mutex> lock(g_pool_mu);
    int best = -1;
    for (size_t k = 0; k < g_pool_free.size(); ++k) {
        const PoolBlock& b = g_pool_free[k];
        if (b.device == dev && b.bytes >= want && b.bytes <= 2 * want && (best < 0 || b.bytes < g_pool_free[best].bytes))
            best = (int)k;
    }
    if (best >= 0) {
        const PoolBlock b = g_pool_free[best];
        g_pool_free[best] = g_pool_free.back();
        g_pool_free.pop_back();
        g_pool_cached -= b.bytes;
        g_pool_live[b.p] = b;
        *out = b.p;
        return cudaSuccess;
    }
    e = cudaMalloc(out, want);
    if (e == cudaErrorMemoryAllocation) {       // give the cached blocks back and try once more
        cudaGetLastError();
        pool_trim_locked(dev);
        e = cudaMalloc(out, want);
    }
    if (e == cudaSuccess) g_pool_live[*out] = PoolBlock{*out, want, dev};
    return e;
}

void kv_free(void* p) {
    if (!p) return;
    std::unique_lock<std::mutex> lock(g_pool_mu);
    auto it = g_pool_live.find(p);
    if (it == g_pool_live.end()) { lock.unlock(); cudaFree(p); return; }
    const PoolBlock b = it->second;
    g_pool_live.erase(it);
    if (g_pool_cached + b.bytes > pool_cap_bytes()) { lock.unlock(); cudaFree(p); return; }
    lock.unlock();
    int prev = -1;
    cudaGetDevice(&prev);
    if (prev != b.device) cudaSetDevice(b.device);
    cudaDeviceSynchronize();                    // what cudaFree would have waited for
    if (prev != b.device && prev >= 0) cudaSetDevice(prev);
    lock.lock();
    g_pool_free.push_back(b);
    g_pool_cached += b.bytes;
}

// Pinned host memory of the handles' read-backs, cached like the device blocks (at most 64 MiB).
struct PinnedBlock { void* p; size_t bytes; };
std::vector<PinnedBlock> g_pinned_free;
size_t g_pinned_cached = 0;
const size_t kPinnedCap = 64ull << 20;

cudaError_t kv_host_malloc(void** out, size_t* bytes) {        // rounds *bytes up
    size_t want = 4096;
    while (want < *bytes) want <<= 1;
    *bytes = want;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        for (size_t k = 0; k < g_pinned_free.size(); ++k)
            if (g_pinned_free[k].bytes == want) {
                *out = g_pinned_free[k].p;
                g_pinned_cached -= want;
                g_pinned_free[k] = g_pinned_free.back();
                g_pinned_free.pop_back();
                return cudaSuccess;
            }
    }
    return cudaHostAlloc(out, want, cudaHostAllocPortable);
}
// no copy from or to the block may be in flight
void kv_host_free(void* p, size_t bytes) {
    if (!p) return;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        if (g_pinned_cached + bytes <= kPinnedCap) {
            g_pinned_free.push_back(PinnedBlock{p, bytes});
            g_pinned_cached += bytes;
            return;
        }
    }
    cudaFreeHost(p);
}

template <typename T>
int dev_alloc(T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    KV_CUDA(kv_malloc((void**)p, count * sizeof(T)));
    return SCHED_OK;
}

int ensure_stage(sched_ctx* h, size_t bytes) {
    if (h->stage_cap >= bytes) return SCHED_OK;
    if (h->d_stage) { kv_free(h->d_stage); h->d_stage = nullptr; h->stage_cap = 0; }
    KV_CUDA(kv_malloc((void**)&h->d_stage, bytes));
    h->stage_cap = bytes;
    return SCHED_OK;
}

int ensure_tel(sched_ctx* h, i64 count) {
    if (h->tel_cap >= count) return SCHED_OK;
    if (h->d_tel) { kv_free(h->d_tel); h->d_tel = nullptr; h->tel_cap = 0; }
    KV_TRY(dev_alloc(&h->d_tel, (size_t)count + 2));
    h->tel_cap = count;
    return SCHED_OK;
}

struct DeviceGuard {
    int prev;
    bool ok;
    explicit DeviceGuard(int dev) : prev(-1), ok(false) {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = (prev == dev) || cudaSetDevice(dev) == cudaSuccess;
    }
    ~DeviceGuard() { if (ok && prev >= 0) cudaSetDevice(prev); }
};

#define KV_ENTER(h)                                                  \
    if (!(h)) return SCHED_E_INVAL;                                  \
    DeviceGuard guard__((h)->device);                                \
    if (!guard__.ok) return kv_cuda_fail(cudaGetLastError(), "cudaSetDevice")

int check_launch(sched_ctx* h) {
    h->launches += 1;
    KV_CUDA(cudaGetLastError());
    return SCHED_OK;
}

int validate_instance(i64 total, const int32_t* s, const int32_t* o, i64 M) {
    for (i64 i = 0; i < total; ++i) {
        if (s[i] < 1 || o[i] < 1) return SCHED_E_INVAL;
        if ((i64)s[i] + (i64)o[i] > M) return SCHED_E_INVAL;
    }
    return SCHED_OK;
}

void free_ctx(sched_ctx* h) {
    if (!h) return;
    void* ptrs[] = {h->d_arena, h->d_rings, h->d_tel, h->d_stage, h->d_sort, h->d_k4, h->d_ls};
    for (void* p : ptrs) if (p) kv_free(p);
    kv_host_free(h->h_pinned, h->pinned_bytes);
    if (h->ev_k3_begin) cudaEventDestroy(h->ev_k3_begin);
    if (h->ev_k3_end) cudaEventDestroy(h->ev_k3_end);
    if (h->own_stream) cudaStreamDestroy(h->own_stream);
    delete h;
}

int k3_warps(const sched_ctx* h) {
    int w = 0;
#define GETW(SIM) w = SIM::kWarps
    KV_DISPATCH_SIM(h, GETW);
#undef GETW
    if (h->ring_cells > 0) {                  // one ring per warp has to fit in shared memory
        const int fit = (int)(((size_t)h->smem_optin - 2048) / ((size_t)h->ring_cells * sizeof(int)));
        if (fit < w) w = fit;
    }
    return w;
}

// The base run's kernel for a handle (sim_chunk.cuh, run_alone): a form each for backlogs of which more than half decode for up
// to 64 rounds and more than a quarter for 1,025 and more; and of each one that asks for four requests at a time where nothing
// waits (run_together).  That pays where the budget holds a tenth of the backlog, so that much of the list starts at once;
// elsewhere its code alone costs 0.03 to 0.07.  Sorted-F as a whole, ms, with it / without, by the share of the backlog that the
// budget holds, 10,000 requests:
//   decodes to 20      0.35 0.73 / 0.91   0.10 0.87 / 0.92   0.05 0.93 / 0.95   0.01 1.15 / 1.10
//   to 256             0.47 0.69 / 0.91   0.12 0.87 / 0.92   0.05 0.97 / 0.97   0.01 1.20 / 1.14
//   to 1,024           0.57 0.74 / 0.84   0.11 0.89 / 0.87   0.06 0.98 / 0.94   0.01 1.24 / 1.16
//   to 2,048           0.65 0.87 / 1.16   0.16 1.19 / 1.19   0.08 1.26 / 1.24   0.04 1.35 / 1.32
typedef void (*BaseRunKernel)(BaseRunParams);
template <int NM, bool kTogether>
BaseRunKernel base_run_form(const sched_ctx* h) {
    typedef ChunkSim<NM> S;
    if (h->brief_share > 0.5) return k3_base_run<S, S::kBrief, kTogether>;
    if (NM > 1 && h->lengthy_share > 0.25) return k3_base_run<S, (NM > 1 ? S::kLengthy : S::kPlain), kTogether>;
    return k3_base_run<S, S::kPlain, kTogether>;
}
template <int NM>
BaseRunKernel base_run_form(const sched_ctx* h) {
    const bool together = (double)h->M > 0.1 * (double)h->n * (h->mean_s + h->mean_o);
    return together ? base_run_form<NM, true>(h) : base_run_form<NM, false>(h);
}
BaseRunKernel base_run_kernel(const sched_ctx* h) {
    switch (h->nm) {
        case 1: return base_run_form<1>(h);
        case 2: return base_run_form<2>(h);
        case 4: return base_run_form<4>(h);
        case 8: return base_run_form<8>(h);
        default: return k3_base_run<HybSim, -1, false>;
    }
}

size_t k3_smem_bytes(const sched_ctx* h) { return (size_t)k3_warps(h) * h->ring_cells * sizeof(int); }

// A sort of rows of n entries merges more than once: it needs a second pair of buffers.
bool sort_needs_two(int n) { return n > K1_MERGE_RUNS * K1_TILE; }

// d_result, d_order and d_batch_off as create_common lays them out: {TEL, batches, status}, n, n + 1 ints
size_t order_at() { return 256; }
size_t offsets_at(int n) { return order_at() + (((size_t)n * sizeof(int) + 255) & ~(size_t)255); }
size_t result_bytes(int n) { return offsets_at(n) + ((size_t)n + 1) * sizeof(int); }

// Orders of up to 4,000,000 requests are handed in and out through the handle's pinned block; larger ones are
// copied from and to the caller's memory (pinning 128 MB for 10,000,000 requests takes sched_init 100 ms).
bool reads_through_pinned(int n) { return 256 + result_bytes(n) <= ((size_t)32 << 20); }

// The chunked simulator's bounds are a round (below 2^30, as are M and the sum of all decodes) plus tokens in use (M) plus
// at most 31 for every request that is resident at the same time (two tokens each): V fits 31 bits, and its bound has to.
bool chunk_sums_fit(i64 n, i64 M) {
    const i64 beside = n < M / 2 ? n : M / 2;
    return M + 32 * n + 32768 < (1ll << 31) && (1ll << 30) + 31 * beside + 65536 < (1ll << 31);
}

int create_common(sched_ctx** out, int B, int n, const int32_t* s, const int32_t* o, i64 M) {
    if (!out) return SCHED_E_INVAL;
    *out = nullptr;
    if (B < 1 || n < 1 || !s || !o || M < 1) return SCHED_E_INVAL;
    if (M >= (1ll << 30)) return SCHED_E_UNSUPPORTED;
    const i64 total = (i64)B * n;
    KV_TRY(validate_instance(total, s, o, M));
    int omax = 0, omin = INT32_MAX, least = INT32_MAX; i64 sum_max = 0, brief = 0; double volume = 0;
    for (int b = 0; b < B; ++b) {
        i64 sum = 0;
        for (int i = 0; i < n; ++i) {
            const int v = o[(i64)b * n + i], size = s[(i64)b * n + i] + v;
            sum += v;
            volume += (double)v * (size - 0.5 * v);
            brief += v < 64 ? size - v + 1 : 0;
            omax = v > omax ? v : omax;
            omin = v < omin ? v : omin;
            least = size < least ? size : least;
        }
        if (sum > sum_max) sum_max = sum;
    }
    // of some 4,096 requests spread over all: enough for a rule, and these sums over all of 1,000,000 are 2 ms
    double short_o = 0, brief_o = 0, lengthy_o = 0, some_s = 0, some_o = 0, looked_at = 0;
    for (i64 k = 0, step = 1 + total / 4096; k < total; k += step) {
        short_o += o[k] <= 32 ? 1.0 : 32.0 / o[k];
        brief_o += o[k] <= 64; lengthy_o += o[k] > 1024;
        some_s += s[k]; some_o += o[k]; looked_at += 1.0;
    }
    if (sum_max + omax >= (1ll << 30)) return SCHED_E_UNSUPPORTED;

    sched_ctx* h = new (std::nothrow) sched_ctx();
    if (!h) return SCHED_E_NOMEM;
    memset(h, 0, sizeof(*h));
    int rc = SCHED_OK;
    do {
        if (cudaGetDevice(&h->device) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), "cudaGetDevice"); break; }
        if (cudaDeviceGetAttribute(&h->sm_count, cudaDevAttrMultiProcessorCount, h->device) != cudaSuccess ||
            cudaDeviceGetAttribute(&h->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device) != cudaSuccess) {
            rc = kv_cuda_fail(cudaGetLastError(), "cudaDeviceGetAttribute"); break;
        }
        h->B = B; h->n = n; h->M = M; h->omax = omax; h->omin = omin; h->least = least; h->volume = volume; h->brief_tokens = (double)brief; h->sum_o_max = sum_max;
        h->mean_s = some_s / looked_at; h->mean_o = some_o / looked_at; h->short_share = short_o / looked_at;
        h->brief_share = brief_o / looked_at; h->lengthy_share = lengthy_o / looked_at;
        h->g_num = 0; h->g_den = 1;
        const int slots = sim_pick_slots(omax);
        h->nm = slots <= 32 ? 1 : slots <= 256 ? slots / 32 : 0;
        if (!chunk_sums_fit(n, M)) h->nm = 0;
        if (const char* kind = getenv("KVSCHED_SIM"))               // testing knob: force the hybrid simulator
            if (strcmp(kind, "hybrid") == 0) h->nm = 0;
        // ints per simulator state, and the part of it that lives in shared memory
        h->L = h->nm == 0 ? 32 * (HybSim::NREG + sim_pick_far_chunks(omax)) : sim_state_ints(h->nm, slots);
        h->ring_cells = h->nm == 0 ? HybSim::ring_cells(h->L) : 32 * slots;
        if (k3_warps(h) < 1) { rc = SCHED_E_UNSUPPORTED; break; }
        if (cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), "cudaStreamCreate"); break; }
        h->stream = h->own_stream;
        if (cudaEventCreate(&h->ev_k3_begin) != cudaSuccess || cudaEventCreate(&h->ev_k3_end) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), "cudaEventCreate"); break; }
        if (B == 1) {
            size_t per = (size_t)h->L * sizeof(int);
            // a candidate replays (stride - 1) / 2 positions on average to reach its first moved one:
            // 0.2 % of the list at 256 snapshots, for which the base run stores 256 states instead of n.
            // An admission of the hybrid simulator costs as much as storing its state, and late ones ten times
            // that, so a move near the end of the list counts: one of 20,000 requests with decodes up to 20,000
            // took 1.65 ms with 256 states and takes 0.20 (the base run 59.8 and 70.7)
            i64 stride = h->nm ? ((i64)n + kSnapshots - 1) / kSnapshots : kSnapStrideHyb;
            if (h->nm && stride < 16) stride = 16;      // the base run stops for every snapshot
            while ((((i64)n + stride - 1) / stride) * (i64)per > (i64)kSnapBudget) stride += 4;
            h->snap_stride = (int)stride;
            h->snap_count = (n + h->snap_stride - 1) / h->snap_stride;
        }
        // every array of a fixed size in one block; first pass: its size, second: the addresses
        size_t used = 0;
        for (int pass = 0; pass < 2 && rc == SCHED_OK; ++pass) {
            if (pass == 1 && (rc = dev_alloc(&h->d_arena, used < kPoolMinBlock ? kPoolMinBlock : used)) != SCHED_OK) break;
            used = 0;
            auto take = [&](auto** ptr, size_t count) {
                typedef typename std::remove_reference<decltype(**ptr)>::type T;
                if (pass == 1) *ptr = (T*)(h->d_arena + used);
                used += (count * sizeof(T) + 255) & ~(size_t)255;
            };
            // what a solver call hands back lies in a row: base TEL, batches, status, best move | order | batch offsets
            take(&h->d_result, 16);
            if (B == 1) { take(&h->d_order, n); take(&h->d_batch_off, n + 1); }
            take(&h->d_s, total); take(&h->d_o, total);
            take(&h->d_tbl_id, total + 2);
            take(&h->d_counter, 4);
            take(&h->d_partials, 2 * 4096); take(&h->d_ticket, 1);
            if (B == 1) {
                take(&h->d_tbl_base, n + 2);
                take(&h->d_base_starts, n);
                take(&h->d_keys_a, n); take(&h->d_keys_b, n);
                take(&h->d_vals_a, n); take(&h->d_vals_b, n);
                if (sort_needs_two(n)) { take(&h->d_keys_more, n); take(&h->d_vals_more, n); }
                take(&h->d_prefP, n + 1); take(&h->d_prefO, n + 1);
                take(&h->d_snap_ring, (size_t)h->snap_count * h->L);
                take(&h->d_snap_hdr, h->snap_count);
            }
        }
        if (rc != SCHED_OK) break;
        h->d_base_tel = (i64*)h->d_result;
        h->d_num_batches = h->d_result + 2;
        h->d_status = h->d_result + 3;
        h->d_best = (i64*)(h->d_result + 4);
        h->d_accepted = h->d_result + 8;
        h->pinned_bytes = 256 + (B == 1 && reads_through_pinned(n) ? result_bytes(n) : 0);
        if (kv_host_malloc(&h->h_pinned, &h->pinned_bytes) != cudaSuccess) { h->h_pinned = nullptr; rc = kv_cuda_fail(cudaGetLastError(), "cudaHostAlloc"); break; }
        cudaStream_t st = h->stream;
#define C(call) if ((call) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), #call); break; }
        C(cudaMemcpyAsync(h->d_s, s, total * sizeof(int), cudaMemcpyHostToDevice, st));
        C(cudaMemcpyAsync(h->d_o, o, total * sizeof(int), cudaMemcpyHostToDevice, st));
        C(cudaMemsetAsync(h->d_tbl_id, 0, (total + 2) * sizeof(int2), st));
        C(cudaMemsetAsync(h->d_status, 0, sizeof(int), st));
        C(cudaMemsetAsync(h->d_ticket, 0, sizeof(unsigned), st));
        C(cudaMemsetAsync(h->d_counter, 0, 4 * sizeof(unsigned), st));
        k3_make_table<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(h->d_s, h->d_o, (int)total, h->d_tbl_id);
        if ((rc = check_launch(h)) != SCHED_OK) break;
        if (B == 1) {
            C(cudaMemsetAsync(h->d_tbl_base, 0, (n + 2) * sizeof(int2), st));
            k3_iota<<<(n + 255) / 256, 256, 0, st>>>(h->d_order, n);
            if ((rc = check_launch(h)) != SCHED_OK) break;
        }
        // opt in to large dynamic shared memory once
        {
            const int dyn = h->smem_optin - 2048;
            cudaError_t e1 = cudaSuccess, e2 = cudaSuccess, e3 = cudaSuccess, e4 = cudaSuccess;
#define SETATTR(N)                                                                                         \
            e1 = cudaFuncSetAttribute(k3_eval_moves<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);  \
            if (e1 == cudaSuccess) e1 = cudaFuncSetAttribute(k3_eval_moves<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn);  \
            e2 = cudaFuncSetAttribute(k3_eval_orders<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn); \
            if (e2 == cudaSuccess) e2 = cudaFuncSetAttribute(k3_eval_orders<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn); \
            e3 = cudaFuncSetAttribute(k3_eval_policy<N, int>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn - 2048); \
            if (e3 == cudaSuccess) e3 = cudaFuncSetAttribute(k3_eval_policy<N, i64>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn - 2048); \
            e4 = cudaFuncSetAttribute(base_run_kernel(h), cudaFuncAttributeMaxDynamicSharedMemorySize, dyn)
            KV_DISPATCH_SIM(h, SETATTR);
#undef SETATTR
            if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess || e4 != cudaSuccess) {
                rc = kv_cuda_fail(cudaGetLastError(), "cudaFuncSetAttribute(MaxDynamicSharedMemorySize)"); break;
            }
        }
        C(cudaStreamSynchronize(st));       // s, o may be pageable host memory owned by the caller
#undef C
    } while (0);
    if (rc != SCHED_OK) { free_ctx(h); return rc; }
    *out = h;
    return SCHED_OK;
}

// `rows` lists of n entries in ascending (key, value) order -> out.  More than one tile: through
// tmp_keys / tmp_vals (rows * n entries each); more than one merge: and through more_keys / more_vals.
template <class KEY>
int sort_rows(sched_ctx* h, const KEY& src, int n, i64 rows, u64* tmp_keys, int* tmp_vals, u64* more_keys, int* more_vals, int* out) {
    const int tiles = (n + K1_TILE - 1) / K1_TILE;
    const i64 total = rows * n, ctas = rows * tiles;
    if (total >= (1ll << 31) || ctas >= (1ll << 31)) return SCHED_E_UNSUPPORTED;
    int threads = 32;
    while (threads < n && threads < K1_TILE) threads <<= 1;
    k1_tile_sort<<<(unsigned)ctas, threads, 0, h->stream>>>(src, n, tiles, tiles > 1 ? tmp_keys : nullptr, tiles > 1 ? tmp_vals : out);
    KV_TRY(check_launch(h));
    int merges = 0;
    for (i64 most = 1; most < tiles; most *= K1_MERGE_RUNS) ++merges;
    i64 run = K1_TILE;
    for (; merges > 0; --merges) {
        // as few runs per merge as the merges that are left can do with
        const int runs = (int)((n + run - 1) / run);
        int group = 2;
        for (;; ++group) {
            i64 reach = 1;
            for (int k = 0; k < merges && reach < runs; ++k) reach *= group;
            if (reach >= runs) break;
        }
        k1_tile_merge<<<(unsigned)((total + K1_MERGE_THREADS - 1) / K1_MERGE_THREADS), K1_MERGE_THREADS, 0, h->stream>>>(
            tmp_keys, tmp_vals, n, total, (int)run, group, bits_of((u64)run), merges > 1 ? more_keys : nullptr, merges > 1 ? more_vals : out);
        KV_TRY(check_launch(h));
        run *= group;
        u64* const k = tmp_keys; tmp_keys = more_keys; more_keys = k;
        int* const v = tmp_vals; tmp_vals = more_vals; more_vals = v;
    }
    return SCHED_OK;
}

// Base order -> position-ordered table, snapshots, base TEL.
BaseRunParams base_run_params(sched_ctx* h) {
    BaseRunParams p;
    memset(&p, 0, sizeof(p));
    p.tbl_id = h->d_tbl_id; p.tbl_base = h->d_tbl_base; p.order = h->d_order;
    p.n = h->n; p.L = h->L; p.M = (int)h->M; p.stride = h->snap_stride; p.snap_count = h->snap_count;
    p.snap_ring = h->d_snap_ring; p.snap_hdr = h->d_snap_hdr; p.starts_pos = h->d_base_starts;
    p.base_tel = h->d_base_tel; p.status = h->d_status;
    return p;
}

int run_base(sched_ctx* h, const BaseRunParams& p) {
    base_run_kernel(h)<<<1, K3B_THREADS, (size_t)h->ring_cells * sizeof(int), h->stream>>>(p);
    return check_launch(h);
}

int ensure_base(sched_ctx* h) {
    if (h->base_ready) return SCHED_OK;
    KV_TRY(run_base(h, base_run_params(h)));
    h->base_ready = true;
    return SCHED_OK;
}

// The best of tel[0 .. count) (launch slots, mapped back through index_map), or of d_best with count = 0,
// becomes the base order's next move if it improves; the base run follows.  Leaves d_result complete.
int accept_best(sched_ctx* h, const i64* tel, const int* index_map, i64 count, int sampled, u64 seed, int iteration) {
    BaseRunParams p = base_run_params(h);
    p.accept = 1;
    p.tel = tel; p.index_map = index_map; p.count = count;
    p.best = h->d_best; p.accepted = h->d_accepted; p.scratch = h->d_vals_b;
    p.sampled = sampled; p.seed = seed; p.iteration = iteration;
    return run_base(h, p);
}

// one warp per candidate: CTAs needed for `count` candidates
unsigned k3_grid(const sched_ctx* h, i64 count) {
    const int w = k3_warps(h);
    const i64 ctas = (count + w - 1) / w;
    return (unsigned)(ctas < 1 ? 1 : ctas);
}

// Candidates that run side by side in one wave need no launch order: 8 warps per SM cost four launches
// less (12 of 33 us of a 120-move sweep) and no longer tail.
i64 ordered_from(const sched_ctx* h) { return 8ll * h->sm_count; }
// slot -> candidate of the last launch_moves() of `count` candidates, nullptr: the same
const int* last_launch_order(const sched_ctx* h, i64 count) {
    return count > ordered_from(h) ? (const int*)h->d_k4 + h->n + 1 + count : nullptr;
}

// K4: launch order of `count` candidates, bucketed by first moved position (longest suffix first)
int order_candidates(sched_ctx* h, const MoveSource& src, i64 count) {
    const size_t need = ((size_t)h->n + 1 + 2 * (size_t)count) * sizeof(int) + 256;
    if (h->k4_cap < need) {
        if (h->d_k4) { kv_free(h->d_k4); h->d_k4 = nullptr; h->k4_cap = 0; }
        KV_CUDA(kv_malloc((void**)&h->d_k4, need));
        h->k4_cap = need;
    }
    int* bins = (int*)h->d_k4;
    int* first_pos = bins + h->n + 1;
    int* launch_order = first_pos + count;
    KV_CUDA(cudaMemsetAsync(bins, 0, ((size_t)h->n + 1) * sizeof(int), h->stream));
    const unsigned blocks = (unsigned)((count + 255) / 256);
    k4_first_pos_histogram<<<blocks, 256, 0, h->stream>>>(src, h->n, count, bins, first_pos);
    KV_TRY(check_launch(h));
    k4_scan_bins<<<1, 1024, 0, h->stream>>>(bins, h->n);
    KV_TRY(check_launch(h));
    k4_scatter_by_first_pos<<<blocks, 256, 0, h->stream>>>(first_pos, h->n, count, bins, launch_order);
    KV_TRY(check_launch(h));
    return SCHED_OK;
}

// Moves with a warp each on the simulator for short windows (sim_chunk.cuh)?  Measured over 216 sweeps of 16,000 moves, the
// share of short decodes (mean of min(1, 32 / o)) against the time with it over that without: 0.985 and more 0.79 to 0.92,
// 0.95 to 0.985 0.94 (0.92 to 0.98), 0.94 0.98 (0.95 to 1.01), 0.90 1.00 (0.98 to 1.03), below 1.03 (1.01 to 1.05).
bool short_windows(const sched_ctx* h, bool want_starts) { return !want_starts && h->nm == 1 && h->short_share >= 0.93; }

// One thread per candidate instead of one warp (k3_lanes.cuh)?  Its work goes with the rounds that pass, the
// other kernel's with the admissions: rounds per request is the backlog's volume (sum of s o + o^2 / 2) over
// n M, within a few per cent of the base run's.  Up to 94,720 candidates (56,832 for decodes beyond 1,025) run
// side by side, so its time hardly moves below that and the other's is proportional to the count.  Measured,
// warp against thread, ms:
//   rounds per request  2.9 (n = 10,000)   7.6 (10,000)   12.4 (1,000)   18.9 (4,000)   24.8 (1,000)
//   16,000 moves          7.1 /  8.4        8.6 / 14.4     1.0 / 1.7      4.7 / 11.7     1.3 / 3.2
//   24,000               10.5 /  8.9       12.7 / 15.9     1.5 / 1.8      7.0 / 12.7     2.0 / 3.5
//   32,000               13.9 /  9.4       16.8 / 16.2     2.0 / 1.9      9.3 / 13.1     2.6 / 3.6
//   48,000               20.8 / 10.4       25.2 / 18.4     3.0 / 2.1     13.8 / 14.8     3.9 / 4.1
//   96,000               41.4 / 15.1       50.1 / 25.9     5.9 / 3.0     27.5 / 21.0     7.7 / 5.7
//   decodes to 2,048    4.5 (n = 2,000)   10.8 (2,000)    14.8 (2,000)
//   32,000                3.8 /  4.1        5.1 / 7.6      5.9 /  9.2
//   48,000                5.7 /  4.3        7.6 / 8.0      8.7 / 10.4
//   96,000               11.4 /  5.7       15.1 / 12.2    17.4 / 16.4
// Two kinds of backlog cost a thread more per admission (log-normal decodes, prefills uniform up to 2,000):
//   short decodes: a window that ends in one of the two chunks kept as cells takes its share back from them one by one,
//   which the share of decodes up to a chunk (each counted as 32 / o beyond) tells.  Mean 20 (share 0.94): 40,000 moves of
//   10,000, 0.5 / 2 / 6 rounds per request 16.3 / 20.0, 19.8 / 30.7, 27.6 / 49.7; mean 82 (0.56): 16.4 / 9.3, 18.4 / 14.7,
//   21.2 / 24.2;
//   long decodes on short prefills: memory is used by tokens still to come, what a request waits for lies chunks
//   ahead, and every wait walks the events up to there.  Prefills up to 20, decodes of mean 344, 10,000 requests, 40,000
//   moves, 0.5 / 1 / 2 / 6 rounds per request 16.0 / 9.4, 16.4 / 17.8, 17.3 / 43.5, 20.8 / 179; prefills up to 2,000: 16.0 / 6.9,
//   16.4 / 8.6, 17.0 / 11.6, 19.5 / 28.2; decodes of mean 692 (to 2,048), prefills up to 20: 20.8 / 8.7, 21.2 / 14.7, 22.2 / 19.0,
//   26.2 / 57.5.  Use of memory falls by s / rounds per round and varies by (s + o) sqrt(rounds ahead / rounds), hence
//   the form in (1 + o / s) sqrt(rounds); its square and the caps are fitted.  Only where time goes on for
//   longer than a decode: otherwise nearly everything runs side by side.
// A line fitted again to 1,164 sweeps (1,000 mixed requests at 24 rounds per request: the thread from 50,000 moves instead of
// 85,000) took 7.60 instead of 4.06 ms for a backlog drawn at random, so the line before it stands.  Longer decodes than its ring of events, schedules with more rounds per request than were
// measured, and backlogs whose candidate could pass 32 bits of waiting time in its sum of starts or of tokens in a chunk
// (lane_sums_fit) keep the warp.
constexpr double LANE_ROUNDS = 25.0, LANE_MIN = 18000.0, LANE_MIN_PER_ROUND = 1500.0, LANE_LONG = 1.55;

// candidates from which on a thread each is the faster one
double lanes_from(const sched_ctx* h) {
    const double rounds = h->volume / ((double)h->n * (double)h->M), n = (double)h->n;
    double need = LANE_MIN + LANE_MIN_PER_ROUND * rounds, ahead = (1.0 + h->mean_o / h->mean_s) * (1.0 + h->mean_o / h->mean_s);
    if (rounds > LANE_ROUNDS) return INFINITY;
    if (h->nm == 1) {
        if (h->short_share > 0.3) need += 11000.0 * rounds * (h->short_share - 0.3);
        if (ahead > 1.3) need += 8700.0 * rounds * (fmin(ahead, 3.0) - 1.3);
        if (h->short_share > 0.75) need += 150000.0 * (h->short_share - 0.75);
        if (short_windows(h, false)) need *= 1.3;              // against the warp's simulator for those
        ahead = fmin(ahead, 8.0);
    } else {
        need *= LANE_LONG;
        if (h->short_share > 0.4) need *= 1.0 + (h->short_share - 0.4) * rounds / 3.0;
        // candidates further apart in a long list also leave one another's rounds: 40,000 moves of 10,000 and of 2,000
        // requests with a share of 0.72, 6 rounds per request: 28.1 / 60 and 5.6 / 11.4
        if (h->short_share > 0.4 && n > 2000.0) need *= 1.0 + (n - 2000.0) * rounds / 48000.0;
        ahead = fmin(0.6 * ahead, 3.6);
    }
    const double far = ahead * sqrt(rounds);
    if (n * rounds >= (double)h->omax && far > 5.0) need = far > 8.0 ? INFINITY : need * (1.0 + 0.55 * (far - 5.0));
    return need;
}

// A thread keeps the bound of the chunk that t lies in, and its cells less the ramps that have come in since, in 32 bits.
// Both take s + 1 and up to a chunk's rounds from every request that starts in the chunk: those that outlast it
// hold M tokens at most, those that end in it M per round of the chunk.  Beyond 2^30 (budgets from 2^24 on, and then
// only with decodes of a few rounds) the warp has to do it: its cells are exact.
bool lane_sums_fit(const sched_ctx* h) {
    const double rounds = h->nm == 1 ? 32.0 : 64.0, M = (double)h->M;
    const double ends = fmin(h->brief_tokens, M * rounds / h->omin), starts = fmin((double)h->n, 0.5 * (ends + M));
    return 2.0 * M + ends + rounds * (starts + 2.0) < 1073741824.0;
}

bool lanes_fit(const sched_ctx* h, i64 count, bool want_starts) {
    if (want_starts || (h->nm != 1 && h->nm != 2) || count <= ordered_from(h)) return false;
    return (double)count >= lanes_from(h) && (i64)h->n * (h->omax + 64) <= INT32_MAX && lane_sums_fit(h);
}

// The handle's block of rings in device memory, of at least `bytes`; false if there is no memory for it.
bool grow_rings(sched_ctx* h, size_t bytes) {
    if (h->rings_cap >= bytes) return true;
    if (h->d_rings) { kv_free(h->d_rings); h->d_rings = nullptr; h->rings_cap = 0; }
    if (kv_malloc(&h->d_rings, bytes) != cudaSuccess) { cudaGetLastError(); h->d_rings = nullptr; return false; }
    h->rings_cap = bytes;
    return true;
}

// SCHED_OK with *done = false: no memory for the rings of events, nothing was launched.
template <int CH, typename WORD>
int run_lanes(sched_ctx* h, LaneParams& q, bool* done) {
    typedef LaneSim<CH, WORD> S;
    const i64 need = ((i64)q.groups + S::kWarps - 1) / S::kWarps, most = (i64)S::kCtas * h->sm_count;
    const int grid = (int)(need < most ? need : most);
    const size_t bytes = (size_t)grid * S::kWarps * S::kRingWords * sizeof(WORD);
    *done = false;
    if (!grow_rings(h, bytes)) return SCHED_OK;
    q.rings = h->d_rings;
    q.counter = h->d_counter + 1;
    KV_CUDA(cudaMemsetAsync(q.counter, 0, sizeof(unsigned), h->stream));
    KV_CUDA(cudaFuncSetAttribute(k3_lane_moves<CH, WORD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::kSmem));
    KV_CUDA(cudaEventRecord(h->ev_k3_begin, h->stream));
    k3_lane_moves<CH, WORD><<<grid, 32 * S::kWarps, S::kSmem, h->stream>>>(q);
    *done = true;
    return SCHED_OK;
}

int launch_lanes(sched_ctx* h, const MoveEvalParams& p, bool* done) {
    LaneParams q;
    memset(&q, 0, sizeof(q));
    q.m = p; q.omax = h->omax; q.least = h->least;
    q.groups = (int)((p.count + 31) / 32);
    // the requests that end in one round hold M tokens at most: sum of (s+o - least) and number in 32 bits?
    q.shift = bits_of((u64)(h->M - h->least));
    const bool narrow = q.shift + bits_of((u64)(h->M / h->least)) <= 32;
    if (!narrow) q.shift = 32;
    if (h->nm == 1) return narrow ? run_lanes<32, unsigned>(h, q, done) : run_lanes<32, u64>(h, q, done);
    return narrow ? run_lanes<64, unsigned>(h, q, done) : run_lanes<64, u64>(h, q, done);
}

// Moves with a warp each whose rings are in device memory (sim_chunk.cuh)?  32 instead of 13 warps per SM
// against a wait for memory per 32 rounds.  Measured, shared against device memory, decodes to 4,096, ms:
//   rounds per request             1               2               3               4.2             16
//   100,000 requests, 7,000 moves  42.7 / 38.5     44.9 / 49.1
//   20,000, 35,000                 40.0 / 34.9     42.1 / 39.9     44.2 / 49.4     46.7 / 63.4
//   20,000, 4,000                  4.79 / 4.80     5.03 / 5.58                     5.67 / 8.11
//   20,000, 2,400                  3.20 / 4.17                                     3.86 / 5.95
//   2,000, 100,000                 11.4 / 10.1     12.0 / 11.6                     13.4 / 19.0     20.1 / 49.6
// The two cross near 2 rounds per request and at 27 warps per SM, and differ by a tenth there.
bool device_rings_fit(const sched_ctx* h, i64 count, bool want_starts) {
    return !want_starts && h->nm == 4 && count >= 27ll * h->sm_count && h->volume <= 2.0 * (double)h->n * (double)h->M;
}

// 512 MB of rings per launch.  SCHED_OK with *done = false: no memory for them, nothing was launched.
int moves_from_device_rings(sched_ctx* h, MoveEvalParams& p, bool* done) {
    typedef ChunkSim<4, true> S;
    const size_t bytes = (size_t)h->ring_cells * sizeof(int);
    i64 most = (i64)(((size_t)512 << 20) / bytes);
    if (most > p.count) most = p.count;
    *done = false;
    if (!grow_rings(h, bytes * most)) return SCHED_OK;
    p.rings = (int*)h->d_rings;
    KV_CUDA(cudaEventRecord(h->ev_k3_begin, h->stream));
    for (i64 at = 0; at < p.count; at += most) {
        if (at > 0) KV_TRY(check_launch(h));               // the caller counts the last launch
        p.first_slot = at;
        p.end_slot = at + most < p.count ? at + most : p.count;
        const i64 ctas = (p.end_slot - at + S::kWarps - 1) / S::kWarps;
        k3_eval_moves<S, false><<<(unsigned)ctas, S::kWarps * 32, 0, h->stream>>>(p);
    }
    *done = true;
    return SCHED_OK;
}

// by_slot: TELs are left in launch-slot order (h->d_k4's launch_order maps a slot to its candidate
// until the next call); the sweeps that only need the arg-min use it, see launch_argmin.
int launch_moves(sched_ctx* h, int mode, const i64* codes, i64 first, u64 seed, int iteration,
                 i64 count, i64* tel_out, int* starts_out, bool by_slot = false) {
    if (count <= 0) return SCHED_OK;
    if (count >= (1ll << 31)) return SCHED_E_UNSUPPORTED;
    KV_TRY(ensure_base(h));
    MoveEvalParams p;
    memset(&p, 0, sizeof(p));
    const size_t smem = k3_smem_bytes(h);
    p.n = h->n; p.L = h->L; p.M = (int)h->M; p.stride = h->snap_stride;
    p.tbl_base = h->d_tbl_base;
    p.snap_ring = h->d_snap_ring; p.snap_hdr = h->d_snap_hdr; p.snap_count = h->snap_count;
    p.src.mode = mode; p.src.codes = codes; p.src.first = first; p.src.seed = seed; p.src.iteration = iteration;
    p.count = count; p.tel_out = tel_out; p.tel_by_slot = by_slot ? 1 : 0; p.starts_out = starts_out;
    p.base_order = h->d_order; p.base_starts_pos = h->d_base_starts;
    p.status = h->d_status;
    if (count > ordered_from(h)) {
        KV_TRY(order_candidates(h, p.src, count));
        p.launch_order = last_launch_order(h, count);
    }
    bool done = false;                               // ev_k3_begin is recorded behind the search for memory
    if (lanes_fit(h, count, starts_out != nullptr)) KV_TRY(launch_lanes(h, p, &done));
    else if (device_rings_fit(h, count, starts_out != nullptr)) KV_TRY(moves_from_device_rings(h, p, &done));
    if (!done) {
        p.first_slot = 0; p.end_slot = count;
        KV_CUDA(cudaEventRecord(h->ev_k3_begin, h->stream));
        if (short_windows(h, starts_out != nullptr)) {
            k3_eval_moves<ChunkSim<1, false, true>, false><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p);
            done = true;
        }
    }
    if (!done) {
#define RUN(N)                                                                                    \
    if (starts_out) k3_eval_moves<N, true><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p);  \
    else k3_eval_moves<N, false><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p)
    KV_DISPATCH_SIM(h, RUN);
#undef RUN
    }
    KV_TRY(check_launch(h));
    KV_CUDA(cudaEventRecord(h->ev_k3_end, h->stream));
    h->ev_valid = true;
    h->evaluations += count;
    return SCHED_OK;
}

int launch_argmin(sched_ctx* h, const i64* tel, i64 count, i64 index_base, const i64* prior, i64* best_out,
                  const int* index_map = nullptr) {
    i64 blocks = (count / 2 + K5_THREADS - 1) / K5_THREADS;
    if (blocks < 1) blocks = 1;
    if (blocks > 4 * h->sm_count) blocks = 4 * h->sm_count;
    if (blocks > 4096) blocks = 4096;
    k5_argmin<<<(unsigned)blocks, K5_THREADS, 0, h->stream>>>(tel, count, index_base, index_map, prior, h->d_partials, h->d_ticket, best_out);
    return check_launch(h);
}

i64 neighbourhood_size(int n, int nb, i64 samples) {
    const i64 nsw = (i64)n * (n - 1) / 2;
    return nb == SCHED_NBHD_SWAP ? nsw : nb == SCHED_NBHD_SWAP_INSERT ? nsw + (i64)n * (n - 1) : samples;
}

// Checked build only: the word in which KV_IDX records the first index that left its array.  Reads
// it after the device is idle, clears it, and turns a recorded index into SCHED_E_INTERNAL with the
// site and value in sched_last_cuda_error().
int read_checked_word() {
#ifdef KVSCHED_CHECKED
    unsigned long long w = 0ull;
    KV_CUDA(cudaDeviceSynchronize());
    KV_CUDA(cudaMemcpyFromSymbol(&w, kv_checked_word, sizeof(w)));
    if (w != 0ull) {
        const unsigned long long zero = 0ull;
        cudaMemcpyToSymbol(kv_checked_word, &zero, sizeof(zero));
        long long idx = (long long)(w & 0xffffffffffull);
        if (idx & (1ll << 39)) idx -= (1ll << 40);
        snprintf(g_last_cuda_error, sizeof(g_last_cuda_error), "checked build: index %lld outside its array at site %d",
                 idx, (int)(w >> 40));
        return SCHED_E_INTERNAL;
    }
#endif
    return SCHED_OK;
}

// what the status word of an idle stream says
int after_status(sched_ctx* h, int status) {
    if (status != KV_DEV_OK) {
        h->base_ready = false;                       // the base run may be what gave up
        cudaMemsetAsync(h->d_status, 0, sizeof(int), h->stream);
        return SCHED_E_INTERNAL;
    }
    return read_checked_word();
}

int read_status(sched_ctx* h) {
    int* hp = (int*)h->h_pinned;
    KV_CUDA(cudaMemcpyAsync(hp, h->d_status, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    KV_CUDA(cudaStreamSynchronize(h->stream));
    return after_status(h, *hp);
}

#ifdef KVSCHED_CHECKED
__global__ void kv_check_index_probe(long long idx, long long limit, int* sink) {
    *sink = (int)KV_IDX(idx, limit, 9999);
}
#endif

bool is_permutation(const int32_t* a, int n, std::vector<unsigned char>& seen) {
    seen.assign(n, 0);
    for (int q = 0; q < n; ++q) {
        int v = a[q];
        if (v < 0 || v >= n || seen[v]) return false;
        seen[v] = 1;
    }
    return true;
}

}  // namespace

extern "C" {

int sched_init(sched_handle* out, int32_t n, const int32_t* s, const int32_t* o, int64_t M) {
    return create_common(out, 1, n, s, o, M);
}

int sched_init_batch(sched_handle* out, int32_t B, int32_t n_each, const int32_t* s, const int32_t* o, int64_t M) {
    if (n_each > 1024) return SCHED_E_UNSUPPORTED;
    int rc = create_common(out, B, n_each, s, o, M);
    if (rc == SCHED_OK) (*out)->batch_handle = true;
    return rc;
}

int sched_set_stream(sched_handle h, void* cuda_stream) {
    KV_ENTER(h);
    KV_CUDA(cudaStreamSynchronize(h->stream));
    h->stream = cuda_stream ? (cudaStream_t)cuda_stream : h->own_stream;
    return SCHED_OK;
}

int sched_sync(sched_handle h) {
    KV_ENTER(h);
    return read_status(h);
}

int sched_set_prefill_weight(sched_handle h, int32_t alpha_num, int32_t alpha_den) {
    if (!h) return SCHED_E_INVAL;
    if (alpha_num < 0 || alpha_den < 1 || alpha_num > (1 << 20) || alpha_den > (1 << 20)) return SCHED_E_INVAL;
    h->g_num = alpha_num; h->g_den = alpha_den;
    return SCHED_OK;
}

int sched_set_base_order(sched_handle h, const int32_t* order) {
    KV_ENTER(h);
    if (h->batch_handle || !order) return SCHED_E_INVAL;
    std::vector<unsigned char> seen;
    if (!is_permutation(order, h->n, seen)) return SCHED_E_NOT_PERMUTATION;
    KV_CUDA(cudaMemcpyAsync(h->d_order, order, (size_t)h->n * sizeof(int), cudaMemcpyHostToDevice, h->stream));
    KV_CUDA(cudaStreamSynchronize(h->stream));
    h->base_ready = false;
    return SCHED_OK;
}

int sched_get_base_order(sched_handle h, int32_t* order_out) {
    KV_ENTER(h);
    if (h->batch_handle || !order_out) return SCHED_E_INVAL;
    KV_CUDA(cudaMemcpyAsync(order_out, h->d_order, (size_t)h->n * sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    KV_CUDA(cudaStreamSynchronize(h->stream));
    return SCHED_OK;
}

// bad: nullable device word; orders and start times are evaluated only if it is 0 when their kernel starts
static int eval_batch_dev(sched_handle h, int kind, i64 count, const void* candidates, i64* tel_out, uint8_t* feasible_out,
                          int32_t* starts_out, const int* bad) {
    if (count < 0 || !tel_out || (count > 0 && !candidates)) return SCHED_E_INVAL;
    if (count == 0) return SCHED_OK;
    if (count >= (1ll << 31)) return SCHED_E_UNSUPPORTED;
    const int n = h->n;
    if (kind == SCHED_CAND_POLICY) {
        if (n >= 65536) return SCHED_E_UNSUPPORTED;                    // ids are 16-bit inside the kernel
        const bool narrow = (i64)n * h->M < (1ll << 31);               // prefix sums of s+o fit 32 bits
        const size_t shared_so = ((size_t)n * 8 + 15) & ~(size_t)15;
        const size_t per_warp = k3_policy_warp_bytes(n, h->ring_cells, narrow ? 4 : 8);
        const size_t room = (size_t)h->smem_optin - 4096;
        if (shared_so + per_warp > room) return SCHED_E_UNSUPPORTED;
        int W = (int)((room - shared_so) / per_warp);                  // pairs of one instance per CTA
        if (W > K3P_MAX_WARPS) W = K3P_MAX_WARPS;
        if ((i64)W > count) W = (int)count;
        const int groups = (int)((count + W - 1) / W);
        const size_t smem = shared_so + (size_t)W * per_warp;
        const i64 ctas = (i64)h->B * groups;
        if (ctas >= (1ll << 31)) return SCHED_E_UNSUPPORTED;
#define RUN(N)                                                                                                       \
        if (narrow) k3_eval_policy<N, int><<<(unsigned)ctas, 32 * W, smem, h->stream>>>(h->d_s, h->d_o, n, h->L, (int)h->M, h->omax, \
                                                                  (const int*)candidates, (int)count, groups, \
                                                                  (i64*)tel_out, starts_out, h->d_status);   \
        else k3_eval_policy<N, i64><<<(unsigned)ctas, 32 * W, smem, h->stream>>>(h->d_s, h->d_o, n, h->L, (int)h->M, h->omax, \
                                                                  (const int*)candidates, (int)count, groups, \
                                                                  (i64*)tel_out, starts_out, h->d_status)
        KV_CUDA(cudaEventRecord(h->ev_k3_begin, h->stream));
        KV_DISPATCH_SIM(h, RUN);
#undef RUN
        KV_TRY(check_launch(h));
        KV_CUDA(cudaEventRecord(h->ev_k3_end, h->stream));
        h->ev_valid = true;
        h->evaluations += (i64)h->B * count;
        if (feasible_out) KV_CUDA(cudaMemsetAsync(feasible_out, 1, (size_t)((i64)h->B * count), h->stream));
        return SCHED_OK;
    }
    if (h->batch_handle) return SCHED_E_INVAL;
    if (kind == SCHED_CAND_MOVE) {
        KV_TRY(launch_moves(h, 0, (const i64*)candidates, 0, 0, 0, count, (i64*)tel_out, starts_out));
        if (feasible_out) KV_CUDA(cudaMemsetAsync(feasible_out, 1, (size_t)count, h->stream));
        return SCHED_OK;
    }
    if (kind == SCHED_CAND_ORDER) {
        OrderEvalParams p;
        memset(&p, 0, sizeof(p));
        const size_t smem = k3_smem_bytes(h);
        p.n = n; p.L = h->L; p.M = (int)h->M; p.tbl_id = h->d_tbl_id;
        p.orders = (const int*)candidates; p.count = count; p.tel_out = (i64*)tel_out; p.starts_out = starts_out;
        p.bad = bad; p.status = h->d_status;
        KV_CUDA(cudaEventRecord(h->ev_k3_begin, h->stream));
#define RUN(N)                                                                                     \
        if (starts_out) k3_eval_orders<N, true><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p);  \
        else k3_eval_orders<N, false><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p)
        KV_DISPATCH_SIM(h, RUN);
#undef RUN
        KV_TRY(check_launch(h));
        KV_CUDA(cudaEventRecord(h->ev_k3_end, h->stream));
        h->ev_valid = true;
        h->evaluations += count;
        if (feasible_out) KV_CUDA(cudaMemsetAsync(feasible_out, 1, (size_t)count, h->stream));
        return SCHED_OK;
    }
    if (kind == SCHED_CAND_START_TIMES) {
        if (starts_out) return SCHED_E_INVAL;
        const i64 total = count * n;
        if (total >= (1ll << 31)) return SCHED_E_UNSUPPORTED;
        // ids of every candidate by ascending (start, id)
        const bool tiled = n > K1_TILE, two = sort_needs_two(n);
        const size_t pair = sizeof(u64) + sizeof(int);
        const size_t need = (size_t)total * (sizeof(int) + (tiled ? pair : 0) + (two ? pair : 0)) + 64;
        if (h->sort_cap < need) {
            if (h->d_sort) { kv_free(h->d_sort); h->d_sort = nullptr; h->sort_cap = 0; }
            KV_CUDA(kv_malloc((void**)&h->d_sort, need));
            h->sort_cap = need;
        }
        u64* tmp_keys = tiled ? (u64*)h->d_sort : nullptr;
        u64* more_keys = two ? tmp_keys + total : nullptr;
        int* tmp_vals = tiled ? (int*)(tmp_keys + (two ? 2 : 1) * total) : nullptr;
        int* more_vals = two ? tmp_vals + total : nullptr;
        int* ids = two ? more_vals + total : tiled ? tmp_vals + total : (int*)h->d_sort;
        KV_TRY(sort_rows(h, K1StartKey{(const int*)candidates}, n, count, tmp_keys, tmp_vals, more_keys, more_vals, ids));
        StartsEvalParams p;
        memset(&p, 0, sizeof(p));
        p.n = n; p.M = (int)h->M; p.tbl_id = h->d_tbl_id;
        p.starts = (const int*)candidates; p.sorted_ids = ids; p.count = count;
        p.tel_out = (i64*)tel_out; p.feasible_out = feasible_out; p.bad = bad;
        if (h->nm > 0) {
            p.L = h->L;
            const size_t smem = k3_smem_bytes(h);
            switch (h->nm) {
#define RUN(N) k3_check_starts<ChunkSim<N>><<<k3_grid(h, count), k3_warps(h) * 32, smem, h->stream>>>(p)
                case 1: RUN(1); break;
                case 2: RUN(2); break;
                case 4: RUN(4); break;
                default: RUN(8); break;
#undef RUN
            }
        } else {
            p.L = (h->omax + 8 + 31) & ~31; p.counter = h->d_counter;
            KV_CUDA(cudaMemsetAsync(h->d_counter, 0, sizeof(unsigned), h->stream));
            int sw = (int)(((size_t)h->smem_optin - 2048) / ((size_t)p.L * sizeof(int)));
            if (sw > K3S_WARPS) sw = K3S_WARPS;
            if (sw < 1) return SCHED_E_UNSUPPORTED;
            const i64 sctas = (count + sw - 1) / sw;
            KV_CUDA(cudaFuncSetAttribute(k3_check_starts_cells, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 2048));
            k3_check_starts_cells<<<(unsigned)(sctas < h->sm_count ? sctas : h->sm_count), sw * 32,
                                    (size_t)sw * p.L * sizeof(int), h->stream>>>(p);
        }
        KV_TRY(check_launch(h));
        h->evaluations += count;
        return SCHED_OK;
    }
    return SCHED_E_INVAL;
}

int sched_eval_batch_dev(sched_handle h, int kind, int64_t count, const void* candidates,
                         int64_t* tel_out, uint8_t* feasible_out, int32_t* starts_out) {
    KV_ENTER(h);
    return eval_batch_dev(h, kind, count, candidates, (i64*)tel_out, feasible_out, starts_out, nullptr);
}

int sched_eval_batch(sched_handle h, int kind, int64_t count, const void* candidates,
                     int64_t* tel_out, uint8_t* feasible_out, int32_t* starts_out) {
    KV_ENTER(h);
    if (count < 0 || !tel_out || (count > 0 && !candidates)) return SCHED_E_INVAL;
    if (count == 0) return SCHED_OK;
    const int n = h->n;
    size_t cand_bytes = 0; i64 outs = count;
    const bool on_host = count <= kHostCheckMax / n;
    if (kind == SCHED_CAND_ORDER) {
        if (h->batch_handle) return SCHED_E_INVAL;
        if (on_host || n > kDeviceCheckMax) {
            std::vector<unsigned char> seen;
            for (i64 c = 0; c < count; ++c)
                if (!is_permutation((const int32_t*)candidates + c * n, n, seen)) return SCHED_E_NOT_PERMUTATION;
        }
        cand_bytes = (size_t)count * n * sizeof(int);
    } else if (kind == SCHED_CAND_MOVE) {
        if (h->batch_handle || n < 2) return SCHED_E_INVAL;
        const i64 total = neighbourhood_size(n, SCHED_NBHD_SWAP_INSERT, 0);
        for (i64 c = 0; c < count; ++c) {
            i64 code = ((const i64*)candidates)[c];
            if (code < 0 || code >= total) return SCHED_E_INVAL;
        }
        cand_bytes = (size_t)count * sizeof(i64);
    } else if (kind == SCHED_CAND_START_TIMES) {
        if (h->batch_handle || starts_out) return SCHED_E_INVAL;
        if (on_host)
            for (i64 k = 0; k < count * n; ++k)
                if ((unsigned)((const int32_t*)candidates)[k] >= (1u << 30)) return SCHED_E_INVAL;
        cand_bytes = (size_t)count * n * sizeof(int);
    } else if (kind == SCHED_CAND_POLICY) {
        for (i64 c = 0; c < count; ++c) {
            int v = ((const int32_t*)candidates)[c];
            if (v < SCHED_POLICY_FCFS || v > SCHED_POLICY_SORTED_F) return SCHED_E_INVAL;
        }
        cand_bytes = (size_t)count * sizeof(int);
        outs = (i64)h->B * count;
    } else {
        return SCHED_E_INVAL;
    }
    // staging layout: candidates | tel | feasible | starts
    const size_t off_tel = (cand_bytes + 255) & ~(size_t)255;
    const size_t off_feas = off_tel + (((size_t)outs * sizeof(i64) + 255) & ~(size_t)255);
    const size_t off_starts = off_feas + (((size_t)outs + 255) & ~(size_t)255);
    const size_t starts_bytes = starts_out ? (size_t)outs * n * sizeof(int) : 0;
    KV_TRY(ensure_stage(h, off_starts + starts_bytes + 256));
    char* base = (char*)h->d_stage;
    KV_CUDA(cudaMemcpyAsync(base, candidates, cand_bytes, cudaMemcpyHostToDevice, h->stream));
    // orders and start times that are not a few are checked where they have been copied to (a pass over 777
    // orders of 1,531 takes 8 us there and 1.2 ms here).  The evaluation behind the check does nothing if it
    // failed: an order of 2^20 times the longest request would be a schedule of hours, of more rounds than
    // the simulators count
    const bool on_device = !on_host && ((kind == SCHED_CAND_ORDER && n <= kDeviceCheckMax) || kind == SCHED_CAND_START_TIMES);
    const int* bad = on_device ? h->d_result + kResultBad : nullptr;
    if (on_device) {
        KV_CUDA(cudaMemsetAsync(h->d_result + kResultBad, 0, sizeof(int), h->stream));
        if (kind == SCHED_CAND_ORDER) {
            const size_t bits = (((size_t)n + 31) / 32) * sizeof(unsigned);
            KV_CUDA(cudaFuncSetAttribute(k3_check_orders, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 1024));
            k3_check_orders<<<(unsigned)(count < 65535 ? count : 65535), 256, bits, h->stream>>>((const int*)base, n, count, h->d_result + kResultBad);
        } else {
            const i64 total = count * n;
            const i64 blocks = (total + 1023) / 1024;
            k3_check_start_range<<<(unsigned)(blocks < 65535 ? blocks : 65535), 256, 0, h->stream>>>((const int*)base, total, h->d_result + kResultBad);
        }
        KV_TRY(check_launch(h));
    }
    const i64 evaluations = h->evaluations;
    int rc = eval_batch_dev(h, kind, count, base, (i64*)(base + off_tel), feasible_out ? (uint8_t*)(base + off_feas) : nullptr,
                            starts_out ? (int32_t*)(base + off_starts) : nullptr, bad);
    if (rc != SCHED_OK) { cudaStreamSynchronize(h->stream); return rc; }
    if (on_device) {
        const int* res = (const int*)h->h_pinned;
        KV_CUDA(cudaMemcpyAsync(h->h_pinned, h->d_result, 16 * sizeof(int), cudaMemcpyDeviceToHost, h->stream));
        KV_CUDA(cudaStreamSynchronize(h->stream));
        if (res[kResultBad]) {
            h->evaluations = evaluations;
            return kind == SCHED_CAND_ORDER ? SCHED_E_NOT_PERMUTATION : SCHED_E_INVAL;
        }
    }
    KV_CUDA(cudaMemcpyAsync(tel_out, base + off_tel, (size_t)outs * sizeof(i64), cudaMemcpyDeviceToHost, h->stream));
    if (feasible_out) KV_CUDA(cudaMemcpyAsync(feasible_out, base + off_feas, (size_t)outs, cudaMemcpyDeviceToHost, h->stream));
    if (starts_out) KV_CUDA(cudaMemcpyAsync(starts_out, base + off_starts, starts_bytes, cudaMemcpyDeviceToHost, h->stream));
    return read_status(h);
}

int sched_sweep_dev(sched_handle h, int sampled, uint64_t seed, int32_t iteration,
                    int64_t first_code, int64_t count, int64_t* tel_out, int64_t* best_out) {
    KV_ENTER(h);
    if (h->batch_handle || h->n < 2 || count <= 0 || first_code < 0 || !best_out) return SCHED_E_INVAL;
    if (!sampled && first_code + count > neighbourhood_size(h->n, SCHED_NBHD_SWAP_INSERT, 0)) return SCHED_E_INVAL;
    if (((uintptr_t)tel_out & 7) || ((uintptr_t)best_out & 7)) return SCHED_E_INVAL;
    i64* tel = (i64*)tel_out;
    for (i64 done = 0; done < count; done += kSweepChunk) {
        const i64 c = count - done < kSweepChunk ? count - done : kSweepChunk;
        i64* dst;
        if (tel) dst = tel + done;
        else { KV_TRY(ensure_tel(h, c)); dst = h->d_tel; }
        const bool by_slot = tel == nullptr;       // nobody reads the scratch TELs by candidate index
        KV_TRY(launch_moves(h, sampled ? 2 : 1, nullptr, first_code + done, seed, iteration, c, dst, nullptr, by_slot));
        KV_TRY(launch_argmin(h, dst, c, first_code + done, done ? (const i64*)best_out : nullptr, (i64*)best_out,
                             by_slot ? last_launch_order(h, c) : nullptr));
    }
    return SCHED_OK;
}

static int phase1_dp(sched_handle h);
static int phase1_quantile(sched_handle h, u64 seed);

static int sorted_f_common_dev(sched_handle h, int solver, int32_t* order_out, int32_t* batch_offsets_out,
                               int32_t* num_batches_out, int64_t* tel_out, u64 seed = 0) {
    KV_ENTER(h);
    if (h->batch_handle) return SCHED_E_INVAL;
    const int n = h->n;
    cudaStream_t st = h->stream;
    const int* list = h->d_vals_a;              // the batches one behind the other
    if (solver == 0) {
        // S1: ascending (s+o, o, index)
        KV_TRY(sort_rows(h, K1RequestKey{h->d_s, h->d_o, SCHED_POLICY_SORTED_F}, n, 1, h->d_keys_a, h->d_vals_b, h->d_keys_more, h->d_vals_more, h->d_vals_a));
        // S2: prefix sums + F-metric batch boundaries; the sums in shared memory where they fit
        const size_t bytes = 2 * ((size_t)n + 1) * sizeof(i64);
        const bool fits = bytes <= (size_t)h->smem_optin - 4096;
        KV_CUDA(cudaFuncSetAttribute(k2_prefix_f, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 4096));
        k2_prefix_f<<<1, K2_THREADS, fits ? bytes : 0, st>>>(h->d_s, h->d_o, h->d_vals_a, n, h->M, fits ? nullptr : h->d_prefP,
                                                             fits ? nullptr : h->d_prefO, h->d_batch_off, h->d_num_batches,
                                                             (i64)h->g_num, (i64)h->g_den);
        KV_TRY(check_launch(h));
    } else if (solver == 2) {
        KV_TRY(phase1_dp(h));
    } else if (solver == 3) {
        KV_TRY(phase1_quantile(h, seed));
    } else {
        // Algorithm 3: ascending (s+o, index), then first fit + improving swaps, batch after batch
        KV_TRY(sort_rows(h, K1RequestKey{h->d_s, h->d_o, SCHED_POLICY_TOTAL_SIZE}, n, 1, h->d_keys_a, h->d_vals_b, h->d_keys_more, h->d_vals_more, h->d_vals_a));
        if ((i64)h->g_num * h->M + (i64)h->g_den * h->omax >= (1ll << 31)) return SCHED_E_UNSUPPORTED;   // 32-bit weights
        // the solver's arrays in shared memory (21 bytes per request) up to about 11,000 requests
        const size_t bytes = k2l_bytes<unsigned short>(n);
        if (n < 65536 && bytes <= (size_t)h->smem_optin - 2048) {
            KV_CUDA(cudaFuncSetAttribute(k2_local_swap<unsigned short, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 2048));
            k2_local_swap<unsigned short, true><<<1, K2L_THREADS, bytes, st>>>(h->d_s, h->d_o, h->d_vals_a, n, h->M, h->g_num, h->g_den, nullptr,
                                                                         h->d_vals_b, h->d_batch_off, h->d_num_batches, h->d_status);
        } else {
            if (!h->d_ls) KV_TRY(dev_alloc(&h->d_ls, 7 * (size_t)n + 32));
            k2_local_swap<int, false><<<1, K2L_THREADS, 0, st>>>(h->d_s, h->d_o, h->d_vals_a, n, h->M, h->g_num, h->g_den, h->d_ls,
                                                          h->d_vals_b, h->d_batch_off, h->d_num_batches, h->d_status);
        }
        KV_TRY(check_launch(h));
        list = h->d_vals_b;
    }
    // each batch by ascending (o, index)
    KV_TRY(sort_rows(h, K1BatchKey{h->d_o, list, h->d_batch_off, h->d_num_batches}, n, 1, h->d_keys_a,
                     list == h->d_vals_a ? h->d_vals_b : h->d_vals_a, h->d_keys_more, h->d_vals_more, h->d_order));
    h->base_ready = false;
    KV_TRY(ensure_base(h));
    if (order_out) KV_CUDA(cudaMemcpyAsync(order_out, h->d_order, (size_t)n * sizeof(int), cudaMemcpyDeviceToDevice, st));
    if (batch_offsets_out) KV_CUDA(cudaMemcpyAsync(batch_offsets_out, h->d_batch_off, (size_t)(n + 1) * sizeof(int), cudaMemcpyDeviceToDevice, st));
    if (num_batches_out) KV_CUDA(cudaMemcpyAsync(num_batches_out, h->d_num_batches, sizeof(int), cudaMemcpyDeviceToDevice, st));
    if (tel_out) KV_CUDA(cudaMemcpyAsync(tel_out, h->d_base_tel, sizeof(i64), cudaMemcpyDeviceToDevice, st));
    return SCHED_OK;
}

static int sorted_f_common_host(sched_handle h, int solver, int32_t* order_out, int32_t* batch_offsets_out,
                                int32_t* num_batches_out, int64_t* tel_out, u64 seed = 0) {
    KV_ENTER(h);
    KV_TRY(sorted_f_common_dev(h, solver, nullptr, nullptr, nullptr, nullptr, seed));
    const int n = h->n;
    char* hp = (char*)h->h_pinned;
    const bool pinned = reads_through_pinned(n);
    KV_CUDA(cudaMemcpyAsync(hp, h->d_result, pinned ? result_bytes(n) : 16 * sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    KV_CUDA(cudaStreamSynchronize(h->stream));
    const int nb = ((int*)hp)[2], status = ((int*)hp)[3];
    KV_TRY(after_status(h, status));
    if (tel_out) *tel_out = *(i64*)hp;
    if (num_batches_out) *num_batches_out = nb;
    const size_t order_bytes = (size_t)n * sizeof(int), offset_bytes = ((size_t)nb + 1) * sizeof(int);
    if (pinned) {
        if (order_out) memcpy(order_out, hp + order_at(), order_bytes);
        if (batch_offsets_out) memcpy(batch_offsets_out, hp + offsets_at(n), offset_bytes);
    } else {
        if (order_out) KV_CUDA(cudaMemcpyAsync(order_out, h->d_order, order_bytes, cudaMemcpyDeviceToHost, h->stream));
        if (batch_offsets_out) KV_CUDA(cudaMemcpyAsync(batch_offsets_out, h->d_batch_off, offset_bytes, cudaMemcpyDeviceToHost, h->stream));
        KV_CUDA(cudaStreamSynchronize(h->stream));
    }
    return SCHED_OK;
}

// Algorithm 2 batch after batch; leaves the batches (members in ascending index) in d_vals_a and the
// boundaries in d_batch_off / d_num_batches.  Where two tables fit into shared memory ((n+1)(M+1) up to
// 28,000 cells) in one launch; larger ones with one launch per request, synchronised once per batch
// (n <= 128 batches).
static int phase1_dp(sched_handle h) {
    const int n = h->n;
    if (n > 128) return SCHED_E_UNSUPPORTED;
    const int W = (int)h->M + 1, words = (W + 31) / 32;
    const i64 cells_max = (i64)(n + 1) * W;
    if (cells_max > (1ll << 26)) return SCHED_E_UNSUPPORTED;
    cudaStream_t st = h->stream;
    const size_t small_bytes = k2d_small_bytes(n, W);
    if (small_bytes <= (size_t)h->smem_optin - 4096) {
        KV_TRY(ensure_stage(h, (size_t)n * (n + 1) * words * sizeof(unsigned)));
        KV_CUDA(cudaFuncSetAttribute(k2d_small, cudaFuncAttributeMaxDynamicSharedMemorySize, h->smem_optin - 4096));
        k2d_small<<<1, K2D_SMALL_THREADS, small_bytes, st>>>(h->d_s, h->d_o, n, W, words, (unsigned*)h->d_stage, h->d_vals_a,
                                                             h->d_batch_off, h->d_num_batches);
        return check_launch(h);
    }
    int *dpA = nullptr, *dpB = nullptr, *small = nullptr;
    unsigned* took = nullptr;
    int rc = SCHED_OK;
    do {
        if ((rc = dev_alloc(&dpA, (size_t)cells_max)) != SCHED_OK) break;
        if ((rc = dev_alloc(&dpB, (size_t)cells_max)) != SCHED_OK) break;
        if ((rc = dev_alloc(&took, (size_t)n * (n + 1) * words)) != SCHED_OK) break;
        if ((rc = dev_alloc(&small, 8)) != SCHED_OK) break;            // {pick k, m, v, -, nr, nb, done, -}
        int init[8] = {0, 0, 0, 0, n, 0, 0, 0};
        int zero = 0;
#define DP_CUDA(call) if ((call) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), #call); break; }
        DP_CUDA(cudaMemcpyAsync(small, init, sizeof(init), cudaMemcpyHostToDevice, st));
        DP_CUDA(cudaMemcpyAsync(h->d_batch_off, &zero, sizeof(int), cudaMemcpyHostToDevice, st));
        k3_iota<<<(n + 255) / 256, 256, 0, st>>>(h->d_vals_b, n);       // remaining list, ascending index
        if ((rc = check_launch(h)) != SCHED_OK) break;
        int nr = n;
        int* hp = (int*)h->h_pinned;
        while (nr > 0 && rc == SCHED_OK) {
            const int rows = nr + 1;
            const i64 cells = (i64)rows * W;
            k2d_init<<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(dpA, cells);
            if ((rc = check_launch(h)) != SCHED_OK) break;
            int *cur = dpA, *nxt = dpB;
            const i64 threads = (i64)rows * words;
            for (int a = 0; a < nr; ++a) {
                k2d_step<<<(unsigned)((threads + 127) / 128), 128, 0, st>>>(cur, nxt, took + (size_t)a * rows * words, rows, W, words,
                                                                             h->d_s, h->d_o, h->d_vals_b, a);
                if ((rc = check_launch(h)) != SCHED_OK) break;
                int* tmp = cur; cur = nxt; nxt = tmp;
            }
            if (rc != SCHED_OK) break;
            k2d_select<<<1, 1024, 0, st>>>(cur, rows, W, small);
            if ((rc = check_launch(h)) != SCHED_OK) break;
            k2d_apply<<<1, 128, 0, st>>>(h->d_s, h->d_o, took, W, words, rows, small, h->d_vals_b, small + 4,
                                         h->d_vals_a, h->d_batch_off, small + 5, small + 6);
            if ((rc = check_launch(h)) != SCHED_OK) break;
            DP_CUDA(cudaMemcpyAsync(hp, small + 4, sizeof(int), cudaMemcpyDeviceToHost, st));
            DP_CUDA(cudaStreamSynchronize(st));
            if (*hp >= nr) { rc = SCHED_E_INTERNAL; break; }            // every batch places at least one request
            nr = *hp;
        }
        if (rc != SCHED_OK) break;
        DP_CUDA(cudaMemcpyAsync(h->d_num_batches, small + 5, sizeof(int), cudaMemcpyDeviceToDevice, st));
        DP_CUDA(cudaStreamSynchronize(st));
#undef DP_CUDA
    } while (0);
    cudaStreamSynchronize(st);
    if (dpA) kv_free(dpA);
    if (dpB) kv_free(dpB);
    if (took) kv_free(took);
    if (small) kv_free(small);
    return rc;
}

// Algorithm 4 batch after batch; leaves the batches (members in ascending (o, index)) in d_vals_a and
// the boundaries in d_batch_off / d_num_batches.
static int phase1_quantile(sched_handle h, u64 seed) {
    const int n = h->n;
    cudaStream_t st = h->stream;
    // fixed-point ratio key: 2^F must exceed the product of two sizes s+o <= M, and o * 2^F must fit
    const int F = 2 * bits_of((u64)h->M);
    if (F + bits_of((u64)h->omax) > 63) return SCHED_E_UNSUPPORTED;
    // the three orders: the list by (o, index), its places by size, its places by ratio
    int* list = h->d_vals_b;
    int* by_size = (int*)h->d_keys_b;
    int* by_ratio = by_size + n;
    KV_TRY(sort_rows(h, K1RequestKey{h->d_s, h->d_o, SCHED_POLICY_SOF}, n, 1, h->d_keys_a, h->d_vals_a, h->d_keys_more, h->d_vals_more, list));
    KV_TRY(sort_rows(h, K2qSlotKey{h->d_s, h->d_o, list, 0}, n, 1, h->d_keys_a, h->d_vals_a, h->d_keys_more, h->d_vals_more, by_size));
    KV_TRY(sort_rows(h, K2qSlotKey{h->d_s, h->d_o, list, F}, n, 1, h->d_keys_a, h->d_vals_a, h->d_keys_more, h->d_vals_more, by_ratio));
    const size_t bytes = k2q_bytes<unsigned short>(n), room = (size_t)h->smem_optin - sizeof(K2qShared) - 1024;
    const unsigned* leading = nullptr;
    int batches = 0;
    if (n >= kLeadingFrom) {
        // as many batches as there may be: the requests' sizes over M, and half as many again for what batches leave unused
        const double expected = (double)n * (h->mean_s + h->mean_o) / (double)h->M, room_for = (double)(kLeadingBytes / ((size_t)n * sizeof(unsigned)));
        const double most = fmin(16.0 + 1.5 * expected, fmin(room_for, (double)n));
        batches = room_for >= expected ? (int)most : 0;
        if (batches > 0 && ensure_stage(h, (size_t)batches * n * sizeof(unsigned)) != SCHED_OK) {
            cudaGetLastError();                          // without memory for them the solver makes its keys itself
            batches = 0;
        }
        if (batches > 0) {
            leading = (const unsigned*)h->d_stage;
            k2q_leading<<<2 * h->sm_count, 256, 0, st>>>(list, n, batches, seed, (unsigned*)h->d_stage);
            KV_TRY(check_launch(h));
        }
    }
    if (n < 65536 && bytes <= room) {
        KV_CUDA(cudaFuncSetAttribute(k2_quantile<unsigned short>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room));
        k2_quantile<unsigned short><<<1, K2Q_THREADS, bytes, st>>>(h->d_s, h->d_o, list, by_size, by_ratio, n, h->M, seed, nullptr, leading, batches,
                                                                  h->d_vals_a, h->d_batch_off, h->d_num_batches, h->d_status);
    } else {
        if (!h->d_ls) KV_TRY(dev_alloc(&h->d_ls, 7 * (size_t)n + 32));
        k2_quantile<int><<<1, K2Q_THREADS, 0, st>>>(h->d_s, h->d_o, list, by_size, by_ratio, n, h->M, seed, h->d_ls, leading, batches,
                                                    h->d_vals_a, h->d_batch_off, h->d_num_batches, h->d_status);
    }
    return check_launch(h);
}

int sched_sorted_f_dev(sched_handle h, int32_t* order_out, int32_t* batch_offsets_out,
                       int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_dev(h, 0, order_out, batch_offsets_out, num_batches_out, tel_out);
}

int sched_sorted_f_local_swap_dev(sched_handle h, int32_t* order_out, int32_t* batch_offsets_out,
                                  int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_dev(h, 1, order_out, batch_offsets_out, num_batches_out, tel_out);
}

int sched_sorted_f_local_swap(sched_handle h, int32_t* order_out, int32_t* batch_offsets_out,
                              int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_host(h, 1, order_out, batch_offsets_out, num_batches_out, tel_out);
}

int sched_sorted_f_dp(sched_handle h, int32_t* order_out, int32_t* batch_offsets_out,
                      int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_host(h, 2, order_out, batch_offsets_out, num_batches_out, tel_out);
}

int sched_sorted_f_quantile(sched_handle h, uint64_t seed, int32_t* order_out, int32_t* batch_offsets_out,
                            int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_host(h, 3, order_out, batch_offsets_out, num_batches_out, tel_out, (u64)seed);
}

int sched_sorted_f(sched_handle h, int32_t* order_out, int32_t* batch_offsets_out,
                   int32_t* num_batches_out, int64_t* tel_out) {
    return sorted_f_common_host(h, 0, order_out, batch_offsets_out, num_batches_out, tel_out);
}

int sched_local_search(sched_handle h, int neighbourhood, int32_t iters, uint64_t seed,
                       int64_t samples_per_iter, int32_t* order_inout, int64_t* tel_out,
                       int32_t* iters_done_out, int64_t* trace_out) {
    KV_ENTER(h);
    if (h->batch_handle || iters < 0) return SCHED_E_INVAL;
    if (neighbourhood < SCHED_NBHD_SWAP || neighbourhood > SCHED_NBHD_SAMPLED) return SCHED_E_INVAL;
    if (neighbourhood == SCHED_NBHD_SAMPLED && samples_per_iter < 1) return SCHED_E_INVAL;
    const int n = h->n;
    cudaStream_t st = h->stream;
    char* hp = (char*)h->h_pinned;
    const bool pinned = reads_through_pinned(n);
    if (order_inout && pinned) {                     // every path below waits for the stream
        std::vector<unsigned char> seen;
        if (!is_permutation(order_inout, n, seen)) return SCHED_E_NOT_PERMUTATION;
        KV_CUDA(cudaStreamSynchronize(st));
        memcpy(hp, order_inout, (size_t)n * sizeof(int));
        KV_CUDA(cudaMemcpyAsync(h->d_order, hp, (size_t)n * sizeof(int), cudaMemcpyHostToDevice, st));
        h->base_ready = false;
    } else if (order_inout) {
        KV_TRY(sched_set_base_order(h, order_inout));
    }
    const int sampled = neighbourhood == SCHED_NBHD_SAMPLED ? 1 : 0;
    const i64 total = n >= 2 ? neighbourhood_size(n, neighbourhood, samples_per_iter) : 0;
    KV_TRY(ensure_base(h));
    const int* res = (const int*)hp;                 // d_result as read back
    int it = 0;
    for (; it < iters && total > 0; ++it) {
        KV_TRY(ensure_tel(h, total < kSweepChunk ? total : kSweepChunk));
        const bool small = total <= kAcceptSmall;    // the accepting CTA looks for the best itself
        for (i64 done = 0; done < total; done += kSweepChunk) {
            const i64 c = total - done < kSweepChunk ? total - done : kSweepChunk;
            KV_TRY(launch_moves(h, sampled ? 2 : 1, nullptr, done, seed, it, c, h->d_tel, nullptr, true));
            if (!small) KV_TRY(launch_argmin(h, h->d_tel, c, done, done ? h->d_best : nullptr, h->d_best, last_launch_order(h, c)));
        }
        KV_TRY(accept_best(h, h->d_tel, small ? last_launch_order(h, total) : nullptr, small ? total : 0, sampled, seed, it));
        KV_CUDA(cudaMemcpyAsync(hp, h->d_result, 16 * sizeof(int), cudaMemcpyDeviceToHost, st));
        KV_CUDA(cudaStreamSynchronize(st));
        KV_TRY(after_status(h, res[3]));
        const i64 base_tel = ((const i64*)hp)[0], best_tel = ((const i64*)hp)[2], best_code = ((const i64*)hp)[3];
        if (trace_out) { trace_out[2 * it] = best_code; trace_out[2 * it + 1] = best_tel; }
        if (res[8] != 0) {
            // the re-simulated base order must reproduce the TEL that won the sweep
            if (base_tel != best_tel) return SCHED_E_INTERNAL;
        } else if (!sampled) {
            ++it;
            break;
        }
    }
    KV_CUDA(cudaMemcpyAsync(hp, h->d_result, pinned ? order_at() + (size_t)n * sizeof(int) : 16 * sizeof(int), cudaMemcpyDeviceToHost, st));
    KV_CUDA(cudaStreamSynchronize(st));
    KV_TRY(after_status(h, res[3]));
    if (order_inout && pinned) memcpy(order_inout, hp + order_at(), (size_t)n * sizeof(int));
    else if (order_inout) KV_TRY(sched_get_base_order(h, order_inout));
    if (tel_out) *tel_out = *(const i64*)hp;
    if (iters_done_out) *iters_done_out = it;
    return SCHED_OK;
}

int sched_accept_move(sched_handle h, int64_t best_tel, int64_t best_index, int sampled, uint64_t seed,
                      int32_t iteration, int32_t* accepted_out, int64_t* tel_out) {
    KV_ENTER(h);
    if (h->batch_handle || h->n < 2 || best_index < 0 || iteration < 0) return SCHED_E_INVAL;
    const int n = h->n;
    if (!sampled && best_index >= neighbourhood_size(n, SCHED_NBHD_SWAP_INSERT, 0)) return SCHED_E_INVAL;
    cudaStream_t st = h->stream;
    KV_TRY(ensure_base(h));
    i64* hp = (i64*)h->h_pinned;
    KV_CUDA(cudaStreamSynchronize(st));
    hp[0] = best_tel; hp[1] = best_index;
    KV_CUDA(cudaMemcpyAsync(h->d_best, hp, 2 * sizeof(i64), cudaMemcpyHostToDevice, st));
    KV_TRY(accept_best(h, nullptr, nullptr, 0, sampled ? 1 : 0, seed, iteration));
    KV_CUDA(cudaMemcpyAsync(hp, h->d_result, 16 * sizeof(int), cudaMemcpyDeviceToHost, st));
    KV_CUDA(cudaStreamSynchronize(st));
    const int* res = (const int*)hp;                 // d_result as read back
    KV_TRY(after_status(h, res[3]));
    const bool accepted = res[8] != 0;
    // the re-simulated order must reproduce the TEL that the caller's sweep reported for this move
    if (accepted && hp[0] != best_tel) return SCHED_E_INTERNAL;
    if (accepted_out) *accepted_out = accepted ? 1 : 0;
    if (tel_out) *tel_out = hp[0];
    return SCHED_OK;
}

int sched_last_eval_kernel_ms(sched_handle h, float* ms_out) {
    KV_ENTER(h);
    if (!ms_out || !h->ev_valid) return SCHED_E_INVAL;
    KV_CUDA(cudaEventSynchronize(h->ev_k3_end));
    KV_CUDA(cudaEventElapsedTime(ms_out, h->ev_k3_begin, h->ev_k3_end));
    return SCHED_OK;
}

int sched_online_simulate(int32_t B, int32_t n_max, const int32_t* n_each, const int32_t* arrival,
                          const int32_t* s, const int32_t* o, int64_t M, int32_t policy, int32_t period,
                          int32_t lookahead, int32_t* start_out, int64_t* latency_out, float* kernel_ms_out) {
    if (B < 1 || n_max < 1 || n_max > K6_MAX_N || !n_each || !arrival || !s || !o || !start_out || !latency_out)
        return SCHED_E_INVAL;
    if (policy != SCHED_POLICY_FCFS && policy != SCHED_POLICY_SOF && policy != SCHED_POLICY_SORTED_F) return SCHED_E_INVAL;
    if (period < 1 || lookahead < 1 || M < 2) return SCHED_E_INVAL;
    if (M >= (1ll << 30) || lookahead > K6_MAX_LOOKAHEAD) return SCHED_E_UNSUPPORTED;
    int omax = 1;
    for (int b = 0; b < B; ++b) {
        const int n = n_each[b];
        if (n < 1 || n > n_max) return SCHED_E_INVAL;
        const size_t base = (size_t)b * n_max;
        i64 sum_o = 0;
        for (int i = 0; i < n; ++i) {
            const int ai = arrival[base + i], si = s[base + i], oi = o[base + i];
            if (ai < 0 || si < 1 || oi < 1 || (i64)si + oi > M) return SCHED_E_INVAL;
            if (i > 0 && ai < arrival[base + i - 1]) return SCHED_E_INVAL;
            if (ai >= (1 << 29)) return SCHED_E_UNSUPPORTED;
            omax = oi > omax ? oi : omax;
            sum_o += oi;
        }
        if (sum_o >= (1ll << 29)) return SCHED_E_UNSUPPORTED;
    }
    if (omax > K6_MAX_O) return SCHED_E_UNSUPPORTED;
    OnlineParams P;
    memset(&P, 0, sizeof(P));
    P.n_max = n_max; P.M = (int)M; P.policy = policy; P.period = period; P.lookahead = lookahead;
    const int slots = sim_pick_slots(omax), nm = slots <= 32 ? 1 : slots / 32;
    P.L = sim_state_ints(nm, slots);
    const size_t smem = k6_smem_bytes(32 * slots, n_max, lookahead);
    int dev = 0, optin = 0;
    KV_CUDA(cudaGetDevice(&dev));
    KV_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (smem + 1024 > (size_t)optin) return SCHED_E_UNSUPPORTED;
    void (*kernel)(const OnlineParams) = nm == 1 ? k6_online<ChunkSim<1>> : nm == 2 ? k6_online<ChunkSim<2>>
                                       : nm == 4 ? k6_online<ChunkSim<4>> : k6_online<ChunkSim<8>>;
    // the same value for every call: callers on other threads may be between this and their launch
    KV_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024));

    // one block: latency [B], status (8 bytes) | n_each [B] | a, s, o, start [cells each]
    const size_t cells = (size_t)B * n_max;
    const size_t bytes = sizeof(i64) * ((size_t)B + 1) + sizeof(int) * ((size_t)B + 4 * cells);
    char* block = nullptr;
    KV_TRY(dev_alloc(&block, bytes < kPoolMinBlock ? kPoolMinBlock : bytes));
    i64* d_lat = (i64*)block;
    int* d_status = (int*)(d_lat + B);
    int* d_n = (int*)(d_lat + B + 1);
    int* d_a = d_n + B;
    int* d_s = d_a + cells;
    int* d_o = d_s + cells;
    int* d_start = d_o + cells;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = SCHED_OK;
    do {
#define ON_CUDA(call) if ((call) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), #call); break; }
        if (kernel_ms_out) {
            ON_CUDA(cudaEventCreate(&e0));
            ON_CUDA(cudaEventCreate(&e1));
        }
        ON_CUDA(cudaMemcpy(d_n, n_each, sizeof(int) * (size_t)B, cudaMemcpyHostToDevice));
        ON_CUDA(cudaMemcpy(d_a, arrival, sizeof(int) * cells, cudaMemcpyHostToDevice));
        ON_CUDA(cudaMemcpy(d_s, s, sizeof(int) * cells, cudaMemcpyHostToDevice));
        ON_CUDA(cudaMemcpy(d_o, o, sizeof(int) * cells, cudaMemcpyHostToDevice));
        ON_CUDA(cudaMemsetAsync(d_start, 0xff, sizeof(int) * cells, 0));          // -1 where there is no request
        ON_CUDA(cudaMemsetAsync(d_lat, 0, sizeof(i64) * ((size_t)B + 1), 0));
        P.n_each = d_n; P.a = d_a; P.s = d_s; P.o = d_o; P.start_out = d_start; P.latency_out = d_lat; P.status = d_status;
        if (e0) ON_CUDA(cudaEventRecord(e0, 0));
        kernel<<<B, K6_THREADS, smem, 0>>>(P);
        ON_CUDA(cudaGetLastError());
        if (e1) ON_CUDA(cudaEventRecord(e1, 0));
        int status = 0;
        ON_CUDA(cudaMemcpy(&status, d_status, sizeof(int), cudaMemcpyDeviceToHost));
        if (status != 0) { rc = SCHED_E_INTERNAL; break; }
        if ((rc = read_checked_word()) != SCHED_OK) break;
        ON_CUDA(cudaMemcpy(start_out, d_start, sizeof(int) * cells, cudaMemcpyDeviceToHost));
        ON_CUDA(cudaMemcpy(latency_out, d_lat, sizeof(i64) * (size_t)B, cudaMemcpyDeviceToHost));
        if (kernel_ms_out) ON_CUDA(cudaEventElapsedTime(kernel_ms_out, e0, e1));
#undef ON_CUDA
    } while (0);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    kv_free(block);
    return rc;
}

// Shared by the two A_min entry points: validates the scenarios on the host, stages them, runs k7_amin.
// order_host: [B, n_max] host lists, or NULL when order_dev (one device row of n_max entries) is given.
static int amin_run(int32_t B, int32_t n_max, const int32_t* n_each, const int32_t* s, const int32_t* lower,
                    const int32_t* o, int64_t M, const int32_t* order_host, const int32_t* order_dev,
                    int32_t* start_out, int64_t* tel_out, int64_t* evictions_out, int64_t* peak_out,
                    float* kernel_ms_out) {
    if (B < 1 || n_max < 1 || !n_each || !s || !lower || !o || (!order_host && !order_dev) || !start_out || !tel_out)
        return SCHED_E_INVAL;
    if (M < 2) return SCHED_E_INVAL;
    if (n_max > K7_MAX_N || M >= (1ll << 30)) return SCHED_E_UNSUPPORTED;
    int omax = 1;
    std::vector<unsigned char> seen;
    for (int b = 0; b < B; ++b) {
        const int n = n_each[b];
        if (n < 1 || n > n_max) return SCHED_E_INVAL;
        const size_t base = (size_t)b * n_max;
        for (int i = 0; i < n; ++i) {
            const int si = s[base + i], oi = o[base + i], li = lower[base + i];
            if (si < 1 || oi < 1 || li < 1 || li > oi || (i64)si + oi > M) return SCHED_E_INVAL;
            omax = oi > omax ? oi : omax;
        }
        if (order_host) {
            seen.assign((size_t)n, 0);
            for (int q = 0; q < n; ++q) {
                const int id = order_host[base + q];
                if (id < 0 || id >= n || seen[id]) return SCHED_E_NOT_PERMUTATION;
                seen[id] = 1;
            }
        }
    }
    if (omax > K7_MAX_O) return SCHED_E_UNSUPPORTED;
    AminParams P;
    memset(&P, 0, sizeof(P));
    P.n_max = n_max; P.M = (int)M;
    P.L = 32; while (P.L < omax + 2) P.L <<= 1;
    const int slots = sim_pick_slots(omax), nm = slots <= 32 ? 1 : slots / 32;
    P.sim_L = sim_state_ints(nm, slots);
    const size_t smem = k7_smem_bytes(32 * slots, n_max, P.L);
    int dev = 0, optin = 0;
    KV_CUDA(cudaGetDevice(&dev));
    KV_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    if (smem + 1024 > (size_t)optin) return SCHED_E_UNSUPPORTED;
    void (*kernel)(const AminParams) = nm == 1 ? k7_amin<ChunkSim<1>> : nm == 2 ? k7_amin<ChunkSim<2>>
                                     : nm == 4 ? k7_amin<ChunkSim<4>> : k7_amin<ChunkSim<8>>;
    // the same value for every call: callers on other threads may be between this and their launch
    KV_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 1024));

    // one block: tel | evictions | peak [B each], status (8 bytes) | n_each [B] | s, lower, o, order, start [cells each]
    const size_t cells = (size_t)B * n_max, row = sizeof(int) * cells;
    const size_t bytes = sizeof(i64) * (3 * (size_t)B + 1) + sizeof(int) * (size_t)B + 5 * row;
    char* block = nullptr;
    KV_TRY(dev_alloc(&block, bytes < kPoolMinBlock ? kPoolMinBlock : bytes));
    i64* d_res = (i64*)block;
    int* d_status = (int*)(d_res + 3 * (size_t)B);
    int* d_n = (int*)(d_res + 3 * (size_t)B + 1);
    int* d_s = d_n + B;
    int* d_l = d_s + cells;
    int* d_o = d_l + cells;
    int* d_ord = d_o + cells;
    int* d_start = d_ord + cells;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    int rc = SCHED_OK;
    do {
#define AM_CUDA(call) if ((call) != cudaSuccess) { rc = kv_cuda_fail(cudaGetLastError(), #call); break; }
        if (kernel_ms_out) {
            AM_CUDA(cudaEventCreate(&e0));
            AM_CUDA(cudaEventCreate(&e1));
        }
        AM_CUDA(cudaMemcpy(d_n, n_each, sizeof(int) * (size_t)B, cudaMemcpyHostToDevice));
        AM_CUDA(cudaMemcpy(d_s, s, row, cudaMemcpyHostToDevice));
        AM_CUDA(cudaMemcpy(d_l, lower, row, cudaMemcpyHostToDevice));
        AM_CUDA(cudaMemcpy(d_o, o, row, cudaMemcpyHostToDevice));
        if (order_host) AM_CUDA(cudaMemcpy(d_ord, order_host, row, cudaMemcpyHostToDevice));
        AM_CUDA(cudaMemsetAsync(d_start, 0xff, row, 0));                   // -1 where a row has no request
        AM_CUDA(cudaMemsetAsync(d_status, 0, sizeof(i64), 0));
        P.n_each = d_n; P.s = d_s; P.lower = d_l; P.o = d_o;
        P.order = order_host ? d_ord : order_dev;
        P.order_stride = order_host ? (size_t)n_max : 0;
        P.start_out = d_start; P.tel_out = d_res; P.evict_out = d_res + B; P.peak_out = d_res + 2 * (size_t)B;
        P.status = d_status;
        if (e0) AM_CUDA(cudaEventRecord(e0, 0));
        kernel<<<B, 32 * K7_WARPS, smem, 0>>>(P);
        AM_CUDA(cudaGetLastError());
        if (e1) AM_CUDA(cudaEventRecord(e1, 0));
        std::vector<i64> res(3 * (size_t)B + 1);
        AM_CUDA(cudaMemcpy(res.data(), d_res, res.size() * sizeof(i64), cudaMemcpyDeviceToHost));
        if (*(const int*)&res[3 * (size_t)B] != 0) { rc = SCHED_E_INTERNAL; break; }
        if ((rc = read_checked_word()) != SCHED_OK) break;
        AM_CUDA(cudaMemcpy(start_out, d_start, row, cudaMemcpyDeviceToHost));
        memcpy(tel_out, res.data(), sizeof(i64) * (size_t)B);
        if (evictions_out) memcpy(evictions_out, res.data() + B, sizeof(i64) * (size_t)B);
        if (peak_out) memcpy(peak_out, res.data() + 2 * (size_t)B, sizeof(i64) * (size_t)B);
        if (kernel_ms_out) AM_CUDA(cudaEventElapsedTime(kernel_ms_out, e0, e1));
#undef AM_CUDA
    } while (0);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    kv_free(block);
    return rc;
}

int sched_amin_simulate(int32_t B, int32_t n_max, const int32_t* n_each, const int32_t* s, const int32_t* lower,
                        const int32_t* o, int64_t M, const int32_t* order, int32_t* start_out, int64_t* tel_out,
                        int64_t* evictions_out, int64_t* peak_out, float* kernel_ms_out) {
    if (!order) return SCHED_E_INVAL;
    return amin_run(B, n_max, n_each, s, lower, o, M, order, nullptr, start_out, tel_out, evictions_out, peak_out,
                    kernel_ms_out);
}

int sched_sorted_f_amin(int32_t n, const int32_t* s, const int32_t* lower, const int32_t* o, int64_t M,
                        int32_t phase1, int32_t* order_out, int32_t* start_out, int64_t* tel_out,
                        int64_t* evictions_out, int64_t* peak_out) {
    if (n < 1 || !s || !lower || !o || !start_out || !tel_out) return SCHED_E_INVAL;
    if (phase1 != 0 && phase1 != 1) return SCHED_E_INVAL;
    for (int i = 0; i < n; ++i)
        if (s[i] < 1 || o[i] < 1 || lower[i] < 1 || lower[i] > o[i] || (i64)s[i] + o[i] > M) return SCHED_E_INVAL;
    // Phase 1 sees the lower bounds in place of the decode lengths
    sched_handle h = nullptr;
    KV_TRY(sched_init(&h, n, s, lower, M));
    int rc = sorted_f_common_dev(h, phase1, nullptr, nullptr, nullptr, nullptr);
    if (rc == SCHED_OK) rc = sched_sync(h);
    if (rc == SCHED_OK && order_out &&
        cudaMemcpy(order_out, h->d_order, sizeof(int) * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess)
        rc = kv_cuda_fail(cudaGetLastError(), "cudaMemcpy(order_out)");
    if (rc == SCHED_OK)
        rc = amin_run(1, n, &n, s, lower, o, M, nullptr, h->d_order, start_out, tel_out, evictions_out, peak_out, nullptr);
    sched_destroy(h);
    return rc;
}

int sched_build_flags(void) {
#ifdef KVSCHED_CHECKED
    return SCHED_BUILD_CHECKED;
#else
    return 0;
#endif
}

int sched_debug_check_index(int64_t index, int64_t limit) {
#ifdef KVSCHED_CHECKED
    int* sink = nullptr;
    KV_CUDA(cudaMalloc((void**)&sink, sizeof(int)));
    kv_check_index_probe<<<1, 1>>>((long long)index, (long long)limit, sink);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaFree(sink);
    if (e != cudaSuccess) return kv_cuda_fail(e, "kv_check_index_probe");
    return read_checked_word();
#else
    (void)index; (void)limit;
    return SCHED_E_UNSUPPORTED;
#endif
}

int sched_debug_set_loop_cap(int32_t cap) {
    const int v = cap < 0 ? 0x7fffffff : cap;
    KV_CUDA(cudaDeviceSynchronize());           // no kernel of this device may see the value change under it
    KV_CUDA(cudaMemcpyToSymbol(kv_test_loop_cap, &v, sizeof(int)));
    KV_CUDA(cudaDeviceSynchronize());
    return SCHED_OK;
}

int sched_release_cached_memory(void) {
    std::lock_guard<std::mutex> lock(g_pool_mu);
    pool_trim_locked(-1);
    for (const PinnedBlock& b : g_pinned_free) cudaFreeHost(b.p);
    g_pinned_free.clear();
    g_pinned_cached = 0;
    return SCHED_OK;
}

int sched_stats(sched_handle h, int64_t* kernel_launches_out, int64_t* evaluations_out) {
    if (!h) return SCHED_E_INVAL;
    if (kernel_launches_out) *kernel_launches_out = h->launches;
    if (evaluations_out) *evaluations_out = h->evaluations;
    return SCHED_OK;
}

int sched_destroy(sched_handle h) {
    if (!h) return SCHED_E_INVAL;
    DeviceGuard guard(h->device);
    cudaStreamSynchronize(h->stream);
    free_ctx(h);
    return SCHED_OK;
}

const char* sched_strerror(int code) {
    switch (code) {
        case SCHED_OK: return "ok";
        case SCHED_E_INVAL: return "invalid argument";
        case SCHED_E_NOT_PERMUTATION: return "candidate is not a permutation of 0..n-1";
        case SCHED_E_CUDA: return "CUDA runtime error";
        case SCHED_E_NOMEM: return "out of memory";
        case SCHED_E_INTERNAL: return "a bounded device loop hit its cap, or the checked build caught an index outside its array";
        case SCHED_E_UNSUPPORTED: return "size not supported by this build";
        default: return "unknown error code";
    }
}

const char* sched_last_cuda_error(void) { return g_last_cuda_error; }

}  // extern "C"
