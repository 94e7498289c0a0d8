// hc_batch.cu -- the batched form: many range calls on many tables in one
// persistent launch per phase (insert, then find, then erase), optionally
// captured once into a CUDA graph and replayed.
//
// Scheduling.  Every item is cut into chunks of `tile` keys.  A phase of warp runs
// has one warp per chunk; lock-step phases, and runs with blocks_per_sm, are a
// persistent grid whose warps take the next chunk from a counter.  A warp finds the
// item its chunk belongs to by a search over the items' chunk offsets and runs the
// same loops as the one-launch-per-call kernels over the chunk.  Tables of very
// different sizes are therefore balanced at chunk granularity, and no launch is
// spent per table.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/hc.h"
#include "hc_core.cuh"
#include "hc_internal.h"
#include "hc_stream.cuh"
#include "hc_table.h"

namespace hc {

struct BatchItemDev {
    View v;
    const void *keys;
    const void *vals;
    uint8_t *out;
    void *vals_out;
    long long n;
    long long chunk_begin;   // first chunk number of this item within its phase
    int bb;
    int fold;
};

// Work of one phase launch: items [item0, item0 + n_items) of one kind.
struct PhaseDesc {
    int kind;
    int op;
    int bb;        // bucket bytes of every table in the phase
    int item0;
    int n_items;
    long long n_chunks;
    int counter;   // index of this phase's chunk counter
};

constexpr int kCounterBytes = 512;       // room for 36 phases' counters behind the descriptors

template <int KIND, int OP, int BB, int LB, int KPT>
__device__ __forceinline__ void run_chunk(const BatchItemDev &it, long long k0, long long k1) {
    using T = Traits<KIND>;
    constexpr int TILE = Shape<KIND, BB, LB, KPT>::TILE;
    // keys past the chunk end belong to the next chunk: n is clamped to k1
    Counts cnt;
    run_tiles<KIND, BB, LB, KPT, OP>(it.v, (const typename T::Key *)it.keys, (const typename T::Val *)it.vals, nullptr,
                                     it.out, (typename T::Val *)it.vals_out, k1, k0 / TILE, (k1 + TILE - 1) / TILE, 1,
                                     it.fold != 0, cnt);
    if constexpr (OP != OP_FIND) flush_counts(it.v, cnt);
}

// The next chunk of a phase, for the whole warp.
__device__ __forceinline__ long long next_chunk(unsigned long long *counter) {
    unsigned long long c = 0;
    if ((threadIdx.x & 31) == 0) c = atomicAdd(counter, 1ull);
    return (long long)__shfl_sync(0xffffffffu, c, 0);
}

__global__ void k_zero_counters(unsigned long long *c, int n) {
    if (threadIdx.x < n) c[threadIdx.x] = 0ull;
}

// The item that chunk c of a phase belongs to: the last one whose chunk_begin
// is at most c.  The whole warp calls it.
__device__ __forceinline__ int item_of(const BatchItemDev *items, int n_items, long long c) {
    const int lane = threadIdx.x & 31;
    int lo = 0, n = n_items;
    while (n > 1) {
        const int step = (n + 31) / 32, at = lane * step;
        const unsigned m = __ballot_sync(0xffffffffu, at < n && items[lo + (at < n ? at : 0)].chunk_begin <= c);
        const int k = (__popc(m) - 1) * step;              // chunk_begin ascends: m is a run of low bits
        lo += k;
        n = n - k < step ? n - k : step;
    }
    return lo;
}

// One phase launch covers items of one kind, one op and one bucket size (so
// each launch is a small specialisation).  WIDE: one thread per key reading
// the whole bucket (maps: keys and values) or key region (sets); otherwise
// 32-byte lanes.
//
// A counter rather than a warp per chunk: warps of a chunk of up to 1024 keys end
// at very different times, and a block's place is free only when its last one has
// (128 tables, one key per thread: 320 us, 384 with a warp per chunk).
template <int KIND, int OP, int BB, int WIDE, int KPT>
__global__ void __launch_bounds__(256)
k_batch_phase(const BatchItemDev *__restrict__ items, int n_items, long long n_chunks, int tile,
              unsigned long long *counter) {
    constexpr int KRB = Slots<KIND, BB>::KRB;
    constexpr int LB = WIDE ? (Traits<KIND>::MAP ? BB : KRB) : (KRB < 32 ? KRB : 32);
    for (long long c = next_chunk(counter); c < n_chunks; c = next_chunk(counter)) {
        int lo = 0, hi = n_items - 1;                      // last item whose chunk_begin is at most c
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (items[mid].chunk_begin <= c) lo = mid;
            else hi = mid - 1;
        }
        const BatchItemDev it = items[lo];
        const long long k0 = (c - it.chunk_begin) * tile;
        const long long k1 = k0 + tile < it.n ? k0 + tile : it.n;
        debug_range(it.v, k0, k1 - k0, it.n);
        run_chunk<KIND, OP, BB, LB, KPT>(it, k0, k1);
    }
}

// The warp-run form of a phase (keys_per_group 4 or 8, the default): a warp
// works through its chunk in runs of up to R keys with the range kernels' probe
// loops.  Inserts and erases run at the rate at which a compare-and-swap follows
// a read of the same line inside L2 (50 G/s; the tables of the chunks in flight
// are there), lookups at 60 % of the copy peak.  Against lock-step phases whose
// warps took chunks from one counter: 192 set<u64> of 2^10-2^20 slots, 25 M
// operations, 750 -> 547 us; 1024 tables, 127 M operations, 3.21 -> 2.50 ms.
//
// Blocks of 256 threads per SM that it is compiled for: 4 (64 registers) and 3 (80)
// for 128-byte key regions, fewer than the range kernels' (run_blocks), since a phase
// holds its item's fields beside the probes.
// At 5 for every key region all instances spilled, the widest most, and a batch of
// set<u64> with 128-byte buckets was slower than its lock-step phases: 5 M lookups on
// 256 MB 124 -> 143 us, 112 so; erases 70 -> 81, 64; 128 tables' erases 42 -> 49, 34.
constexpr int batch_blocks(int krb) { return krb == 128 ? 3 : 4; }

template <int KIND, int OP, int BB, int R>
__global__ void __launch_bounds__(256, batch_blocks(Slots<KIND, BB>::KRB))
k_batch_run(const BatchItemDev *__restrict__ items, int n_items, long long n_chunks, int tile,
            unsigned long long *counter) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    extern __shared__ __align__(16) unsigned char smem[];
    WarpRun<KIND, OP, R> &w = reinterpret_cast<WarpRun<KIND, OP, R> *>(smem)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    // without a counter: one warp per chunk
    for (long long c = counter ? next_chunk(counter) : ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
         c < n_chunks; c = counter ? next_chunk(counter) : n_chunks) {
        const BatchItemDev &it = items[item_of(items, n_items, c)];
        const View v = it.v;
        const long long k0 = (c - it.chunk_begin) * tile;
        const long long k1 = k0 + tile < it.n ? k0 + tile : it.n;
        Counts cnts;
        for (long long p0 = k0; p0 < k1; p0 += R) {
            const int m = (int)(k1 - p0 < R ? k1 - p0 : R);
            debug_range(v, p0, m, it.n);
            ArraySrc<KIND> src{(const Key *)it.keys + p0, (const Val *)it.vals + p0, nullptr};
            if constexpr (OP == OP_INSERT) insert_run<KIND, BB, false>(v, src, m, w.stack, w.st, cnts);
            else if constexpr (OP == OP_FIND && T::MAP && BB == 32) {
                // as the range lookups (5 M, half present, on a 512 MB table: lock-step
                // phases, which read whole buckets too, 136 us; keys and values apart 145;
                // so 130)
                if ((long long)v.nb * BB >= kWholeBytes) find_run<KIND, BB, true>(v, src, m, w.stack, w.st, w.vals, it.vals_out != nullptr);
                else find_run<KIND, BB, false>(v, src, m, w.stack, w.st, w.vals, it.vals_out != nullptr);
            } else if constexpr (OP == OP_FIND) find_run<KIND, BB, false>(v, src, m, w.stack, w.st, w.vals, it.vals_out != nullptr);
            else erase_run<KIND, BB, false>(v, src, m, w.stack, w.st, cnts);
            for (int i = lane; i < m; i += 32) {
                if (it.out) st_stream(it.out + p0 + i, w.st[i]);
                if constexpr (OP == OP_FIND && T::MAP) {
                    if (it.vals_out) st_stream((Val *)it.vals_out + p0 + i, w.vals[i]);
                }
            }
            __syncwarp();                                  // the results have left before the next run's
        }
        if constexpr (OP != OP_FIND) flush_counts(v, cnts);
    }
}

using PhaseKernel = void (*)(const BatchItemDev *, int, long long, int, unsigned long long *);

template <int KIND, int OP, int BB>
PhaseKernel pick_lb_kpt(int lb, int kpt) {
    if (kpt == 4) return k_batch_run<KIND, OP, BB, 128>;
    if (kpt == 8) return k_batch_run<KIND, OP, BB, 256>;
    if (lb == 0) return kpt == 1 ? k_batch_phase<KIND, OP, BB, 1, 1> : k_batch_phase<KIND, OP, BB, 1, 2>;
    return kpt == 1 ? k_batch_phase<KIND, OP, BB, 0, 1> : k_batch_phase<KIND, OP, BB, 0, 2>;
}

// Dynamic shared memory of a phase launch (the warp-run form's stacks and results).
template <int KIND>
size_t run_smem(int op, int kpt) {
    if (kpt == 4) return op == OP_INSERT ? sizeof(WarpRun<KIND, 0, 128>) : op == OP_FIND ? sizeof(WarpRun<KIND, 1, 128>) : sizeof(WarpRun<KIND, 2, 128>);
    return op == OP_INSERT ? sizeof(WarpRun<KIND, 0, 256>) : op == OP_FIND ? sizeof(WarpRun<KIND, 1, 256>) : sizeof(WarpRun<KIND, 2, 256>);
}

size_t phase_smem(int kind, int op, int kpt, int block) {
    if (kpt < 4) return 0;
    const size_t warp = kind == KIND_SET_U32 ? run_smem<KIND_SET_U32>(op, kpt)
                        : kind == KIND_SET_U64 ? run_smem<KIND_SET_U64>(op, kpt)
                        : kind == KIND_MAP_I64_I32 ? run_smem<KIND_MAP_I64_I32>(op, kpt) : run_smem<KIND_MAP_U64_U64>(op, kpt);
    return warp * (size_t)(block / 32);
}

// A phase kernel with more than the default 48 KB of dynamic shared memory
// must be allowed it before its occupancy is queried or it is launched.
void allow_phase_smem(PhaseKernel k, size_t bytes) {
    if (bytes > 48 * 1024) (void)cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int KIND, int OP>
PhaseKernel pick_bb(int bb, int lb, int kpt) {
    if (bb == 32) return pick_lb_kpt<KIND, OP, 32>(lb, kpt);
    if (bb == 64) return pick_lb_kpt<KIND, OP, 64>(lb, kpt);
    return pick_lb_kpt<KIND, OP, 128>(lb, kpt);
}

template <int KIND>
PhaseKernel pick_op(int op, int bb, int lb, int kpt) {
    if (op == OP_INSERT) return pick_bb<KIND, OP_INSERT>(bb, lb, kpt);
    if (op == OP_FIND) return pick_bb<KIND, OP_FIND>(bb, lb, kpt);
    return pick_bb<KIND, OP_ERASE>(bb, lb, kpt);
}

PhaseKernel pick_kernel(int kind, int op, int bb, int lb, int kpt) {
    switch (kind) {
        case KIND_SET_U32: return pick_op<KIND_SET_U32>(op, bb, lb, kpt);
        case KIND_SET_U64: return pick_op<KIND_SET_U64>(op, bb, lb, kpt);
        case KIND_MAP_I64_I32: return pick_op<KIND_MAP_I64_I32>(op, bb, lb, kpt);
        default: return pick_op<KIND_MAP_U64_U64>(op, bb, lb, kpt);
    }
}

}  // namespace hc

struct hc_batch {
    uint32_t magic;
    int device;
    int block, blocks_per_sm, tile, lane_bytes, kpt;
    bool use_graph;
    void *d_mem = nullptr;
    hc::BatchItemDev *d_items = nullptr;
    unsigned long long *d_counters = nullptr;      // behind the items
    std::vector<hc::PhaseDesc> phases;
    int sms = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

// Errors go to the same thread-local message as the rest of the API (owned
// by hc_api.cu).
hc_rc hc_internal_fail(hc_rc rc, const char *msg);

namespace {

constexpr uint32_t kBatchMagic = 0x48434241u;

// tile 0 in the configuration: keys per chunk chosen from the total work so
// that the chunks can occupy every warp slot of the GPU (64 per SM): a power of
// two from 128 to 1024, to 256 for warp runs (192 set<u64> of 2^10-2^20 slots,
// 25 M operations, with chunks of 128, 256, 512, 1024: 554, 547, 578, 609 us).
int auto_tile(const hc_batch_item *items, int64_t n_items, int kpt) {
    const int most = kpt >= 4 ? 256 : 1024;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                   cudaSuccess || sms <= 0) {
        (void)cudaGetLastError();
        return most;
    }
    long long total = 0;
    for (int64_t i = 0; i < n_items; ++i)
        if (items[i].n > 0) total += items[i].n;
    const long long per_slot = total / ((long long)sms * 64);
    int tile = 128;
    while (tile < most && (long long)tile * 2 <= per_slot) tile *= 2;
    return tile;
}

hc_rc bfail(hc_rc rc, const std::string &msg) { return hc_internal_fail(rc, msg.c_str()); }

hc_rc bcuda(cudaError_t e, const char *what) {
    return bfail(HC_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// Whether the phases' warps take their chunks from counters (a persistent grid).
bool counted(int kpt, int per_sm) { return kpt < 4 || per_sm > 0; }

// Threads per block where the configuration leaves it open (64: warp runs, one
// warp per chunk; a grid of per_sm blocks per SM keeps the warps that it has had).
int default_block(int kpt, int per_sm) { return counted(kpt, per_sm) ? 256 : 64; }

// Blocks of a phase: as many as give every chunk a warp, and for counted phases at
// most per_sm (0: what fits) per SM.
cudaError_t phase_grid(const hc::PhaseDesc &ph, hc::PhaseKernel k, int kpt, int block, size_t smem, int per_sm, int sms,
                       unsigned *grid) {
    long long g = (ph.n_chunks * 32 + block - 1) / block;
    if (counted(kpt, per_sm)) {
        cudaError_t e = cudaSuccess;
        if (per_sm <= 0) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem);
        if (e != cudaSuccess) return e;
        g = std::min<long long>(g, (long long)sms * std::max(per_sm, 1));
    }
    *grid = (unsigned)std::max<long long>(g, 1);
    return cudaSuccess;
}

// Enqueues the phases over descriptors and counters that are on the device.
hc_rc enqueue_phases(const hc::PhaseDesc *phases, int n_phases, const hc::BatchItemDev *d_items,
                     unsigned long long *d_counters, int lane_bytes, int kpt, int block, int per_sm, int tile, int sms,
                     cudaStream_t s) {
    cudaError_t e;
    const bool counters = counted(kpt, per_sm);
    if (n_phases == 0) return HC_OK;
    if (counters) {
        hc::k_zero_counters<<<1, 64, 0, s>>>(d_counters, n_phases);
        e = cudaGetLastError();
        if (e != cudaSuccess) return bcuda(e, "resetting the batch counters");
    }
    for (int p = 0; p < n_phases; ++p) {
        const hc::PhaseDesc &ph = phases[p];
        hc::PhaseKernel k = hc::pick_kernel(ph.kind, ph.op, ph.bb, lane_bytes, kpt);
        const size_t smem = hc::phase_smem(ph.kind, ph.op, kpt, block);
        hc::allow_phase_smem(k, smem);
        unsigned grid = 0;
        e = phase_grid(ph, k, kpt, block, smem, per_sm, sms, &grid);
        if (e != cudaSuccess) return bcuda(e, "querying the occupancy of a batch phase");
        k<<<grid, block, smem, s>>>(d_items + ph.item0, ph.n_items, ph.n_chunks, tile,
                                    counters ? d_counters + ph.counter : nullptr);
        e = cudaGetLastError();
        if (e != cudaSuccess) return bcuda(e, "launching a batch phase");
    }
    return HC_OK;
}

hc_rc enqueue(hc_batch *b, cudaStream_t s) {
    return enqueue_phases(b->phases.data(), (int)b->phases.size(), b->d_items, b->d_counters, b->lane_bytes, b->kpt,
                          b->block, b->blocks_per_sm, b->tile, b->sms, s);
}

}  // namespace

extern "C" {

HC_API hc_rc hc_batch_create(hc_batch **out, const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg,
                             void *stream) {
    if (!out) return bfail(HC_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (n_items < 0 || (n_items > 0 && !items)) return bfail(HC_ERR_ARG, "bad item list");
    hc_batch_config c{};
    if (cfg) c = *cfg;
    const int lb = c.lane_bytes;
    const int kpt = c.keys_per_group ? c.keys_per_group : 8;
    const int block = c.block ? c.block : default_block(kpt, c.blocks_per_sm);
    const int tile = c.tile ? c.tile : auto_tile(items, n_items, kpt);
    if (lb != 0 && lb != 32) return bfail(HC_ERR_ARG, "lane_bytes must be 0 (whole bucket) or 32");
    if (kpt != 1 && kpt != 2 && kpt != 4 && kpt != 8)
        return bfail(HC_ERR_ARG, "keys_per_group must be 1 or 2 (lock-step) or 4 or 8 (warp runs)");
    if (block < 64 || block > 256 || block % 32) return bfail(HC_ERR_ARG, "block must be a multiple of 32 in [64, 256]");
    if (tile < 128 || tile % 128) return bfail(HC_ERR_ARG, "tile must be a positive multiple of 128");

    // items ordered by (op, kind) so each phase launch sees one contiguous run
    std::vector<hc::BatchItemDev> dev;
    std::vector<hc::PhaseDesc> phases;
    for (int op = 0; op < 3; ++op) {
        for (int kind = 0; kind < 4; ++kind)
        for (int bb = 32; bb <= 128; bb *= 2) {
            hc::PhaseDesc ph{kind, op, bb, (int)dev.size(), 0, 0, (int)phases.size()};
            for (int64_t i = 0; i < n_items; ++i) {
                const hc_batch_item &it = items[i];
                if (!it.table || it.table->magic != HC_TABLE_MAGIC) return bfail(HC_ERR_ARG, "item with a bad table");
                if (it.op < 0 || it.op > 2) return bfail(HC_ERR_ARG, "item with a bad op");
                if (it.n < 0) return bfail(HC_ERR_ARG, "item with n < 0");
                if (it.op != op || it.table->kind != kind || it.table->bucket_bytes != bb || it.n == 0) continue;
                const bool map = kind >= HC_MAP_I64_I32;
                const int kb = kind == HC_SET_U32 ? 4 : 8;
                if (!it.d_keys || reinterpret_cast<uintptr_t>(it.d_keys) % kb)
                    return bfail(HC_ERR_ARG, "item keys NULL or misaligned");
                if (op == HC_OP_INSERT && map && !it.d_vals) return bfail(HC_ERR_ARG, "insert item on a map without values");
                if (op == HC_OP_FIND && !it.d_out) return bfail(HC_ERR_ARG, "find item without a found array");
                hc::BatchItemDev d{};
                d.v = it.table->view;
                d.v.rotate = it.n > (long long)d.v.nb ? 1 : 0;
                d.keys = it.d_keys;
                d.vals = map ? it.d_vals : nullptr;
                d.out = it.d_out;
                d.vals_out = map ? it.d_vals_out : nullptr;
                d.n = it.n;
                d.chunk_begin = ph.n_chunks;
                d.bb = it.table->bucket_bytes;
                d.fold = op == HC_OP_FIND ? 0 : it.table->shape[op].fold;
                ph.n_chunks += (it.n + tile - 1) / tile;
                dev.push_back(d);
                ph.n_items++;
            }
            if (ph.n_items) phases.push_back(ph);
        }
    }

    hc_batch *b = new hc_batch();
    b->magic = kBatchMagic;
    b->block = block;
    b->tile = tile;
    b->lane_bytes = lb;
    b->kpt = kpt;
    b->blocks_per_sm = c.blocks_per_sm;
    b->use_graph = c.use_graph != 0;
    b->phases = phases;
    cudaError_t e = cudaGetDevice(&b->device);
    const size_t items_bytes = (dev.size() * sizeof(hc::BatchItemDev) + 255) / 256 * 256;
    if (e == cudaSuccess) e = cudaMalloc(&b->d_mem, items_bytes + hc::kCounterBytes);
    if (e != cudaSuccess) {
        delete b;
        return bcuda(e, "allocating the batch descriptors");
    }
    b->d_items = static_cast<hc::BatchItemDev *>(b->d_mem);
    b->d_counters = reinterpret_cast<unsigned long long *>(static_cast<char *>(b->d_mem) + items_bytes);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (!dev.empty())
        e = cudaMemcpyAsync(b->d_items, dev.data(), dev.size() * sizeof(hc::BatchItemDev), cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    if (e == cudaSuccess && b->use_graph) {
        // capture on a private stream so the caller's stream is never in capture mode
        cudaStream_t cs;
        e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
        if (e == cudaSuccess) {
            e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
            hc_rc rc = HC_OK;
            if (e == cudaSuccess) rc = enqueue(b, cs);
            cudaError_t e2 = cudaStreamEndCapture(cs, &b->graph);
            if (e == cudaSuccess) e = e2;
            if (rc != HC_OK && e == cudaSuccess) e = cudaErrorUnknown;
            if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
            cudaStreamDestroy(cs);
        }
    }
    if (e != cudaSuccess) {
        if (b->exec) cudaGraphExecDestroy(b->exec);
        if (b->graph) cudaGraphDestroy(b->graph);
        cudaFree(b->d_mem);
        delete b;
        return bcuda(e, "building the batch");
    }
    *out = b;
    return HC_OK;
}

HC_API hc_rc hc_batch_launch(hc_batch *b, void *stream) {
    if (!b || b->magic != kBatchMagic) return bfail(HC_ERR_ARG, "invalid batch handle");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (b->exec) {
        cudaError_t e = cudaGraphLaunch(b->exec, s);
        if (e != cudaSuccess) return bcuda(e, "launching the batch graph");
        return HC_OK;
    }
    return enqueue(b, s);
}

HC_API hc_rc hc_batch_destroy(hc_batch *b) {
    if (!b) return HC_OK;
    if (b->magic != kBatchMagic) return bfail(HC_ERR_ARG, "invalid batch handle");
    b->magic = 0;
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    cudaError_t e = cudaFree(b->d_mem);
    delete b;
    if (e != cudaSuccess) return bcuda(e, "cudaFree");
    return HC_OK;
}

}  // extern "C"

// ---- batched form without any device allocation --------------------------
// hc_batch_create allocates its item descriptors with cudaMalloc.  This variant keeps them in one file-scope device array instead,
// for callers that must not allocate device memory themselves.  The array is
// part of the library image: every GPU that loads the library holds it until
// the process exits, and every call shares it.

namespace {

constexpr int kNoAllocMaxItems = 1024;   // items per call (104 KiB of descriptors)
constexpr int kNoAllocMaxPhases = 36;    // 3 operations x 4 container kinds x 3 bucket sizes

struct NoAllocScratch {
    hc::BatchItemDev items[kNoAllocMaxItems];
    unsigned long long counters[64];
};

}  // namespace

// The scratch itself.  Host code must not take its address directly (on the
// host this name is only a stand-in); the device address comes from
// cudaGetSymbolAddress, once per device.
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

namespace {

std::mutex g_noalloc_mu;
NoAllocScratch *g_noalloc_addr[64] = {nullptr};   // device address per device ordinal

// Set-up, once per device, with that device current.
hc_rc noalloc_scratch(int dev, NoAllocScratch **out) {
    if (dev < 0 || dev >= 64) return bfail(HC_ERR_ARG, "device ordinal out of range");
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) return bcuda(e, "cudaGetSymbolAddress of the static batch scratch");
        g_noalloc_addr[dev] = static_cast<NoAllocScratch *>(p);
    }
    *out = g_noalloc_addr[dev];
    return HC_OK;
}

// Host-side staging of the descriptors: per host thread, fixed size, so a
// call allocates no memory on the host either.
thread_local hc::BatchItemDev t_noalloc_items[kNoAllocMaxItems];

}  // namespace

extern "C" {

HC_API hc_rc hc_batch_run_noalloc(const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg,
                                  void *stream) {
    if (n_items < 0 || (n_items > 0 && !items)) return bfail(HC_ERR_ARG, "bad item list");
    if (n_items > kNoAllocMaxItems)
        return bfail(HC_ERR_ARG, "hc_batch_run_noalloc takes at most 1024 items per call (got " +
                                     std::to_string((long long)n_items) + ")");
    hc_batch_config c{};
    if (cfg) c = *cfg;
    const int lb = c.lane_bytes;
    const int kpt = c.keys_per_group ? c.keys_per_group : 8;
    const int block = c.block ? c.block : default_block(kpt, c.blocks_per_sm);
    const int tile = c.tile ? c.tile : auto_tile(items, n_items, kpt);
    if (lb != 0 && lb != 32) return bfail(HC_ERR_ARG, "lane_bytes must be 0 (whole bucket) or 32");
    if (kpt != 1 && kpt != 2 && kpt != 4 && kpt != 8)
        return bfail(HC_ERR_ARG, "keys_per_group must be 1 or 2 (lock-step) or 4 or 8 (warp runs)");
    if (block < 64 || block > 256 || block % 32) return bfail(HC_ERR_ARG, "block must be a multiple of 32 in [64, 256]");
    if (tile < 128 || tile % 128) return bfail(HC_ERR_ARG, "tile must be a positive multiple of 128");
    if (c.use_graph) return bfail(HC_ERR_ARG, "hc_batch_run_noalloc launches directly; use_graph must be 0");

    // descriptors ordered by (op, kind), one phase per non-empty pair
    hc::PhaseDesc phases[kNoAllocMaxPhases];
    int n_phases = 0, n_dev = 0;
    for (int op = 0; op < 3; ++op) {
        for (int kind = 0; kind < 4; ++kind)
        for (int bb = 32; bb <= 128; bb *= 2) {
            hc::PhaseDesc ph{kind, op, bb, n_dev, 0, 0, n_phases};
            for (int64_t i = 0; i < n_items; ++i) {
                const hc_batch_item &it = items[i];
                if (!it.table || it.table->magic != HC_TABLE_MAGIC) return bfail(HC_ERR_ARG, "item with a bad table");
                if (it.op < 0 || it.op > 2) return bfail(HC_ERR_ARG, "item with a bad op");
                if (it.n < 0) return bfail(HC_ERR_ARG, "item with n < 0");
                if (it.op != op || it.table->kind != kind || it.table->bucket_bytes != bb || it.n == 0) continue;
                const bool map = kind >= HC_MAP_I64_I32;
                const int kb = kind == HC_SET_U32 ? 4 : 8;
                if (!it.d_keys || reinterpret_cast<uintptr_t>(it.d_keys) % kb)
                    return bfail(HC_ERR_ARG, "item keys NULL or misaligned");
                if (op == HC_OP_INSERT && map && !it.d_vals) return bfail(HC_ERR_ARG, "insert item on a map without values");
                if (op == HC_OP_FIND && !it.d_out) return bfail(HC_ERR_ARG, "find item without a found array");
                hc::BatchItemDev &d = t_noalloc_items[n_dev++];
                d = hc::BatchItemDev{};
                d.v = it.table->view;
                d.v.rotate = it.n > (long long)d.v.nb ? 1 : 0;
                d.keys = it.d_keys;
                d.vals = map ? it.d_vals : nullptr;
                d.out = it.d_out;
                d.vals_out = map ? it.d_vals_out : nullptr;
                d.n = it.n;
                d.chunk_begin = ph.n_chunks;
                d.bb = it.table->bucket_bytes;
                d.fold = op == HC_OP_FIND ? 0 : it.table->shape[op].fold;
                ph.n_chunks += (it.n + tile - 1) / tile;
                ph.n_items++;
            }
            if (ph.n_items) phases[n_phases++] = ph;
        }
    }
    if (n_phases == 0) return HC_OK;

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return bcuda(e, "cudaGetDevice");
    NoAllocScratch *scratch = nullptr;
    hc_rc rc = noalloc_scratch(dev, &scratch);
    if (rc != HC_OK) return rc;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return bcuda(e, "reading the SM count");

    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // pageable source: the call returns once the descriptors are staged, so
    // the per-thread array may be refilled by the next call
    e = cudaMemcpyAsync(scratch->items, t_noalloc_items, (size_t)n_dev * sizeof(hc::BatchItemDev),
                        cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return bcuda(e, "copying the batch descriptors");
    return enqueue_phases(phases, n_phases, scratch->items, scratch->counters, lb, kpt, block, c.blocks_per_sm, tile, sms,
                          s);
}

}  // extern "C"

// ---- dynamic batched launch with caller scratch ---------------------------
// The served form forms a new batch at every dispatch.  Building a graph or
// allocating descriptors per dispatch would cost more than small requests
// themselves, so the caller hands in a device scratch buffer (one per stream
// it dispatches on) that receives the descriptors.

namespace {

constexpr int kRunMaxItems = 4096;
thread_local hc::BatchItemDev t_run_items[kRunMaxItems];

}  // namespace

extern "C" {

HC_API int64_t hc_batch_scratch_bytes(int64_t n_items) {
    if (n_items < 0 || n_items > kRunMaxItems) return -1;
    return (int64_t)((n_items * sizeof(hc::BatchItemDev) + 255) / 256 * 256 + hc::kCounterBytes);
}

namespace {
hc_rc batch_run(const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg, void *d_scratch,
                int64_t scratch_bytes, void *h_pinned, void *stream);
}

HC_API hc_rc hc_batch_run(const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg, void *d_scratch,
                          int64_t scratch_bytes, void *stream) {
    return batch_run(items, n_items, cfg, d_scratch, scratch_bytes, nullptr, stream);
}

namespace {
hc_rc batch_run(const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg, void *d_scratch,
                int64_t scratch_bytes, void *h_pinned, void *stream) {
    if (n_items < 0 || (n_items > 0 && !items)) return bfail(HC_ERR_ARG, "bad item list");
    if (n_items > kRunMaxItems)
        return bfail(HC_ERR_ARG, "hc_batch_run takes at most 4096 items per call (got " +
                                     std::to_string((long long)n_items) + ")");
    if (n_items == 0) return HC_OK;
    const int64_t need = hc_batch_scratch_bytes(n_items);
    if (!d_scratch || scratch_bytes < need || reinterpret_cast<uintptr_t>(d_scratch) % 256)
        return bfail(HC_ERR_ARG, "scratch must be 256-byte aligned and hold hc_batch_scratch_bytes(n_items) = " +
                                     std::to_string((long long)need) + " bytes");
    hc_batch_config c{};
    if (cfg) c = *cfg;
    const int lb = c.lane_bytes;
    const int kpt = c.keys_per_group ? c.keys_per_group : 8;
    const int block = c.block ? c.block : default_block(kpt, c.blocks_per_sm);
    const int tile = c.tile ? c.tile : auto_tile(items, n_items, kpt);
    if (lb != 0 && lb != 32) return bfail(HC_ERR_ARG, "lane_bytes must be 0 (whole key region) or 32");
    if (kpt != 1 && kpt != 2 && kpt != 4 && kpt != 8)
        return bfail(HC_ERR_ARG, "keys_per_group must be 1 or 2 (lock-step) or 4 or 8 (warp runs)");
    if (block < 64 || block > 256 || block % 32) return bfail(HC_ERR_ARG, "block must be a multiple of 32 in [64, 256]");
    if (tile < 128 || tile % 128) return bfail(HC_ERR_ARG, "tile must be a positive multiple of 128");

    hc::BatchItemDev *desc = h_pinned ? static_cast<hc::BatchItemDev *>(h_pinned) : t_run_items;
    hc::PhaseDesc phases[36];
    int n_phases = 0, n_dev = 0;
    for (int op = 0; op < 3; ++op) {
        for (int kind = 0; kind < 4; ++kind)
        for (int bb = 32; bb <= 128; bb *= 2) {
            hc::PhaseDesc ph{kind, op, bb, n_dev, 0, 0, n_phases};
            for (int64_t i = 0; i < n_items; ++i) {
                const hc_batch_item &it = items[i];
                if (!it.table || it.table->magic != HC_TABLE_MAGIC) return bfail(HC_ERR_ARG, "item with a bad table");
                if (it.op < 0 || it.op > 2) return bfail(HC_ERR_ARG, "item with a bad op");
                if (it.n < 0) return bfail(HC_ERR_ARG, "item with n < 0");
                if (it.op != op || it.table->kind != kind || it.table->bucket_bytes != bb || it.n == 0) continue;
                const bool map = kind >= HC_MAP_I64_I32;
                const int kb = kind == HC_SET_U32 ? 4 : 8;
                if (!it.d_keys || reinterpret_cast<uintptr_t>(it.d_keys) % kb)
                    return bfail(HC_ERR_ARG, "item keys NULL or misaligned");
                if (op == HC_OP_INSERT && map && !it.d_vals) return bfail(HC_ERR_ARG, "insert item on a map without values");
                if (op == HC_OP_FIND && !it.d_out) return bfail(HC_ERR_ARG, "find item without a found array");
                hc::BatchItemDev &d = desc[n_dev++];
                d = hc::BatchItemDev{};
                d.v = it.table->view;
                d.v.rotate = it.n > (long long)d.v.nb ? 1 : 0;
                d.keys = it.d_keys;
                d.vals = map ? it.d_vals : nullptr;
                d.out = it.d_out;
                d.vals_out = map ? it.d_vals_out : nullptr;
                d.n = it.n;
                d.chunk_begin = ph.n_chunks;
                d.bb = it.table->bucket_bytes;
                d.fold = op == HC_OP_FIND ? 0 : it.table->shape[op].fold;
                ph.n_chunks += (it.n + tile - 1) / tile;
                ph.n_items++;
            }
            if (ph.n_items) phases[n_phases++] = ph;
        }
    }
    if (n_phases == 0) return HC_OK;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return bcuda(e, "reading the device");
    auto *d_items = static_cast<hc::BatchItemDev *>(d_scratch);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    e = cudaMemcpyAsync(d_items, desc, (size_t)n_dev * sizeof(hc::BatchItemDev), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return bcuda(e, "copying the batch descriptors");
    auto *d_counters = reinterpret_cast<unsigned long long *>(static_cast<char *>(d_scratch) + need - hc::kCounterBytes);
    return enqueue_phases(phases, n_phases, d_items, d_counters, lb, kpt, block, c.blocks_per_sm, tile, sms, s);
}
}  // namespace

}  // extern "C"

namespace hc {
// hc_batch_run for callers that own page-locked staging for the descriptors
// (the served loop: one buffer per launch slot, reused only after the slot's
// launch completed), so that their copy to the device does not wait for the
// stream.
hc_rc batch_run_pinned(const hc_batch_item *items, int64_t n_items, const hc_batch_config *cfg, void *d_scratch,
                       int64_t scratch_bytes, void *h_pinned, void *stream) {
    return batch_run(items, n_items, cfg, d_scratch, scratch_bytes, h_pinned, stream);
}
size_t batch_desc_bytes(int64_t n_items) { return (size_t)n_items * sizeof(BatchItemDev); }
}  // namespace hc
