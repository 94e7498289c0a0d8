// hc_kernels.cuh -- the one-launch-per-call kernels (insert, find, erase,
// clear, rehash) and their launchers, instantiated once per container
// kind by hc_kind_*.cu.
#pragma once

#include "hc_bulk.cuh"
#include "hc_core.cuh"
#include "hc_internal.h"
#include "hc_stream.cuh"

namespace hc {

// ------------------------------------------------------- range kernels ---
// One tile per warp and as many blocks as the call needs: short-lived warps
// let the block scheduler refill an SM as soon as its slowest probes finish.
// (A persistent grid-stride form that prefetched the next tile measured
// 1.3-2x slower on GB300 for every shape.)

// Launch bounds (threads per block[, minimum resident blocks]): a build option,
// since capping registers trades spills for resident warps.
#ifndef HC_INSERT_MAXT
#define HC_INSERT_MAXT 256
#endif
#ifndef HC_INSERT_MINB
#define HC_INSERT_MINB 1
#endif
#ifndef HC_FIND_MAXT
#define HC_FIND_MAXT 256
#endif
#ifndef HC_FIND_MINB
#define HC_FIND_MINB 6   // 40 registers, no spills: +1-7 % for find and erase on GB300
#endif

template <int KIND, int BB, int LB, int KPT>
__global__ void __launch_bounds__(HC_INSERT_MAXT, HC_INSERT_MINB)
k_insert(View v, const typename Traits<KIND>::Key *keys, const typename Traits<KIND>::Val *vals, long long n,
         uint8_t *status, int fold, const uint8_t *skip) {
    constexpr int TILE = Shape<KIND, BB, LB, KPT>::TILE;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    Counts cnt;
    run_tiles<KIND, BB, LB, KPT, 0>(v, keys, vals, skip, status, nullptr, n, warp, (n + TILE - 1) / TILE, warps,
                                    fold != 0, cnt);
    flush_counts(v, cnt);
}

template <int KIND, int BB, int LB, int KPT>
__global__ void __launch_bounds__(HC_FIND_MAXT, HC_FIND_MINB)
k_find(View v, const typename Traits<KIND>::Key *keys, long long n, uint8_t *found,
       typename Traits<KIND>::Val *vals_out) {
    constexpr int TILE = Shape<KIND, BB, LB, KPT>::TILE;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    Counts cnt;
    run_tiles<KIND, BB, LB, KPT, 1>(v, keys, nullptr, nullptr, found, vals_out, n, warp, (n + TILE - 1) / TILE, warps,
                                    false, cnt);
}

template <int KIND, int BB, int LB, int KPT>
__global__ void __launch_bounds__(HC_FIND_MAXT, HC_FIND_MINB)
k_erase(View v, const typename Traits<KIND>::Key *keys, long long n, uint8_t *status, int fold) {
    constexpr int TILE = Shape<KIND, BB, LB, KPT>::TILE;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    Counts cnt;
    run_tiles<KIND, BB, LB, KPT, 2>(v, keys, nullptr, nullptr, status, nullptr, n, warp, (n + TILE - 1) / TILE, warps,
                                    fold != 0, cnt);
    flush_counts(v, cnt);
}

// ---------------------------------------------------------------- clear ---
// Every bucket all-ones bytes (so every key slot is EMPTY; values need no
// initialisation, a value is read only after its key was found), 32-byte
// stores; the header zeroed; then the padding slots of the last bucket become
// tombstones.

static __global__ void __launch_bounds__(256)
k_fill_empty(unsigned char *keys, unsigned long long bytes, Header *hdr) {
    const unsigned long long chunks = bytes / 32;
    const unsigned long long ones = ~0ull;
    for (unsigned long long c = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; c < chunks;
         c += (unsigned long long)gridDim.x * blockDim.x) {
        asm volatile("st.global.v4.u64 [%0], {%1,%1,%1,%1};" ::"l"(keys + c * 32), "l"(ones) : "memory");
    }
    if (blockIdx.x == 0 && threadIdx.x < sizeof(Header) / 8)
        reinterpret_cast<unsigned long long *>(hdr)[threadIdx.x] = 0ull;
}

template <int KIND, int BB>
__global__ void k_pad_tombstones(View v, unsigned long long first, unsigned long long count) {
    using T = Traits<KIND>;
    using S = Slots<KIND, BB>;
    const unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) {
        const unsigned long long slot = first + i;
        *reinterpret_cast<typename T::Key *>(S::key(v, slot / S::SPB, (int)(slot % S::SPB))) = T::TOMB;
    }
}

// --------------------------------------------------------------- rehash ---
// The stored keys of the old array as runs of the insert loop (the keys are
// distinct, and the new table holds no tombstone but its padding).  A warp reads 256
// slots, all loads at once, and its run is the keys that it finds there, so that a
// step has 32 of them however sparse the old array is (with the slots themselves as
// a run whose EMPTY ones were skipped, 2^27 slots with 2^24 keys under the spatial
// hash took 3.0 ms, and so 2.25).  A key's new home keeps its old home's place in
// proportion, so both arrays are swept in order; neighbouring keys share new
// buckets, so inserts scan them from key-dependent slots (View::rotate).  For small
// or crowded tables and the spatial hashes, whose homes are scattered (next section
// for the others).

// Keys of a run: the live ones of slots [first, first + 256).
template <int KIND, int BB>
struct LiveSlots {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using S = Slots<KIND, BB>;
    const View &old_v;
    unsigned long long first;
    const Key *keys;                 // (shared)
    const uint8_t *at;               // (shared) their slots, counted from `first`
    __device__ __forceinline__ Key key(int i) const { return keys[i]; }
    __device__ __forceinline__ bool skip(int) const { return false; }
    __device__ __forceinline__ Val val(int i) const {
        const unsigned long long p = first + at[i];
        return ld_stream(reinterpret_cast<const Val *>(S::val(old_v, p / S::SPB, (int)(p % S::SPB))));
    }
};

template <int KIND, int BB>
__global__ void __launch_bounds__(256, run_blocks(Slots<KIND, BB>::KRB, false))
k_rehash(View old_v, unsigned long long old_phys, View new_v) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using S = Slots<KIND, BB>;
    constexpr int R = 256;
    __shared__ WarpRun<KIND, OP_INSERT, R> sh[8];
    __shared__ Key live_key[8][R];
    __shared__ uint8_t live_at[8][R];
    __shared__ BlockCounts sum;
    sum.init();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long w0 = (unsigned long long)blockIdx.x * 8;
    const unsigned long long first = (w0 + warp) * R;
    if (first >= old_phys) return;
    Key key[R / 32];
#pragma unroll
    for (int j = 0; j < R / 32; ++j) {
        const unsigned long long p = first + j * 32 + lane;
        key[j] = T::EMPTY;
        if (p < old_phys) key[j] = ld_stream(reinterpret_cast<const Key *>(S::key(old_v, p / S::SPB, (int)(p % S::SPB))));
    }
    int n = 0;
#pragma unroll
    for (int j = 0; j < R / 32; ++j) {
        const bool live = key[j] != T::EMPTY && key[j] != T::TOMB;
        const unsigned m = __ballot_sync(0xffffffffu, live);
        if (live) {
            const int to = n + __popc(m & lanes_below());
            live_key[warp][to] = key[j];
            live_at[warp][to] = (uint8_t)(j * 32 + lane);
        }
        n += __popc(m);
    }
    __syncwarp();
    LiveSlots<KIND, BB> src{old_v, first, live_key[warp], live_at[warp]};
    Counts cnts;
    insert_run<KIND, BB, false>(new_v, src, n, sh[warp].stack, sh[warp].st, cnts);
    const unsigned long long busy = (old_phys + R - 1) / R - w0;       // warps of this block with slots
    sum.flush(new_v, cnts, busy < 8 ? (int)busy : 8);
}

// With the mixing hash a key's new home is at the same share of the new array
// as its old one of the old array, so the rehash of a large table builds the new
// array region by region: a block holds kRegionBytes of it in shared memory,
// walks the same share of the old array, puts each key into its new home or the
// next bucket of the region with room (a counter per bucket hands out slots),
// and writes the region out whole, EMPTY slots included.  Keys whose home is
// elsewhere (their old probe crossed a boundary) or whose probe leaves the
// region go to a list that is inserted when every region is there; until then no
// key of the list is looked for, and a bucket that a placed key has passed is
// full for good.  Every line is read or written once, in order: 2^26 slots of
// 64-byte buckets at load factor 0.6, 1.10 ms (fill and runs) -> 0.54 ms, 2 GiB
// at 4 TB/s; what bounds it now is the placing of the keys of a bucket one after
// another.  32 KB: 512 64-byte buckets, about 1 % of the keys cross a boundary,
// and six blocks share an SM.
constexpr int kRegionBytes = 32768;

struct RehashRest {
    unsigned long long *count;       // keys on the list (may exceed cap: then the list is incomplete)
    unsigned long long *pos;         // their slot positions in the old array
    unsigned long long cap;
};

template <int KIND, int BB>
__global__ void __launch_bounds__(256)
k_rehash_regions(View old_v, View new_v, unsigned long long regions, RehashRest rest) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using S = Slots<KIND, BB>;
    constexpr int SPB = S::SPB, M = kRegionBytes / BB;
    __shared__ __align__(16) unsigned char region[kRegionBytes];
    constexpr unsigned kListed = 256;                         // keys on a block's part of the list
    __shared__ unsigned taken[M];
    __shared__ unsigned long long listed[kListed], list_base;
    __shared__ unsigned n_listed;
    __shared__ BlockCounts sum;
    const int tid = threadIdx.x;
    const unsigned long long g = blockIdx.x;
    const unsigned long long n0 = g * new_v.nb / regions, n1 = (g + 1) * new_v.nb / regions;
    const unsigned long long o0 = g * old_v.nb / regions, o1 = (g + 1) * old_v.nb / regions;
    const int size = (int)(n1 - n0);                          // buckets of this region, at most M
    for (int i = tid; i < kRegionBytes / 16; i += 256) reinterpret_cast<uint4 *>(region)[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    for (int i = tid; i < M; i += 256) taken[i] = 0u;
    if (tid == 0) n_listed = 0u;
    sum.init();
    // the last bucket's padding: never handed out, tombstones
    const int last = n1 == new_v.nb ? size - 1 : -1;
    if (last >= 0)
        for (int x = new_v.pad_from + tid; x < SPB; x += 256)
            *reinterpret_cast<Key *>(region + last * BB + x * S::KB) = T::TOMB;
    Counts cnts;
    for (unsigned long long ob0 = o0; ob0 < o1; ob0 += 256) {
        const unsigned long long ob = ob0 + tid;
        LaneWords<S::KRB> kw;
        uint32_t live = 0;
        Val val[T::MAP ? SPB : 1];
        if (ob < o1) {
            kw.load(bucket_at<BB>(old_v, ob));
#pragma unroll
            for (int x = 0; x < SPB; ++x) {
                const Key k = slot_key<KIND, S::KRB>(kw, x);
                live |= (uint32_t)(k != T::EMPTY && k != T::TOMB) << x;
            }
            if constexpr (T::MAP) {
                if (live) {
                    constexpr int VRB = SPB * (int)sizeof(Val);
                    const unsigned char *p = bucket_at<BB>(old_v, ob) + S::KRB;
                    if constexpr (VRB >= 16) {
#pragma unroll
                        for (int q = 0; q < VRB / 16; ++q) {
                            const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(p) + q);
                            memcpy(&val[q * 16 / (int)sizeof(Val)], &u, 16);
                        }
                    } else {
                        const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p));
                        memcpy(&val[0], &u, 8);
                    }
                }
            }
        }
        uint32_t over = 0;                                    // slots whose keys go to the list
#pragma unroll
        for (int x = 0; x < SPB; ++x) {
            if (!(live >> x & 1u)) continue;
            const Key k = slot_key<KIND, S::KRB>(kw, x);
            const unsigned long long home = first_bucket(new_v, (unsigned long long)k);
            bool placed = false;
            if (home >= n0 && home < n1) {
                for (int b = (int)(home - n0); b < size && !placed; ++b) {
                    const unsigned room = b == last ? (unsigned)new_v.pad_from : (unsigned)SPB;
                    if (*(volatile unsigned *)&taken[b] >= room) continue;
                    const unsigned s = atomicAdd(&taken[b], 1u);
                    if (s >= room) continue;
                    *reinterpret_cast<Key *>(region + b * BB + s * S::KB) = k;
                    if constexpr (T::MAP) {
                        *reinterpret_cast<Val *>(region + b * BB + S::KRB + s * S::VB) = val[x];
                        note_claim_key<KIND>(new_v.hdr, k, (long long)((n0 + b) * SPB + s));
                    }
                    placed = true;
                }
            }
            cnts.new_slot += placed;
            over |= (uint32_t)!placed << x;
        }
#pragma unroll
        for (int x = 0; x < SPB; ++x) {
            if (!(over >> x & 1u)) continue;
            const unsigned at = atomicAdd(&n_listed, 1u);
            if (at < kListed) {
                listed[at] = ob * SPB + x;
            } else {
                const unsigned long long to = atomicAdd(rest.count, 1ull);
                if (to < rest.cap) rest.pos[to] = ob * SPB + x;
            }
        }
    }
    __syncthreads();
    const int mine = (int)(n_listed < kListed ? n_listed : kListed);
    if (tid == 0) list_base = mine ? atomicAdd(rest.count, (unsigned long long)mine) : 0ull;
    __syncthreads();
    uint4 *out = reinterpret_cast<uint4 *>(new_v.buckets + n0 * BB);
    for (int i = tid; i < size * BB / 16; i += 256) out[i] = reinterpret_cast<const uint4 *>(region)[i];
    __syncthreads();
    for (int i = tid; i < mine; i += 256)
        if (list_base + i < rest.cap) rest.pos[list_base + i] = listed[i];
    sum.flush(new_v, cnts, 8);
}

template <int KIND, int BB>
struct ListedSlots {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using S = Slots<KIND, BB>;
    const View &old_v;
    const unsigned long long *pos;
    unsigned long long p = 0;
    __device__ __forceinline__ Key key(int i) {
        p = pos[i];
        return *reinterpret_cast<const Key *>(S::key(old_v, p / S::SPB, (int)(p % S::SPB)));
    }
    __device__ __forceinline__ bool skip(int) const { return false; }
    __device__ __forceinline__ Val val(int) const {          // of the key asked for last
        return *reinterpret_cast<const Val *>(S::val(old_v, p / S::SPB, (int)(p % S::SPB)));
    }
};

// The listed keys, in runs that the grid's warps stride over.
template <int KIND, int BB>
__global__ void __launch_bounds__(256, run_blocks(Slots<KIND, BB>::KRB, false))
k_rehash_rest(View old_v, View new_v, RehashRest rest) {
    constexpr int R = 64;
    __shared__ WarpRun<KIND, OP_INSERT, R> sh[8];
    __shared__ BlockCounts sum;
    sum.init();
    WarpRun<KIND, OP_INSERT, R> &w = sh[threadIdx.x >> 5];
    const unsigned long long n = *rest.count < rest.cap ? *rest.count : rest.cap;
    const unsigned long long stride = (unsigned long long)gridDim.x * 8 * R;
    Counts cnts;
    for (unsigned long long first = ((unsigned long long)blockIdx.x * 8 + (threadIdx.x >> 5)) * R; first < n; first += stride) {
        ListedSlots<KIND, BB> src{old_v, rest.pos + first};
        insert_run<KIND, BB, false>(new_v, src, (int)(n - first < R ? n - first : R), w.stack, w.st, cnts);
    }
    sum.flush(new_v, cnts, 8);
}

// ------------------------------------------------------------ launchers ---

inline unsigned grid_for(long long n, int tile, int block) {
    const long long warps = (n + tile - 1) / tile;                // one tile per warp
    return (unsigned)((warps * 32 + block - 1) / block);
}

template <int KIND, int BB, int LB, int KPT>
cudaError_t launch_range_shape(int op, const View &v, const void *keys, const void *vals, long long n, uint8_t *out,
                               void *vals_out, const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    constexpr int TILE = Shape<KIND, BB, LB, KPT>::TILE;
    const int block = sh.block;
    if (n <= 0) return cudaSuccess;
    const unsigned grid = grid_for(n, TILE, block);
    if (op == OP_INSERT)
        k_insert<KIND, BB, LB, KPT><<<grid, block, 0, s>>>(v, (const Key *)keys, (const Val *)vals, n, out, sh.fold, skip);
    else if (op == OP_FIND)
        k_find<KIND, BB, LB, KPT><<<grid, block, 0, s>>>(v, (const Key *)keys, n, out, (Val *)vals_out);
    else
        k_erase<KIND, BB, LB, KPT><<<grid, block, 0, s>>>(v, (const Key *)keys, n, out, sh.fold);
    return cudaGetLastError();
}

// A kernel launched with more than the default 48 KB of dynamic shared
// memory must be allowed it first.
template <class K>
void allow_smem(K kernel, size_t bytes) {
    if (bytes > 48 * 1024) (void)cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Tables from which on the reach of the address translation is what matters.
constexpr long long kBeyondReach = 512ll << 20;
// The same for key regions of 64 and 128 bytes and calls whose one wave would
// take runs of more than 128 keys: 2^20 keys on 384-496 MB, insert / lookup /
// erase with runs of 64 over one wave of 192 or 224 1.08 / 1.05 / 1.04 (map, 128
// bytes), 1.07 / 1.10 / 1.08 (set, 64), 1.18 / 1.17 / 1.09 (set, 128); on 288 MB
// and less 0.85-0.98 but for lookups in 128-byte set buckets.
constexpr long long kWideReach = 352ll << 20;

// The warp-run kernels (keys_per_group 4 or 8), the length of a run: what makes
// one wave of equal runs of the warps that are resident together, if that is at
// most R keys and the table is within reach (an RGB-D frame of 400,000
// candidates 67 us with runs that fill 1.03 waves, 61 with one wave; the
// L2-resident set<u32> workload 64 and 59); 128 for larger calls.  Beyond reach
// shorter runs spread the wait for requests better (10^6 keys on an 800 MB map:
// insert + lookup + erase 264 us in one wave of 192, 237 with 128, 233 with 64;
// erases of 2^22 keys and more prefer 128 by 4 %).  Maps called with arrays in
// host memory: keys and results take longer on the link than a probe takes, and
// more short runs keep more of them on it; calls on 2^23 slots, us, longer runs ->
// 32: 300,000 inserts 50.8 -> 47.3, lookups 40.2 -> 35.9; 2^20 inserts 127 -> 108,
// lookups 106 -> 80.  From 2^21 on inserts and erases are bound by the link or the
// table and 64 keys are as good.  Sets have less to carry: u64 within 5 %, 2^20
// inserts of u32 20 % slower with 32.  Inserts of fewer than 2^22 keys into maps
// with key regions of 32 bytes or less (`narrow_map`) beyond reach: runs of 32 are
// 1-9 % faster than 64 from 400,000 keys on (2^20 into 50 M slots at 0.7, 32- and
// 64-byte buckets 1.07 and 1.04); sets and 128-byte buckets lose 3-19 %.
inline int run_length(int op, long long n, long long resident, int most, bool beyond, bool host_map, bool narrow_map) {
    if (host_map) return op == OP_FIND || n < (1ll << 21) ? 32 : 64;
    const long long wave = (n + resident * 32 - 1) / (resident * 32) * 32;
    if (beyond && op == OP_INSERT && narrow_map && n < (1ll << 22)) return 32;
    if (beyond) return (int)std::min<long long>(wave, op == OP_ERASE ? 128 : 64);
    return wave <= most ? (int)wave : 128;
}

// Tables from which lanes read wide buckets together (see_bucket; between 256
// MB, where it costs 0-17 %, and 512 MB, where it gains 5-50 %).
constexpr long long kTogetherBytes = kBeyondReach;

template <int KIND, int BB, int OP, int R, bool TOGETHER>
cudaError_t launch_run_as(const View &v, const void *keys, const void *vals, long long n, uint8_t *out, void *vals_out,
                       const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    using T = Traits<KIND>;
    const long long resident = (long long)sh.sms * run_blocks(Slots<KIND, BB>::KRB, TOGETHER) * 8;
    const long long bytes = (long long)v.nb * BB;
    const bool beyond = bytes >= (Slots<KIND, BB>::KRB > 32 && n > resident * 128 ? kWideReach : kBeyondReach);
    const int run = run_length(OP, n, resident, R, beyond, sh.host && T::MAP,
                               T::MAP && Slots<KIND, BB>::KRB <= 32);
    const long long per_block = (long long)(sh.block / 32) * run;
    const unsigned grid = (unsigned)((n + per_block - 1) / per_block);
    const size_t smem = sizeof(WarpRun<KIND, OP, R>) * (sh.block / 32);
    allow_smem(k_run<KIND, BB, OP, R, TOGETHER>, smem);
    k_run<KIND, BB, OP, R, TOGETHER><<<grid, sh.block, smem, s>>>(v, (const typename T::Key *)keys, (const typename T::Val *)vals,
                                                        skip, n, run, out, (typename T::Val *)vals_out);
    return cudaGetLastError();
}

template <int KIND, int BB, int OP, int R>
cudaError_t launch_run(const View &v, const void *keys, const void *vals, long long n, uint8_t *out, void *vals_out,
                       const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    if constexpr (Slots<KIND, BB>::KRB > 32) {
        if ((long long)v.nb * BB >= kTogetherBytes)
            return launch_run_as<KIND, BB, OP, R, true>(v, keys, vals, n, out, vals_out, sh, skip, s);
    }
    if constexpr (OP == OP_FIND && Traits<KIND>::MAP && BB == 32) {
        if ((long long)v.nb * BB >= kWholeBytes)
            return launch_run_as<KIND, BB, OP, R, true>(v, keys, vals, n, out, vals_out, sh, skip, s);
    }
    return launch_run_as<KIND, BB, OP, R, false>(v, keys, vals, n, out, vals_out, sh, skip, s);
}

template <int KIND, int BB, int KPT, int S>
cudaError_t launch_find_pair(const View &v, const void *keys, long long n, uint8_t *out, void *vals_out, int block,
                             cudaStream_t s) {
    using T = Traits<KIND>;
    const long long chunk = (long long)(block / 2) * KPT;
    const unsigned grid = (unsigned)((n + chunk - 1) / chunk);
    const size_t smem = (size_t)chunk * (sizeof(typename T::Key) + sizeof(typename T::Val) + 1);
    k_find_pair<KIND, BB, KPT, S><<<grid, block, smem, s>>>(v, (const typename T::Key *)keys, n, out,
                                                            (typename T::Val *)vals_out);
    return cudaGetLastError();
}

template <int KIND, int BB, int LB>
cudaError_t launch_range_kpt(int op, const View &v, const void *keys, const void *vals, long long n, uint8_t *out,
                             void *vals_out, const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    if (sh.keys_per_group >= 4) {       // warp runs, or a lane pair per map key
        if constexpr (Traits<KIND>::MAP && LB == BB && Slots<KIND, BB>::KRB * 2 == BB) {
            if (n <= 0) return cudaSuccess;
            if (op == OP_FIND) {
                if (sh.keys_per_group == 4) return launch_find_pair<KIND, BB, 4, 2>(v, keys, n, out, vals_out, sh.block, s);
                if (sh.keys_per_group == 8) return launch_find_pair<KIND, BB, 8, 4>(v, keys, n, out, vals_out, sh.block, s);
            }
            return cudaErrorInvalidValue;
        }
        if constexpr (LB == Slots<KIND, BB>::KRB) {
            if (n <= 0) return cudaSuccess;
            const bool small = sh.keys_per_group == 4;
            if (!small && sh.keys_per_group != 8) return cudaErrorInvalidValue;
            if (op == OP_INSERT)
                return small ? launch_run<KIND, BB, OP_INSERT, 128>(v, keys, vals, n, out, nullptr, sh, skip, s)
                             : launch_run<KIND, BB, OP_INSERT, 256>(v, keys, vals, n, out, nullptr, sh, skip, s);
            if (op == OP_FIND)
                return small ? launch_run<KIND, BB, OP_FIND, 128>(v, keys, nullptr, n, out, vals_out, sh, nullptr, s)
                             : launch_run<KIND, BB, OP_FIND, 256>(v, keys, nullptr, n, out, vals_out, sh, nullptr, s);
            return small ? launch_run<KIND, BB, OP_ERASE, 128>(v, keys, nullptr, n, out, nullptr, sh, skip, s)
                         : launch_run<KIND, BB, OP_ERASE, 256>(v, keys, nullptr, n, out, nullptr, sh, skip, s);
        }
        return cudaErrorInvalidValue;
    }
    switch (sh.keys_per_group) {
        case 1: return launch_range_shape<KIND, BB, LB, 1>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
        case 2: return launch_range_shape<KIND, BB, LB, 2>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int KIND, int BB>
cudaError_t launch_range_lb(int op, const View &v, const void *keys, const void *vals, long long n, uint8_t *out,
                            void *vals_out, const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    constexpr int KRB = Slots<KIND, BB>::KRB;
    if constexpr (Traits<KIND>::MAP) {
        if (sh.lane_bytes == 16) return launch_range_kpt<KIND, BB, 16>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
    }
    if constexpr (KRB >= 32)
        if (sh.lane_bytes == 32) return launch_range_kpt<KIND, BB, 32>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
    if constexpr (KRB >= 64)
        if (sh.lane_bytes == 64) return launch_range_kpt<KIND, BB, 64>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
    if constexpr (KRB >= 128)
        if (sh.lane_bytes == 128) return launch_range_kpt<KIND, BB, 128>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
    if constexpr (Traits<KIND>::MAP)   // one thread reads keys and values
        if (sh.lane_bytes == BB) return launch_range_kpt<KIND, BB, BB>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
    return cudaErrorInvalidValue;
}

template <int KIND>
cudaError_t launch_range(int op, const View &v, int bucket_bytes, const void *keys, const void *vals, long long n,
                         uint8_t *out, void *vals_out, const LaunchShape &sh, const uint8_t *skip, cudaStream_t s) {
    switch (bucket_bytes) {
        case 32: return launch_range_lb<KIND, 32>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
        case 64: return launch_range_lb<KIND, 64>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
        case 128: return launch_range_lb<KIND, 128>(op, v, keys, vals, n, out, vals_out, sh, skip, s);
        default: return cudaErrorInvalidValue;
    }
}

// The three passes of a bulk call on one piece of n <= kBulkPiece keys.  64
// threads (two warps) per probing block: 24 blocks per SM hold 40 registers, 16
// (wider key regions) 64.
template <int KIND, int BB, int OP>
cudaError_t launch_bulk_op(const View &v, const void *keys, const void *vals, long long n, uint8_t *out, void *vals_out,
                           int parts, void *scratch, cudaStream_t s) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    constexpr bool VIN = T::MAP && OP == OP_INSERT;
    constexpr int KRB = Slots<KIND, BB>::KRB, NT = 64, R = 256, MINB = KRB <= 32 ? 24 : 16;
    BulkScratch sc;
    bulk_scratch(&sc, static_cast<unsigned char *>(scratch), n, parts, (int)sizeof(Key), T::MAP ? (int)sizeof(Val) : 0, OP);
    const int chunks = (int)((n + kBulkChunk - 1) / kBulkChunk);
    const unsigned long long part_mul = (unsigned long long)(((unsigned __int128)parts << 64) / v.nb);
    const size_t smem = (size_t)kBulkChunk * (sizeof(Key) + (VIN ? sizeof(Val) : 0) + 2);
    allow_smem(k_bulk_split<KIND, VIN>, smem);
    k_bulk_split<KIND, VIN><<<chunks, kBulkThreads, smem, s>>>(v, (const Key *)keys, (const Val *)vals, n, parts,
                                                               part_mul, sc);
    // as many runs per warp as fill its keys without spilling into a second round
    const long long want = (long long)R * 7 / 8 * parts / kBulkChunk;
    const int runs = (int)std::max<long long>(1, std::min<long long>(want, kBulkRuns));
    const int groups = (chunks + runs - 1) / runs;
    const unsigned grid = (unsigned)(((long long)parts * groups * 32 + NT - 1) / NT);
    k_bulk_probe<KIND, BB, OP, NT, R, MINB><<<grid, NT, 0, s>>>(v, sc, chunks, parts, groups, runs, vals_out != nullptr);
    if (T::MAP && OP == OP_FIND && vals_out)
        k_bulk_join<Key, Val, true><<<chunks, kBulkThreads, 0, s>>>(n, sc, out, (Val *)vals_out);
    else if (out)
        k_bulk_join<Key, Val, false><<<chunks, kBulkThreads, 0, s>>>(n, sc, out, nullptr);
    return cudaGetLastError();
}

template <int KIND, int BB>
cudaError_t launch_bulk_bb(int op, const View &v, const void *keys, const void *vals, long long n, uint8_t *out,
                           void *vals_out, int parts, void *scratch, cudaStream_t s) {
    switch (op) {
        case OP_INSERT: return launch_bulk_op<KIND, BB, OP_INSERT>(v, keys, vals, n, out, nullptr, parts, scratch, s);
        case OP_FIND: return launch_bulk_op<KIND, BB, OP_FIND>(v, keys, nullptr, n, out, vals_out, parts, scratch, s);
        default: return launch_bulk_op<KIND, BB, OP_ERASE>(v, keys, nullptr, n, out, nullptr, parts, scratch, s);
    }
}

// A bulk call on n keys of any number, piece after piece through one scratch.
template <int KIND>
cudaError_t launch_bulk(int op, const View &v, int bucket_bytes, const void *keys, const void *vals, long long n,
                        uint8_t *out, void *vals_out, int parts, void *scratch, cudaStream_t s) {
    using T = Traits<KIND>;
    const auto *k = static_cast<const typename T::Key *>(keys);
    const auto *val = static_cast<const typename T::Val *>(vals);
    auto *vo = static_cast<typename T::Val *>(vals_out);
    for (long long at = 0; at < n; at += kBulkPiece) {
        const long long m = std::min<long long>(kBulkPiece, n - at);
        const void *pk = k + at, *pv = val ? val + at : nullptr;
        uint8_t *po = out ? out + at : nullptr;
        void *pvo = vo ? vo + at : nullptr;
        cudaError_t e;
        switch (bucket_bytes) {
            case 32: e = launch_bulk_bb<KIND, 32>(op, v, pk, pv, m, po, pvo, parts, scratch, s); break;
            case 64: e = launch_bulk_bb<KIND, 64>(op, v, pk, pv, m, po, pvo, parts, scratch, s); break;
            case 128: e = launch_bulk_bb<KIND, 128>(op, v, pk, pv, m, po, pvo, parts, scratch, s); break;
            default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <int KIND, int BB>
cudaError_t launch_clear_bb(const View &v, unsigned long long phys, unsigned long long capacity, int sm_count,
                            cudaStream_t s) {
    const unsigned long long bytes = v.nb * BB;   // whole buckets: a multiple of 32
    const unsigned long long chunks = bytes / 32;
    unsigned grid = (unsigned)std::min<unsigned long long>((chunks + 255) / 256, (unsigned long long)sm_count * 8);
    if (grid == 0) grid = 1;
    k_fill_empty<<<grid, 256, 0, s>>>(v.buckets, bytes, v.hdr);
    if (phys > capacity) {
        const unsigned long long pad = phys - capacity;
        k_pad_tombstones<KIND, BB><<<(unsigned)((pad + 127) / 128), 128, 0, s>>>(v, capacity, pad);
    }
    return cudaGetLastError();
}

template <int KIND>
cudaError_t launch_clear(const View &v, unsigned long long phys, unsigned long long capacity, int bucket_bytes,
                         int sm_count, cudaStream_t s) {
    switch (bucket_bytes) {
        case 32: return launch_clear_bb<KIND, 32>(v, phys, capacity, sm_count, s);
        case 64: return launch_clear_bb<KIND, 64>(v, phys, capacity, sm_count, s);
        case 128: return launch_clear_bb<KIND, 128>(v, phys, capacity, sm_count, s);
        default: return cudaErrorInvalidValue;
    }
}

template <int KIND>
cudaError_t launch_rehash_regions(const View &old_v, const View &new_v, int bucket_bytes, unsigned long long *count,
                                  unsigned long long *pos, unsigned long long cap, int sms, cudaStream_t s) {
    const RehashRest rest{count, pos, cap};
    const unsigned long long most = kRegionBytes / bucket_bytes, regions = (new_v.nb + most - 1) / most;
    cudaError_t e = cudaMemsetAsync(new_v.hdr, 0, sizeof(Header), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, sizeof *count, s);
    if (e != cudaSuccess) return e;
    const unsigned few = (unsigned)(sms * 4);
    switch (bucket_bytes) {
        case 32: k_rehash_regions<KIND, 32><<<(unsigned)regions, 256, 0, s>>>(old_v, new_v, regions, rest);
                 k_rehash_rest<KIND, 32><<<few, 256, 0, s>>>(old_v, new_v, rest); break;
        case 64: k_rehash_regions<KIND, 64><<<(unsigned)regions, 256, 0, s>>>(old_v, new_v, regions, rest);
                 k_rehash_rest<KIND, 64><<<few, 256, 0, s>>>(old_v, new_v, rest); break;
        case 128: k_rehash_regions<KIND, 128><<<(unsigned)regions, 256, 0, s>>>(old_v, new_v, regions, rest);
                  k_rehash_rest<KIND, 128><<<few, 256, 0, s>>>(old_v, new_v, rest); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int KIND>
cudaError_t launch_rehash(const View &old_v, unsigned long long old_phys, const View &new_v, int bucket_bytes,
                          int sm_count, cudaStream_t s) {
    (void)sm_count;
    View to = new_v;
    to.rotate = 1;
    const unsigned grid = (unsigned)((old_phys + 2047) / 2048);       // 8 runs of 256 slots per block
    switch (bucket_bytes) {
        case 32: k_rehash<KIND, 32><<<grid, 256, 0, s>>>(old_v, old_phys, to); break;
        case 64: k_rehash<KIND, 64><<<grid, 256, 0, s>>>(old_v, old_phys, to); break;
        case 128: k_rehash<KIND, 128><<<grid, 256, 0, s>>>(old_v, old_phys, to); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace hc

// Explicit per-kind entry points used by the host API.
#define HC_INSTANTIATE_KIND(KIND, NAME)                                                                             \
    namespace hc {                                                                                                  \
    cudaError_t NAME##_range(int op, const View &v, int bb, const void *keys, const void *vals, long long n,        \
                             uint8_t *out, void *vals_out, const LaunchShape &sh, const uint8_t *skip,              \
                             cudaStream_t s) {                                                                      \
        return launch_range<KIND>(op, v, bb, keys, vals, n, out, vals_out, sh, skip, s);                            \
    }                                                                                                               \
    cudaError_t NAME##_bulk(int op, const View &v, int bb, const void *keys, const void *vals, long long n,         \
                            uint8_t *out, void *vals_out, int parts, void *scratch, cudaStream_t s) {               \
        return launch_bulk<KIND>(op, v, bb, keys, vals, n, out, vals_out, parts, scratch, s);                       \
    }                                                                                                               \
    cudaError_t NAME##_clear(const View &v, unsigned long long phys, unsigned long long cap, int bb, int sms,       \
                             cudaStream_t s) {                                                                      \
        return launch_clear<KIND>(v, phys, cap, bb, sms, s);                                                        \
    }                                                                                                               \
    cudaError_t NAME##_rehash_regions(const View &ov, const View &nv, int bb, unsigned long long *count,            \
                                      unsigned long long *pos, unsigned long long cap, int sms, cudaStream_t s) {   \
        return launch_rehash_regions<KIND>(ov, nv, bb, count, pos, cap, sms, s);                                    \
    }                                                                                                               \
    cudaError_t NAME##_rehash(const View &ov, unsigned long long ophys, const View &nv, int bb, int sms,            \
                              cudaStream_t s) {                                                                     \
        return launch_rehash<KIND>(ov, ophys, nv, bb, sms, s);                                                      \
    }                                                                                                               \
    }
