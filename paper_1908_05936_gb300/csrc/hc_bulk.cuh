// hc_bulk.cuh -- bulk range calls on tables beyond L2: three passes that let
// the GPU sweep the table once, part by part, instead of reaching for a random
// line of it per request.
//
//   k_bulk_split   a block orders its chunk of kBulkChunk keys (and values) by
//                  table part (one of P equal ranges of buckets) and writes
//                  the chunk in that order to scratch, at the chunk's own
//                  place, with the parts' offsets inside it.  No counts cross
//                  blocks, so any distribution of keys splits the same way.
//   k_bulk_probe   warps take part 0 of every chunk, then part 1, and so on: a
//                  warp gathers a part's runs from a few neighbouring chunks
//                  and probes them like a run of the range kernels.  The warps
//                  in flight share one or two parts, which stay in L2 and
//                  within the reach of the address translation; results go
//                  back to the runs' places.
//   k_bulk_join    a block puts its chunk's results into the input's order.
//
// Why: random reads run at 306 G/s on 64 MB, 78 on 256 MB, 51 on 4 GiB, and
// beyond 512 MB a second request to a line that has just been read costs as
// much as the first (256 MB: nothing), so the range kernels complete about 50 G
// requests/s there whatever DRAM moves: address translation, not bandwidth.
// With a block's lanes in ascending order of address both requests together
// cost what one does.  The probing pass then runs at 60 % of the copy peak
// (lookups; instructions 55 % of issue), the joining pass at 85 %, the
// splitting pass at 56 %.
// Measured against the warp-run kernels (2^28-slot map, 64-byte buckets, 2^26
// keys, G keys/s): present lookups at load factor 0.55 24.0 -> 40.5, inserts
// 0.55 -> 0.8 12.8 -> 22.3, erases 22.2 -> 34.9; 2^26 lookups, half present, at
// 0.8: 3.56 -> 1.89 ms; 30 M set lookups on 10^8 slots 0.84 -> 0.51 ms; the
// 2^28-slot step 25.3 -> 15.4 ms.
// Parts of 32 MB: 16 or 64 MB are within 3 % (4 GiB).  Bringing the next parts
// into L2 ahead of the probes by bulk prefetches loses at every distance from 8
// to 96 MB (lookups 43 -> 32-36 G/s).  256 keys a warp: with 512 or more
// the parts in flight no longer fit L2 (erases 33 -> 28 G/s), with 128 the ends
// of the runs cost more.
#pragma once

#include "hc_core.cuh"
#include "hc_internal.h"
#include "hc_stream.cuh"

namespace hc {

constexpr int kBulkThreads = 512;     // threads of the splitting and joining blocks
static_assert(kBulkParts <= kBulkThreads, "the splitting block scans one part per thread");
constexpr int kBulkRuns = 32;         // runs a probing warp gathers at most: one per lane

static_assert(sizeof(Traits<KIND_MAP_I64_I32>::Val) <= sizeof(Traits<KIND_MAP_I64_I32>::Key) &&
                  sizeof(Traits<KIND_MAP_U64_U64>::Val) <= sizeof(Traits<KIND_MAP_U64_U64>::Key),
              "a lookup's values go over the keys in the scratch");

// The table part of a key: any function of its first bucket that grows with it
// and has `parts` values.  With the mixing hash the bucket is the upper part of
// hash * nb, so the hash's upper word serves as well as the bucket.
__device__ __forceinline__ unsigned part_of(const View &v, unsigned long long key, int parts,
                                            unsigned long long part_mul) {
    if (v.hash_mode == HASH_MIX64) return __umulhi((unsigned)(fmix64(key ^ v.seed) >> 32), (unsigned)parts);
    return (unsigned)__umul64hi(first_bucket(v, key), part_mul);
}

// The E consecutive elements p[i ..) of an array of m (those inside it), by one
// load where the array is aligned for it.
template <class T, int E, class Load, class Load1>
__device__ __forceinline__ void bulk_load(T (&to)[E], const T *p, int i, int m, bool vec, Load load, Load1 load1) {
    if (vec && i + E <= m) {
        load(to, p + i);
    } else {
#pragma unroll
        for (int e = 0; e < E; ++e) to[e] = i + e < m ? load1(p + i + e) : T();
    }
}

// Latency of its phases (load, count, scan, place, store) is what bounds the
// splitting block; reading the keys twice (the second time from L2) instead of
// keeping them in registers lets three or four blocks share an SM (2^24 keys:
// 0.097 -> 0.079 ms), and the part comes from the hash's upper word (2^26 keys:
// 0.295 -> 0.264 ms with the fourth block, 18 bytes a key at 4.6 TB/s).
template <int KIND, bool VALS>
__global__ void __launch_bounds__(kBulkThreads, VALS ? 3 : 4)
k_bulk_split(View v, const typename Traits<KIND>::Key *keys, const typename Traits<KIND>::Val *vals, long long n,
             int parts, unsigned long long part_mul, BulkScratch sc) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    constexpr int NT = kBulkThreads, C = kBulkChunk;
    constexpr int E = 16 / (int)sizeof(Key);              // keys per 16-byte piece
    constexpr int J = C / NT / E;                          // pieces per thread
    extern __shared__ __align__(16) unsigned char smem[];
    Key *sk = reinterpret_cast<Key *>(smem);
    Val *sv = reinterpret_cast<Val *>(smem + C * sizeof(Key));
    uint16_t *so = reinterpret_cast<uint16_t *>(smem + C * (sizeof(Key) + (VALS ? sizeof(Val) : 0)));
    __shared__ unsigned bins[kBulkParts];
    __shared__ unsigned warp_sum[NT / 32];

    const int tid = threadIdx.x;
    const long long c0 = (long long)blockIdx.x * C;
    const int m = (int)(n - c0 < C ? n - c0 : C);
    debug_range(v, c0, m, n);
    const Key *gk = keys + c0;
    const bool vec = (reinterpret_cast<uintptr_t>(gk) & 15) == 0;
    bins[tid] = 0u;
    __syncthreads();
    uint32_t at[J][E];                                     // part << 16 | rank inside it
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int i = (tid + j * NT) * E;
        Key k[E];
        bulk_load(k, gk, i, m, vec,
                  [](Key (&to)[E], const Key *p) { const uint4 u = __ldcg(reinterpret_cast<const uint4 *>(p)); memcpy(to, &u, 16); },
                  [](const Key *p) { return __ldcg(p); });
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (i + e < m) {
                const unsigned p = part_of(v, (unsigned long long)k[e], parts, part_mul);
                at[j][e] = p << 16 | atomicAdd(&bins[p], 1u);
            }
    }
    __syncthreads();
    const unsigned mine = bins[tid];                       // exclusive prefix sum over the parts
    const unsigned lane = tid & 31u, warp = tid >> 5;
    unsigned incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= (unsigned)d) incl += y;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    unsigned before = incl - mine;
    for (unsigned w = 0; w < warp; ++w) before += warp_sum[w];
    bins[tid] = before;
    uint16_t *offs = sc.offs + (long long)blockIdx.x * (parts + 1);
    if (tid < parts) offs[tid] = (uint16_t)before;
    if (tid == 0) offs[parts] = (uint16_t)m;
    __syncthreads();
    // the keys again (they are in L2), now to their places
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int i = (tid + j * NT) * E;
        Key k[E];
        Val val[E];
        bulk_load(k, gk, i, m, vec,
                  [](Key (&to)[E], const Key *p) { const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(p)); memcpy(to, &u, 16); },
                  [](const Key *p) { return ld_stream(p); });
        if constexpr (VALS) {
            constexpr int VP = E * (int)sizeof(Val);       // bytes of the values beside a piece of keys: 8 or 16
            const Val *gv = vals + c0;
            bulk_load(val, gv, i, m, (reinterpret_cast<uintptr_t>(gv) & (VP - 1)) == 0,
                      [](Val (&to)[E], const Val *p) {
                          if constexpr (VP == 16) { const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(p)); memcpy(to, &u, 16); }
                          else { const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p)); memcpy(to, &u, 8); }
                      },
                      [](const Val *p) { return ld_stream(p); });
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (i + e < m) {
                const unsigned to = bins[at[j][e] >> 16] + (at[j][e] & 0xffffu);
                sk[to] = k[e];
                if constexpr (VALS) sv[to] = val[e];
                so[to] = (uint16_t)(i + e);
            }
    }
    __syncthreads();
    // whole 16-byte pieces; the scratch arrays have room to the end of the last chunk's piece
    auto copy = [&](void *to, const void *from, int bytes) {
        uint4 *d = reinterpret_cast<uint4 *>(to);
        const uint4 *s = reinterpret_cast<const uint4 *>(from);
        for (int i = tid; i < (bytes + 15) / 16; i += NT) __stcs(d + i, s[i]);
    };
    copy(reinterpret_cast<Key *>(sc.keys) + c0, sk, m * (int)sizeof(Key));
    if constexpr (VALS) copy(reinterpret_cast<Val *>(sc.vals) + c0, sv, m * (int)sizeof(Val));
    copy(sc.order + c0, so, m * 2);
}

// The runs of one part in up to 32 neighbouring chunks, as one run of keys.
template <int KIND>
struct RunsSrc {
    using Key = typename Traits<KIND>::Key;
    using Val = typename Traits<KIND>::Val;
    const Key *keys;
    const Val *vals;
    const unsigned *start, *upto;          // (shared) first place of a run; keys of it and the runs before it
    unsigned at = 0;
    // place of key i in the scratch
    __device__ __forceinline__ unsigned place(int i) const {
        int lo = 0;                        // first run whose upto is above i
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (upto[lo + step - 1] <= (unsigned)i) lo += step;
        return start[lo] + ((unsigned)i - (lo ? upto[lo - 1] : 0u));
    }
    __device__ __forceinline__ Key key(int i) { at = place(i); return ld_stream(keys + at); }
    __device__ __forceinline__ Val val(int) const { return ld_stream(vals + at); }   // of the key asked for last
    __device__ __forceinline__ bool skip(int) const { return false; }
};

// One warp: the runs of part (warp / groups) in `runs` chunks, R keys at a
// time (one pass, unless the part holds more than its share).  `want`: a lookup
// brings values back.
template <int KIND, int BB, int OP, int NT, int R, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_bulk_probe(View v, BulkScratch sc, int chunks, int parts, int groups, int runs, bool want) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    constexpr bool WHOLE = T::MAP && OP == OP_FIND && BB == 32;    // (2^26 present ones, 4 GiB: 37.4 -> 40.8 G/s)
    __shared__ WarpRun<KIND, OP, R> sh[NT / 32];
    __shared__ unsigned s_start[NT / 32][32], s_upto[NT / 32][32];
    __shared__ BlockCounts sum;
    if constexpr (OP != OP_FIND) sum.init();
    WarpRun<KIND, OP, R> &w = sh[threadIdx.x >> 5];
    unsigned *start = s_start[threadIdx.x >> 5], *upto = s_upto[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int wid = blockIdx.x * (NT / 32) + (threadIdx.x >> 5);
    const int part = wid / groups;
    if (part >= parts) return;
    const int first = (wid % groups) * runs;
    const int cnt = chunks - first < runs ? chunks - first : runs;
    unsigned a = 0, len = 0;
    if (lane < cnt) {
        const uint16_t *o = sc.offs + (long long)(first + lane) * (parts + 1) + part;
        a = o[0];
        len = o[1] - a;
    }
    unsigned incl = len;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    const int total = (int)__shfl_sync(0xffffffffu, incl, 31);
    Counts cnts;
    for (int base = 0; base < total; base += R) {
        const int m = total - base < R ? total - base : R;
        // the places of this pass: keys [base, base + m) of the warp's runs
        const int before = (int)(incl - len) - base;
        start[lane] = (unsigned)(first + lane) * kBulkChunk + a + (before < 0 ? (unsigned)-before : 0u);
        upto[lane] = (int)incl > base ? incl - (unsigned)base : 0u;
        __syncwarp();
        RunsSrc<KIND> src{reinterpret_cast<const Key *>(sc.keys), reinterpret_cast<const Val *>(sc.vals), start, upto};
        if constexpr (OP == OP_INSERT) insert_run<KIND, BB, false>(v, src, m, w.stack, w.st, cnts);
        else if constexpr (OP == OP_FIND) find_run<KIND, BB, WHOLE>(v, src, m, w.stack, w.st, w.vals, want);
        else erase_run<KIND, BB, false>(v, src, m, w.stack, w.st, cnts);
        for (int i = lane; i < m; i += 32) {
            const unsigned to = src.place(i);
            st_stream(sc.out + to, w.st[i]);
            if constexpr (OP == OP_FIND && T::MAP) {
                if (want) st_stream(reinterpret_cast<Val *>(reinterpret_cast<Key *>(sc.keys) + to), w.vals[i]);
            }
        }
        __syncwarp();
    }
    if constexpr (OP != OP_FIND) {
        const int busy = parts * groups - blockIdx.x * (NT / 32);      // warps of this block with a part
        sum.flush(v, cnts, busy < NT / 32 ? busy : NT / 32);
    }
}

template <class Key, class Val, bool VALS>
__global__ void __launch_bounds__(kBulkThreads)
k_bulk_join(long long n, BulkScratch sc, uint8_t *out, Val *vals_out) {
    constexpr int NT = kBulkThreads, C = kBulkChunk, J = C / NT;
    __shared__ __align__(16) Val sv[VALS ? C : 1];
    __shared__ __align__(16) uint8_t ss[C];
    const int tid = threadIdx.x;
    const long long c0 = (long long)blockIdx.x * C;
    const int m = (int)(n - c0 < C ? n - c0 : C);
    uint16_t o[J];
    uint8_t r[J];
    Val val[J];
    const Key *gv = reinterpret_cast<const Key *>(sc.keys) + c0;
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int i = tid + j * NT;
        if (i < m) {
            o[j] = __ldcs(sc.order + c0 + i);
            r[j] = __ldcs(sc.out + c0 + i);
            if constexpr (VALS) val[j] = ld_stream(reinterpret_cast<const Val *>(gv + i));
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int i = tid + j * NT;
        if (i < m) {
            ss[o[j]] = r[j];
            if constexpr (VALS) sv[o[j]] = val[j];
        }
    }
    __syncthreads();
    for (int i = tid; i < m; i += NT) {
        if (out) st_stream(out + c0 + i, ss[i]);
        if constexpr (VALS) st_stream(vals_out + c0 + i, sv[i]);
    }
}

}  // namespace hc
