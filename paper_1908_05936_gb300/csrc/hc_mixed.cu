// hc_mixed.cu -- free-running mixed batches: inserts, finds and erases of one
// call run at once (Section 4, "Guarantees": concurrency across all
// operations).  Per key, the results are those of some serial order of that
// key's operations; inserts claim EMPTY slots only, and a map insert claims
// its slot with the CLAIM marker, stores the value, then the key, exactly as
// the in-kernel functions of include/hc_device.cuh do (whose waiting rule and
// special keys it shares).
//
// The kernel has the shape of the range kernels (warp runs): a warp works
// through a run of operations, those that stay undecided wait on its stack.  In
// a step all compare-and-swaps go out together; a map insert's claim and its
// publication happen in the same step, around one fence that also orders the
// step's lookups of found keys before their value reads; no claim is left in
// progress from one step to the next, so a wait on a claim always ends.  Results
// leave in coalesced stores, counters with one atomic per block.
//
// Against a kernel that staged a block's operations and kept two per thread in
// flight (50 / 30 / 20 inserts, lookups, erases): 2^22 on a 256 MB map 236 -> 216
// us, on a 256 MB set 149 -> 130, 2^18 on a 16 MB map 50 -> 32, 2^24 on a 4 GiB
// map 1.08 -> 1.06 ms; what bounds the large ones is a map insert's three
// scattered requests (claim, value, key) after its read.  Eight blocks per SM (64
// registers): without the cap 244 us for the first, at ten 1.09 ms for the last.
#include <algorithm>
#include <cstdint>

#include "hc.h"
#include "hc_device.cuh"
#include "hc_internal.h"
#include "hc_stream.cuh"

namespace hc {

namespace {

constexpr int kMixedBlock = 128;  // threads per block
constexpr int kMixedRun = 128;    // operations per run at most

enum : uint8_t { MOP_INSERT = 0, MOP_FIND = 1, MOP_ERASE = 2 };

// The operations on keys that live outside the regular slots' probing: the
// side-slot patterns, and for maps the key equal to CLAIM.  Rare, so they go
// through the in-kernel functions (which count for themselves).
template <int KIND, int BB>
__device__ __noinline__ void special_op(const View &v, uint8_t op, typename Traits<KIND>::Key k,
                                        typename Traits<KIND>::Val *val, uint8_t *st) {
    using T = Traits<KIND>;
    if (op == MOP_INSERT) {
        *st = (uint8_t)hcd::detail::insert<KIND, BB>(v, k, (unsigned long long)*val).status;
        *val = typename T::Val();
    } else if (op == MOP_FIND) {
        const long long pos = hcd::detail::find<KIND, BB>(v, k);
        *st = pos != hcd::END;
        *val = pos != hcd::END ? hcd::detail::value_at<KIND, BB>(v, pos) : typename T::Val();
    } else {
        *st = (uint8_t)hcd::detail::erase<KIND, BB>(v, k);
        *val = typename T::Val();
    }
}

// The operations in flight of a warp: key, bucket << 16 | kind << 14 | position
// in the run, an insert's value.
template <int KIND>
struct MixedRun {
    using T = Traits<KIND>;
    unsigned long long at[kStack];
    typename T::Key key[kStack];
    typename T::Val val[T::MAP ? kStack : 1];
    typename T::Val vals[T::MAP ? kMixedRun : 1];            // found values out
    unsigned lost;                                           // swaps lost to other keys and waits for claims
    uint8_t st[kMixedRun];
};

template <int KIND, int BB>
__global__ void __launch_bounds__(kMixedBlock, 8)
k_mixed_run(View v, const uint8_t *ops, const typename Traits<KIND>::Key *keys, const typename Traits<KIND>::Val *vals,
            long long n, int run, uint8_t *status, typename Traits<KIND>::Val *vals_out) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using Sl = Slots<KIND, BB>;
    constexpr int SPB = Sl::SPB, WARPS = kMixedBlock / 32;
    __shared__ MixedRun<KIND> sh[WARPS];
    __shared__ BlockCounts sum;
    sum.init();
    MixedRun<KIND> &w = sh[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const long long w0 = (long long)blockIdx.x * WARPS;
    const long long c0 = (w0 + (threadIdx.x >> 5)) * run;
    if (c0 >= n) return;
    const int cnt = (int)(n - c0 < run ? n - c0 : run);
    debug_range(v, c0, cnt, n);
    keys += c0;
    ops += c0;
    if constexpr (T::MAP) vals += c0;

    Counts cnts;
    int next = 0, top = 0;
    Key ahead = Key();
    Val ahead_val = Val();
    uint8_t ahead_op = 0;
    auto fetch = [&](int i) {
        if (i >= cnt) return;
        ahead = ld_stream(keys + i);
        if constexpr (T::MAP) ahead_val = ld_stream(vals + i);
        ahead_op = ld_stream(ops + i);
    };
    fetch(lane);
    if (lane == 0) w.lost = 0u;              // (a __syncwarp follows before the first swap)
    // One more lost swap or wait; whether the run's operations have met more of
    // them than kMaxRestarts each (the limit that keeps the loop finite).
    auto too_many = [&]() { return atomicAdd(&w.lost, 1u) >= (unsigned)cnt * kMaxRestarts; };
    unsigned long long reach = 0;
    for (;; ++reach) {
        Key key;
        Val val = Val();
        uint8_t op;
        unsigned long long b = 0;
        int idx;
        bool act;
        if (top < 32 && next < cnt) {
            key = ahead;
            val = ahead_val;
            op = ahead_op == MOP_INSERT ? MOP_INSERT : ahead_op == MOP_FIND ? MOP_FIND : MOP_ERASE;
            idx = next + lane;
            act = idx < cnt;
            next += 32;
            fetch(next + lane);
            bool special = side_index<KIND>(key) >= 0;
            if constexpr (T::MAP) special = special || key == T::CLAIM;
            if (act && special) {
                Val out = val;
                special_op<KIND, BB>(v, op, key, &out, &w.st[idx]);
                if constexpr (T::MAP) w.vals[idx] = out;
                act = false;
            }
            b = first_bucket(v, (unsigned long long)key);
        } else if (top > 0) {
            const int take = top < 32 ? top : 32;
            top -= take;
            act = lane < take;
            const int p = top + (act ? lane : 0);
            const unsigned long long e = w.at[p];
            key = w.key[p];
            if constexpr (T::MAP) val = w.val[p];
            idx = (int)(e & 0x3fffu);
            op = (uint8_t)(e >> 14 & 3u);
            b = e >> 16;
        } else {
            break;
        }
        __syncwarp();                        // entries are read before this step's survivors overwrite them
        const Seen seen = see_bucket<KIND, BB, false, true>(v, act, b, key);
        // an operation is over with result st; a map's value is 0 but for a found key
        bool left = act;
        auto done = [&](uint32_t st) {
            w.st[idx] = (uint8_t)st;
            if constexpr (T::MAP) w.vals[idx] = Val();
            left = false;
        };
        int q = -1;                          // the slot of this step's swap, or of a found key's value
        bool swap = false;
        if (act) {
            const uint32_t le = seen.empty;
            bool full = false;
            if (op == MOP_INSERT) {
                const int rot = slot_rotation<SPB>((unsigned long long)key);
                bool wait = false;
                if (seen.hit) {              // stored (and, for maps, published with its value)
                    done(ST_EXISTS);
                } else {
                    if constexpr (T::MAP) {  // the stored CLAIM-pattern key, or claims in progress
                        if (seen.tomb) wait = hcd::detail::must_wait<SPB>(v, b, seen.tomb, le, rot);
                    }
                    if (wait) {              // the bucket is read again
                        if (too_many()) {    // a claim that never resolves
                            atomicOr(&v.hdr->err, ERR_PROBE_BOUND);
                            cnts.over = 1;
                            done(ST_OVERFLOW);
                        }
                    } else if (le) {
                        q = hcd::detail::first_from<SPB>(le, rot);
                        swap = true;
                    } else {
                        full = true;
                    }
                }
            } else if (seen.hit) {
                q = __ffs(seen.hit) - 1;
                swap = op == MOP_ERASE;
                if constexpr (!T::MAP) {
                    if (!swap) done(1u);
                }
            } else if (le) {
                done(op == MOP_FIND ? 0u : (uint32_t)ST_NOT_FOUND);
            } else {
                full = true;
            }
            if (full) {
                b = next_bucket(v, b);
                if (came_round(v, (unsigned long long)key, b, reach)) {
                    if (op == MOP_INSERT) cnts.over = 1;
                    done(op == MOP_INSERT ? (uint32_t)ST_OVERFLOW : op == MOP_FIND ? 0u : (uint32_t)ST_NOT_FOUND);
                }
            }
        }
        bool publish = false;
        if (swap) {
            unsigned char *slot = Sl::key(v, b, q);
            if (op == MOP_ERASE) {
                // a failed swap means a concurrent erase of the same key won
                const bool won = cas_key<KIND>(slot, key, T::TOMB) == key;
                cnts.del += won ? 1u : 0u;
                done(won ? (uint32_t)ST_ERASED : (uint32_t)ST_NOT_FOUND);
            } else {
                const Key old = cas_key<KIND>(slot, T::EMPTY, T::MAP ? T::CLAIM : key);
                if (old == T::EMPTY) {
                    ++cnts.ins;
                    ++cnts.new_slot;
                    if constexpr (T::MAP) {
                        store_val<KIND, BB>(v, b, q, (unsigned long long)val);
                        publish = true;
                    } else {
                        done(ST_INSERTED);
                    }
                } else if (!T::MAP && old == key) {
                    done(ST_EXISTS);         // an equal key won the slot
                } else if (too_many()) {
                    atomicOr(&v.hdr->err, ERR_PROBE_BOUND);
                    cnts.over = 1;
                    done(ST_OVERFLOW);
                }
                // otherwise another key took the slot: the same bucket is read again
            }
        }
        if constexpr (T::MAP) {
            const bool reading = act && left && op == MOP_FIND && q >= 0;
            if (publish || reading) {
                // the claimed slots' values before their keys; the found keys'
                // loads before their values' loads
                __threadfence();
                if (publish) {
                    hcd::detail::store_key<KIND>(Sl::key(v, b, q), key);
                    done(ST_INSERTED);
                } else {
                    w.vals[idx] = (Val)load_val<KIND, BB>(v, b, q);
                    w.st[idx] = 1;
                    left = false;
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int p = top + __popc(mask & lanes_below());
            w.at[p] = b << 16 | (unsigned)op << 14 | (unsigned)idx;
            w.key[p] = key;
            if constexpr (T::MAP) w.val[p] = val;
        }
        top += __popc(mask);
        __syncwarp();
    }
    __syncwarp();
    for (int i = lane; i < cnt; i += 32) {
        if (status) st_stream(status + c0 + i, w.st[i]);
        if constexpr (T::MAP) {
            if (vals_out) st_stream(vals_out + c0 + i, w.vals[i]);
        }
    }
    const long long busy = (n + run - 1) / run - w0;         // warps of this block with operations
    sum.flush(v, cnts, (int)(busy < WARPS ? busy : WARPS));
}

template <int KIND, int BB>
cudaError_t launch_bb(const View &v, const uint8_t *ops, const void *keys, const void *vals, long long n,
                      uint8_t *status, void *vals_out, cudaStream_t s) {
    using T = Traits<KIND>;
    // at least 32 warps on each of 128 SMs before runs grow
    const int run = (int)std::min<long long>(kMixedRun, (n + 4096 * 32 - 1) / (4096 * 32) * 32);
    const long long per_block = (long long)(kMixedBlock / 32) * run;
    const unsigned grid = (unsigned)((n + per_block - 1) / per_block);
    k_mixed_run<KIND, BB><<<grid, kMixedBlock, 0, s>>>(v, ops, (const typename T::Key *)keys, (const typename T::Val *)vals,
                                                       n, run, status, (typename T::Val *)vals_out);
    return cudaGetLastError();
}

template <int KIND>
cudaError_t launch(const hc_device_view &dv, const uint8_t *ops, const void *keys, const void *vals, long long n,
                   uint8_t *status, void *vals_out, cudaStream_t s) {
    const hcd::Table<KIND> t(dv);
    switch (dv.bucket_bytes) {
        case 32: return launch_bb<KIND, 32>(t.view(), ops, keys, vals, n, status, vals_out, s);
        case 64: return launch_bb<KIND, 64>(t.view(), ops, keys, vals, n, status, vals_out, s);
        default: return launch_bb<KIND, 128>(t.view(), ops, keys, vals, n, status, vals_out, s);
    }
}

}  // namespace

cudaError_t mixed_ops(const hc_device_view &dv, const uint8_t *ops, const void *keys, const void *vals, long long n,
                      uint8_t *status, void *vals_out, cudaStream_t s) {
    switch (dv.kind) {
        case HC_SET_U32: return launch<KIND_SET_U32>(dv, ops, keys, nullptr, n, status, nullptr, s);
        case HC_SET_U64: return launch<KIND_SET_U64>(dv, ops, keys, nullptr, n, status, nullptr, s);
        case HC_MAP_I64_I32: return launch<KIND_MAP_I64_I32>(dv, ops, keys, vals, n, status, vals_out, s);
        default: return launch<KIND_MAP_U64_U64>(dv, ops, keys, vals, n, status, vals_out, s);
    }
}

}  // namespace hc
