// hc_stream.cuh -- the default range kernels (warp runs), shared by the
// batched form, and the lane-pair lookup.
#pragma once

#include "hc_core.cuh"

// Lookups read buckets through L1 (the read-only path) when 1: a lookup
// never runs together with a modifying call on its table, so the line a
// probe brings into L1 is still valid when a matching key's value is read
// from it right after.  0: L2 only, as the modifying kernels read.
#ifndef HC_FIND_L1
#define HC_FIND_L1 0
#endif

namespace hc {

// The staging of one array of a block chunk (m <= blockDim.x * KPT elements)
// into shared memory, in two steps so that a thread issues the loads of all
// its pieces of every staged array before it stores any: load() reads
// 16-byte pieces tid, tid + nt, ... when src is 16-byte aligned (element by
// element otherwise, and for a tail shorter than 16 bytes) into registers;
// store() writes them to dst (shared, 16-byte aligned).
template <class T, int KPT>
struct Stage {
    static constexpr int E = 16 / (int)sizeof(T);          // elements per 16-byte piece
    static constexpr int J = (KPT + E - 1) / E;            // pieces per thread
    uint4 piece[J];
    T elem[KPT];
    bool vec;

    __device__ __forceinline__ void load(const T *src, int m) {
        const int nt = blockDim.x, tid = threadIdx.x;
        vec = (reinterpret_cast<uintptr_t>(src) & 15) == 0;
        if (vec) {
            const int nv = m / E;
            const uint4 *s4 = reinterpret_cast<const uint4 *>(src);
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int u = tid + j * nt;
                if (u < nv) piece[j] = __ldcs(s4 + u);
            }
            const int i = nv * E + tid;                     // the tail: fewer than E elements
            if (i < m) elem[0] = ld_stream(src + i);
        } else {
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                const int i = tid + j * nt;
                if (i < m) elem[j] = ld_stream(src + i);
            }
        }
    }

    __device__ __forceinline__ void store(T *dst, int m) const {
        const int nt = blockDim.x, tid = threadIdx.x;
        if (vec) {
            const int nv = m / E;
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int u = tid + j * nt;
                if (u < nv) reinterpret_cast<uint4 *>(dst)[u] = piece[j];
            }
            const int i = nv * E + tid;
            if (i < m) dst[i] = elem[0];
        } else {
#pragma unroll
            for (int j = 0; j < KPT; ++j) {
                const int i = tid + j * nt;
                if (i < m) dst[i] = elem[j];
            }
        }
    }
};

template <int LB>
__device__ __forceinline__ void load_find(LaneWords<LB> &lw, const unsigned char *p) {
    if constexpr (HC_FIND_L1 && LB >= 32) {
#pragma unroll
        for (int q = 0; q < LB / 32; ++q)
            asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];"
                         : "=l"(lw.w[4 * q]), "=l"(lw.w[4 * q + 1]), "=l"(lw.w[4 * q + 2]), "=l"(lw.w[4 * q + 3])
                         : "l"(p + 32 * q));
    } else {
        lw.load(p);
    }
}

template <int KIND, int BB>
__device__ __forceinline__ unsigned long long load_find_val(const View &v, unsigned long long b, int s) {
    using T = Traits<KIND>;
    if constexpr (HC_FIND_L1 && T::MAP)
        return (unsigned long long)__ldg(reinterpret_cast<const typename T::Val *>(Slots<KIND, BB>::val(v, b, s)));
    else
        return load_val<KIND, BB>(v, b, s);
}

// ---------------------------------------------------------- warp stacks ---
// The probe loops of the range kernels.  A warp works through a run of keys in
// steps; in a step every lane reads one bucket for one key.  Keys that stay
// undecided go onto the warp's stack in shared memory, and a step takes 32 of
// them as soon as there are that many, the next 32 keys of the run otherwise.
// So all lanes of a step do the same thing on a key of their own until the run
// ends, and the state of a key in flight is one stack entry (about 40-50
// registers a thread against 64-128 with two whole probes in registers).
//
// What bounds it: beyond L2, the device's scattered requests (about 50 G/s on
// a 4 GiB table); inside L2, latency and, with a loop in which every lane
// refills its own probe as soon as it ends, instructions: such a loop runs its
// whole body, hashing included, for the few lanes at each point of it.
// Against that loop (keys staged per block, two probes in flight per thread):
// a pass over 400,000 RGB-D candidates (lookup, insert, lookup, erase; spatial
// hash, 12.5 M slots) 129 -> 72 us; 10^6 inserts + lookups + erases on a
// 50 M-slot map at load factor 0.7, 331 -> 236 us; 2^26 lookups, half of them
// present, on 2^28 slots at 0.8, 4.21 -> 3.56 ms; 30 M set lookups on 10^8
// slots, 0.93 -> 0.84 ms; a 4097-key lookup, call included, 25 -> 17 us.
constexpr int kStack = 64;           // entries: below 32 left by a step, 32 more pushed by it
constexpr int kFewKeys = 20;         // a step's new keys that go to the stack first

__device__ __forceinline__ unsigned lanes_below() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Whether bucket `next`, the one after the bucket a key has just read, is the
// key's first bucket again: only then have all nb buckets been read.  A key is
// at most `reach` buckets from home, so there is nothing to compute before.
__device__ __forceinline__ bool came_round(const View &v, unsigned long long key, unsigned long long next,
                                           unsigned long long reach) {
    return reach + 1 >= v.nb && next == first_bucket(v, key);
}

// The end of a run, when at most 16 keys are left: G = 32 / 16, 8, 4, 2 or 1
// lanes share a key and read its next G buckets at once, so that the last long
// probe sequences of a run take a few steps instead of one per bucket.
// Neighbouring buckets share lines, which a warp's load asks for once.
// (2^20 inserts into 2^22 L2-resident slots, load factor 0.6 -> 0.85: 7.7 G/s
// without, 13.5 G/s with; 2^24 absent lookups on 2^28 slots at 0.75: 17.9 and
// 20.4 G/s.)
struct Drain {
    int group;               // lanes per key
    int entry, sub;          // this lane's stack entry and its bucket after the entry's
    unsigned base;           // first lane of the group
    __device__ __forceinline__ explicit Drain(int top) {
        const int lg = top > 8 ? 1 : top > 4 ? 2 : top > 2 ? 3 : top > 1 ? 4 : 5;
        const int lane = threadIdx.x & 31;
        group = 1 << lg;
        entry = lane >> lg;
        sub = lane & (group - 1);
        base = (unsigned)(lane & ~(group - 1));
    }
    // bits [0, group) = pred of the group's lanes; the whole warp calls it
    __device__ __forceinline__ unsigned ballot(bool pred) const {
        const unsigned m = __ballot_sync(0xffffffffu, pred) >> base;
        return group == 32 ? m : m & ((1u << group) - 1u);
    }
    // Buckets that a key at bucket b has not read yet (up to `group` of them;
    // exact only when it can have come round).
    __device__ __forceinline__ int unread(const View &v, unsigned long long key, unsigned long long b,
                                          unsigned long long reach) const {
        if (reach + group < v.nb) return group;
        const unsigned long long home = first_bucket(v, key);
        const unsigned long long rest = home > b ? home - b : home + v.nb - b;
        return rest < (unsigned long long)group ? (int)rest : group;
    }
    __device__ __forceinline__ static unsigned long long bucket(const View &v, unsigned long long b, int ahead) {
        b += ahead;
        return b >= v.nb ? b - v.nb : b;
    }
};

// What a key finds in a bucket, one bit per slot (free-running batches look for
// claims in progress in place of tombstones).
struct Seen {
    uint32_t hit, empty, tomb;
};

// Reads bucket b of every lane with `act` and compares it with the lane's key;
// the whole warp calls it.  TOGETHER (key regions of 64 or 128 bytes): 2 or 4
// lanes read a bucket together, one key of the group after another, so that a
// bucket is one request however wide it is, and put their findings together;
// otherwise a lane reads its own bucket, a request per 32 bytes.  Beyond the
// reach of the address translation, where requests are what bounds a lookup,
// the first wins; inside it the shuffles cost more than the requests.  set<u64>,
// load factor 0.6, 2^22 present lookups, own -> together, G/s: 64-byte buckets
// 1 GiB 26.4 -> 40.3, 512 MB 31.8 -> 41.7, 64 MB (2^20) 57 -> 47; 128-byte 1 GiB
// 13.7 -> 23.8, 64 MB 34.8 -> 28.9; map<i64,i32>, 128-byte buckets (64 of keys):
// 512 MB 20.8 -> 28.1, 256 MB (2^20, load factor 0.7) 29.9 -> 30.1, its inserts
// 15.2 -> 13.1.
template <int KIND, int BB, bool TOGETHER, bool CLAIMS = false>
__device__ __forceinline__ Seen see_bucket(const View &v, bool act, unsigned long long b,
                                           typename Traits<KIND>::Key key) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Sl = Slots<KIND, BB>;
    constexpr int SPB = Sl::SPB;
    constexpr Key MARK = CLAIMS ? T::CLAIM : T::TOMB;
    if constexpr (!TOGETHER || Sl::KRB <= 32) {
        Seen m{0u, 0u, 0u};
        if (act) {
            LaneWords<Sl::KRB> lw;
            lw.load(bucket_at<BB>(v, b));
#pragma unroll
            for (int x = 0; x < SPB; ++x) {
                const Key ks = slot_key<KIND, Sl::KRB>(lw, x);
                m.hit |= (uint32_t)(ks == key) << x;
                m.empty |= (uint32_t)(ks == T::EMPTY) << x;
                m.tomb |= (uint32_t)(ks == MARK) << x;
            }
        }
        return m;
    } else {
        constexpr int G = Sl::KRB / 32, PS = SPB / G;        // lanes per bucket, slots per lane
        const int lane = threadIdx.x & 31, sub = lane & (G - 1), base = lane & ~(G - 1);
        const unsigned acts = __ballot_sync(0xffffffffu, act);
        LaneWords<32> lw[G];
#pragma unroll
        for (int r = 0; r < G; ++r) {
            const unsigned long long rb = __shfl_sync(0xffffffffu, b, base + r);
            if (acts >> (base + r) & 1u) lw[r].load(bucket_at<BB>(v, rb) + sub * 32);
        }
        Seen mine{0u, 0u, 0u};
#pragma unroll
        for (int r = 0; r < G; ++r) {
            const Key rk = __shfl_sync(0xffffffffu, key, base + r);
            Seen m{0u, 0u, 0u};
            if (acts >> (base + r) & 1u) {
#pragma unroll
                for (int x = 0; x < PS; ++x) {
                    const Key ks = slot_key<KIND, 32>(lw[r], x);
                    m.hit |= (uint32_t)(ks == rk) << x;
                    m.empty |= (uint32_t)(ks == T::EMPTY) << x;
                    m.tomb |= (uint32_t)(ks == MARK) << x;
                }
            }
            if constexpr (SPB <= 8) {
                uint32_t w = (m.hit | m.empty << 8 | m.tomb << 16) << (sub * PS);
#pragma unroll
                for (int d = 1; d < G; d <<= 1) w |= __shfl_xor_sync(0xffffffffu, w, d);
                m = Seen{w & 0xffu, w >> 8 & 0xffu, w >> 16};
            } else {
                m = Seen{m.hit << (sub * PS), m.empty << (sub * PS), m.tomb << (sub * PS)};
#pragma unroll
                for (int d = 1; d < G; d <<= 1) {
                    m.hit |= __shfl_xor_sync(0xffffffffu, m.hit, d);
                    m.empty |= __shfl_xor_sync(0xffffffffu, m.empty, d);
                    m.tomb |= __shfl_xor_sync(0xffffffffu, m.tomb, d);
                }
            }
            if (r == sub) mine = m;
        }
        return mine;
    }
}

// Map lookups in 32-byte buckets (TOGETHER): a lane reads its whole bucket, so
// that a hit's value is no request of its own; val is the value where seen.hit.
// Lookups that hit, keys alone -> whole buckets, G/s: map<u64,u64> 128 MB 47.6 ->
// 51.0, 256 MB 34.5 -> 38.5, 512 MB 29.2 -> 40.9, 2 GiB 21.4 -> 32.1; map<i64,i32>
// 128 MB 52.3 -> 50.3, 256 MB 31.7 -> 38.9, 2 GiB 22.2 -> 33.3; lookups that miss
// are the same from 256 MB on, and 4-9 % slower inside L2.  Wider buckets, read
// by lanes together, gain 15-30 % on hits and lose as much on misses: not done.
constexpr long long kWholeBytes = 256ll << 20;    // tables from which on lookups do so
template <int KIND, int BB>
__device__ __forceinline__ Seen see_whole_bucket(const View &v, bool act, unsigned long long b,
                                                 typename Traits<KIND>::Key key, typename Traits<KIND>::Val &val) {
    using T = Traits<KIND>;
    using Val = typename T::Val;
    using Sl = Slots<KIND, BB>;
    static_assert(T::MAP && BB == 32, "one lane reads a bucket");
    Seen m{0u, 0u, 0u};
    if (act) {
        LaneWords<32> lw;
        lw.load(bucket_at<BB>(v, b));
        unsigned long long u = 0;
#pragma unroll
        for (int x = 0; x < Sl::SPB; ++x) {
            constexpr int V0 = Sl::KRB / (int)sizeof(Val);               // the first value, counted in values
            const auto ks = slot_key<KIND, Sl::KRB>(*reinterpret_cast<const LaneWords<Sl::KRB> *>(&lw), x);
            const unsigned long long word = lw.w[(V0 + x) * (int)sizeof(Val) / 8];
            m.hit |= (uint32_t)(ks == key) << x;
            m.empty |= (uint32_t)(ks == T::EMPTY) << x;
            if (ks == key) u = sizeof(Val) == 8 ? word : word >> ((V0 + x) * 32 % 64);
        }
        val = (Val)u;
    }
    return m;
}

// Stack entries: the key, its next bucket << 16 | its position in the run, and
// for inserts the value and the first free slot the key has passed (slot
// position << 1 | was EMPTY; all ones: none).
template <int KIND, int OP>
struct Stack {
    using Key = typename Traits<KIND>::Key;
    using Val = typename Traits<KIND>::Val;
    static constexpr bool INS = OP == 0, VAL = INS && Traits<KIND>::MAP;
    unsigned long long at[kStack];
    unsigned long long free_at[INS ? kStack : 1];
    Key key[kStack];
    Val val[VAL ? kStack : 1];
    unsigned lost;                       // inserts: swaps that the run's keys have lost to other keys
};

// Looks up the keys src.key(i), i < cnt (asked for 32 at a time, in order, by
// the whole warp); found flags go to sf[i], values to sv[i], those of hits only
// if `want`: a value is a request of its own (2^22 hits asked for without values,
// 64-byte buckets: 1 GiB 173 -> 110 us, 256 MB 89 -> 83; 128-byte 1 GiB 1.33x).
template <int KIND, int BB, bool TOGETHER, class Src>
__device__ __forceinline__ void find_run(const View &v, Src &src, int cnt, Stack<KIND, 1> &st, uint8_t *sf,
                                         typename Traits<KIND>::Val *sv, bool want) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    constexpr bool WITH_VAL = T::MAP && TOGETHER && BB == 32;
    const int lane = threadIdx.x & 31;
    int next = 0, top = 0;
    Key ahead = lane < cnt ? src.key(lane) : Key();
    int late = -1;                           // a found key whose value is still on its way
    Val late_val = Val();
    unsigned long long reach = 0;
    const int few = v.nb >= 32 ? 16 : 0;     // a group's buckets are distinct
    for (;; ++reach) {
        Key key;
        unsigned long long b = 0;
        int idx;
        bool act;
        if (top < 32 && next < cnt) {
            key = ahead;
            idx = next + lane;
            act = idx < cnt;
            next += 32;
            if (next + lane < cnt) ahead = src.key(next + lane);
            const int side = side_index<KIND>(key);
            if (act && side >= 0) {          // key equal to a marker: side slot
                const uint32_t pres = *((volatile unsigned int *)&v.hdr->side_present[side]);
                sf[idx] = pres ? 1 : 0;
                if constexpr (T::MAP)
                    sv[idx] = pres ? (Val) * ((volatile unsigned long long *)&v.hdr->side_val[side]) : (Val)0;
                act = false;
            }
            b = first_bucket(v, (unsigned long long)key);
        } else if (top > few) {
            const int take = top < 32 ? top : 32;
            top -= take;
            act = lane < take;
            const unsigned long long e = st.at[top + (act ? lane : 0)];
            key = st.key[top + (act ? lane : 0)];
            idx = (int)(e & 0xffffu);
            b = e >> 16;
        } else {
            break;
        }
        __syncwarp();                        // entries are read before this step's survivors overwrite them
        Val val = Val();
        Seen seen;
        if constexpr (WITH_VAL) seen = see_whole_bucket<KIND, BB>(v, act, b, key, val);
        else seen = see_bucket<KIND, BB, TOGETHER>(v, act, b, key);
        if constexpr (T::MAP && !WITH_VAL) {
            if (late >= 0) sv[late] = late_val;
            late = -1;
        }
        bool left = false;
        if (act) {
            if (seen.hit) {
                sf[idx] = 1;
                if constexpr (WITH_VAL) sv[idx] = val;
                else if constexpr (T::MAP) {
                    if (want) {
                        late = idx;
                        late_val = (Val)load_val<KIND, BB>(v, b, __ffs(seen.hit) - 1);
                    }
                }
            } else {
                b = next_bucket(v, b);
                left = !seen.empty && !came_round(v, (unsigned long long)key, b, reach);
                if (!left) {
                    sf[idx] = 0;
                    if constexpr (T::MAP) sv[idx] = (Val)0;
                }
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int p = top + __popc(mask & lanes_below());
            st.at[p] = b << 16 | (unsigned)idx;
            st.key[p] = key;
        }
        top += __popc(mask);
        __syncwarp();
    }
    if constexpr (T::MAP && !WITH_VAL) {
        if (late >= 0) sv[late] = late_val;
    }
    while (top > 0) {
        const Drain d(top);
        const bool act = d.entry < top;
        const int p = act ? d.entry : 0;
        const unsigned long long e = st.at[p];
        const Key key = st.key[p];
        const int idx = (int)(e & 0xffffu);
        unsigned long long b = e >> 16;
        __syncwarp();
        const int unread = d.unread(v, (unsigned long long)key, b, reach);
        const unsigned long long mine = Drain::bucket(v, b, d.sub);
        const Seen seen = see_bucket<KIND, BB, TOGETHER>(v, act && d.sub < unread, mine, key);
        const unsigned stop = d.ballot(seen.hit || seen.empty);
        bool left = false;
        if (act && stop) {
            if (d.sub == __ffs(stop) - 1) {
                sf[idx] = seen.hit ? 1 : 0;
                if constexpr (T::MAP) sv[idx] = seen.hit && want ? (Val)load_val<KIND, BB>(v, mine, __ffs(seen.hit) - 1) : (Val)0;
            }
        } else if (act && d.sub == 0) {
            left = unread == d.group;
            b = Drain::bucket(v, b, d.group);
            left = left && !(reach + d.group >= v.nb && b == first_bucket(v, (unsigned long long)key));
            if (!left) {
                sf[idx] = 0;
                if constexpr (T::MAP) sv[idx] = (Val)0;
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int q = __popc(mask & lanes_below());
            st.at[q] = b << 16 | (unsigned)idx;
            st.key[q] = key;
        }
        top = __popc(mask);
        reach += d.group;
        __syncwarp();
    }
    __syncwarp();
}

// Inserts the keys src.key(i) with values src.val(i), i < cnt, except those
// with src.skip(i) (a find saw them: EXISTS); statuses go to ss[i].  A key that
// loses its slot to another key goes on from that slot's bucket: the buckets
// before it had no free slot, and inserts never free one.  Every lost swap means
// that another key took a slot, so they end by themselves; the limit that keeps
// the loop finite whatever the table holds is on lost swaps, kMaxRestarts a key,
// counted for the run as a whole (steps would not do: without an EMPTY slot a key
// reads every bucket before each swap).  Equal keys inside a warp are not folded
// here (folding is a lock-step option).
template <int KIND, int BB, bool TOGETHER, class Src>
__device__ __forceinline__ void insert_run(const View &v, Src &src, int cnt, Stack<KIND, 0> &st, uint8_t *ss,
                                           Counts &cnts) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using Sl = Slots<KIND, BB>;
    using Lay = Layout<KIND, BB, Sl::KRB>;
    constexpr int LB = Sl::KRB;
    constexpr int SPL = Sl::SPB;
    constexpr unsigned long long NONE = ~0ull;
    const int lane = threadIdx.x & 31;
    int next = 0, top = 0;
    Key ahead = Key();
    Val ahead_val = Val();
    bool ahead_skip = false;
    auto fetch = [&](int i) {
        if (i >= cnt) return;
        ahead = src.key(i);
        if constexpr (T::MAP) ahead_val = src.val(i);
        ahead_skip = src.skip(i);
    };
    fetch(lane);
    if (lane == 0) st.lost = 0u;             // (a __syncwarp follows before the first swap)
    unsigned long long reach = 0;
    const int few = v.nb >= 32 ? 16 : 0;     // a group's buckets are distinct
    // Claims the free slot `at` for key; whether the key stays undecided, with
    // its next bucket in b (it lost the slot to another key).
    auto claim_slot = [&](unsigned long long &at, Key key, Val val, int idx, unsigned long long &b) -> bool {
        const bool was_empty = at & 1;
        const unsigned long long fb = (at >> 1) / SPL;
        const int x = (int)((at >> 1) % SPL);
        const Key expect = was_empty ? T::EMPTY : T::TOMB;
        const Key old = cas_key<KIND>(Sl::key(v, fb, x), expect, key);
        if (old == expect) {
            if constexpr (T::MAP) {
                store_val<KIND, BB>(v, fb, x, (unsigned long long)val);
                note_claim_key<KIND>(v.hdr, key, (long long)(at >> 1));
            }
            ss[idx] = (uint8_t)ST_INSERTED;
            ++cnts.ins;
            cnts.new_slot += was_empty ? 1u : 0u;
            return false;
        }
        if (old == key) {                                    // an equal key won the race
            ss[idx] = (uint8_t)ST_EXISTS;
            return false;
        }
        if (atomicAdd(&st.lost, 1u) >= (unsigned)cnt * kMaxRestarts) {
            atomicOr(&v.hdr->err, ERR_PROBE_BOUND);
            ss[idx] = (uint8_t)ST_OVERFLOW;
            cnts.over = 1;
            return false;
        }
        b = fb;
        at = NONE;
        return true;
    };
    for (;; ++reach) {
        Key key;
        Val val = Val();
        unsigned long long b = 0, at = NONE;
        int idx;
        bool act;
        if (top < 32 && next < cnt) {
            key = ahead;
            val = ahead_val;
            idx = next + lane;
            act = idx < cnt;
            if (act && ahead_skip) {
                ss[idx] = (uint8_t)ST_EXISTS;
                act = false;
            }
            next += 32;
            fetch(next + lane);
            const int side = side_index<KIND>(key);
            if (act && side >= 0) {          // key equal to a marker: side slot
                const bool won = atomicCAS(&v.hdr->side_present[side], 0u, 1u) == 0u;
                if (won) {
                    if constexpr (T::MAP) v.hdr->side_val[side] = (unsigned long long)val;
                    ++cnts.ins;
                }
                ss[idx] = won ? (uint8_t)ST_INSERTED : (uint8_t)ST_EXISTS;
                act = false;
            }
            // a step for a few keys costs what one for 32 does: keys among many
            // that are skipped wait on the stack for company (the insert of a
            // 400,000-candidate frame, 88 % of them found before, 18.6 -> 15.9
            // us; an ordered insert + lookup + erase of 2^22 draws 720 -> 699)
            const unsigned mask = __ballot_sync(0xffffffffu, act);
            if (mask == 0u) continue;        // (all skipped: nothing to hash)
            b = first_bucket(v, (unsigned long long)key);
            if (__popc(mask) <= kFewKeys) {
                if (act) {
                    const int p = top + __popc(mask & lanes_below());
                    st.at[p] = b << 16 | (unsigned)idx;
                    st.free_at[p] = NONE;
                    st.key[p] = key;
                    if constexpr (T::MAP) st.val[p] = val;
                }
                top += __popc(mask);
                __syncwarp();
                continue;
            }
        } else if (top > few) {
            const int take = top < 32 ? top : 32;
            top -= take;
            act = lane < take;
            const int p = top + (act ? lane : 0);
            const unsigned long long e = st.at[p];
            key = st.key[p];
            if constexpr (T::MAP) val = st.val[p];
            at = st.free_at[p];
            idx = (int)(e & 0xffffu);
            b = e >> 16;
        } else {
            break;
        }
        __syncwarp();                        // entries are read before this step's survivors overwrite them
        const Seen seen = see_bucket<KIND, BB, TOGETHER>(v, act, b, key);
        const uint32_t le = seen.empty;
        bool left = false, claim = false;
        if (act) {
            if (seen.hit) {                  // already stored
                ss[idx] = (uint8_t)ST_EXISTS;
            } else {
                if (at == NONE) {            // first free slot, rotated scan
                    const uint32_t lf = le | (seen.tomb & claimable<KIND, BB, LB>(v, b, 0));
                    if (lf) {
                        const int rot = v.rotate ? slot_rotation<Lay::SPB>((unsigned long long)key) : 0;
                        const uint32_t hi = lf & (Lay::ALL & ~((1u << rot) - 1u));
                        const int x = __ffs(hi ? hi : lf) - 1;
                        at = (b * SPL + x) << 1 | (le >> x & 1u);
                    }
                }
                claim = le != 0;
                if (!claim) {
                    b = next_bucket(v, b);
                    left = !came_round(v, (unsigned long long)key, b, reach);
                    claim = !left && at != NONE;             // only tombstones were free
                    if (!left && !claim) {                   // no free slot anywhere
                        ss[idx] = (uint8_t)ST_OVERFLOW;
                        cnts.over = 1;
                    }
                }
            }
        }
        if (claim) left = claim_slot(at, key, val, idx, b);
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int p = top + __popc(mask & lanes_below());
            st.at[p] = b << 16 | (unsigned)idx;
            st.free_at[p] = at;
            st.key[p] = key;
            if constexpr (T::MAP) st.val[p] = val;
        }
        top += __popc(mask);
        __syncwarp();
    }
    while (top > 0) {
        const Drain d(top);
        const bool act = d.entry < top;
        const int p = act ? d.entry : 0;
        const unsigned long long e = st.at[p];
        const Key key = st.key[p];
        Val val = Val();
        if constexpr (T::MAP) val = st.val[p];
        unsigned long long at = st.free_at[p];
        const int idx = (int)(e & 0xffffu);
        unsigned long long b = e >> 16;
        __syncwarp();
        const int unread = d.unread(v, (unsigned long long)key, b, reach);
        const unsigned long long mine = Drain::bucket(v, b, d.sub);
        const Seen seen = see_bucket<KIND, BB, TOGETHER>(v, act && d.sub < unread, mine, key);
        const uint32_t le = seen.empty;
        unsigned long long here = NONE;                      // first free slot of this lane's bucket
        {
            const uint32_t lf = le | (seen.tomb & claimable<KIND, BB, LB>(v, mine, 0));
            if (lf) {
                const int rot = v.rotate ? slot_rotation<Lay::SPB>((unsigned long long)key) : 0;
                const uint32_t hi = lf & (Lay::ALL & ~((1u << rot) - 1u));
                const int x = __ffs(hi ? hi : lf) - 1;
                here = (mine * SPL + x) << 1 | (le >> x & 1u);
            }
        }
        const unsigned stop = d.ballot(seen.hit || le);
        const unsigned stored = d.ballot(seen.hit != 0);
        const unsigned some = d.ballot(here != NONE);
        const unsigned first = stop & (0u - stop);           // the bucket that ends the probe, if any
        const unsigned upto = first ? (first - 1u) | first : 0xffffffffu;
        const unsigned from = some & upto;                   // free slots the probe passes
        const unsigned long long passed =
            __shfl_sync(0xffffffffu, here, (int)d.base + (from ? __ffs(from) - 1 : 0));
        bool left = false;
        if (act && d.sub == 0) {
            if (at == NONE && from) at = passed;
            bool claim = first != 0;
            if (first & stored) {                            // already stored
                ss[idx] = (uint8_t)ST_EXISTS;
                claim = false;
            } else if (!first) {
                b = Drain::bucket(v, b, d.group);
                left = unread == d.group &&
                       !(reach + d.group >= v.nb && b == first_bucket(v, (unsigned long long)key));
                claim = !left && at != NONE;                 // only tombstones were free
                if (!left && !claim) {                       // no free slot anywhere
                    ss[idx] = (uint8_t)ST_OVERFLOW;
                    cnts.over = 1;
                }
            }
            if (claim) left = claim_slot(at, key, val, idx, b);
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int q = __popc(mask & lanes_below());
            st.at[q] = b << 16 | (unsigned)idx;
            st.free_at[q] = at;
            st.key[q] = key;
            if constexpr (T::MAP) st.val[q] = val;
        }
        top = __popc(mask);
        reach += d.group;
        __syncwarp();
    }
    __syncwarp();
}

// Erases the keys src.key(i), i < cnt, except those with src.skip(i) (later
// occurrences: NOT_FOUND); statuses go to ss[i].  A failed swap means an equal
// key of the same call erased the slot first: that key reports ERASED, this one
// NOT_FOUND.
template <int KIND, int BB, bool TOGETHER, class Src>
__device__ __forceinline__ void erase_run(const View &v, Src &src, int cnt, Stack<KIND, 2> &st, uint8_t *ss,
                                          Counts &cnts) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Sl = Slots<KIND, BB>;
    const int lane = threadIdx.x & 31;
    int next = 0, top = 0;
    Key ahead = Key();
    bool ahead_skip = false;
    auto fetch = [&](int i) {
        if (i >= cnt) return;
        ahead = src.key(i);
        ahead_skip = src.skip(i);
    };
    fetch(lane);
    unsigned long long reach = 0;
    const int few = v.nb >= 32 ? 16 : 0;     // a group's buckets are distinct
    for (;; ++reach) {
        Key key;
        unsigned long long b = 0;
        int idx;
        bool act;
        if (top < 32 && next < cnt) {
            key = ahead;
            idx = next + lane;
            act = idx < cnt;
            if (act && ahead_skip) {
                ss[idx] = (uint8_t)ST_NOT_FOUND;
                act = false;
            }
            next += 32;
            fetch(next + lane);
            const int side = side_index<KIND>(key);
            if (act && side >= 0) {          // key equal to a marker: side slot
                const bool won = atomicCAS(&v.hdr->side_present[side], 1u, 0u) == 1u;
                cnts.del += won ? 1u : 0u;
                ss[idx] = won ? (uint8_t)ST_ERASED : (uint8_t)ST_NOT_FOUND;
                act = false;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, act);      // as in insert_run
            if (mask == 0u) continue;
            b = first_bucket(v, (unsigned long long)key);
            if (__popc(mask) <= kFewKeys) {
                if (act) {
                    const int p = top + __popc(mask & lanes_below());
                    st.at[p] = b << 16 | (unsigned)idx;
                    st.key[p] = key;
                }
                top += __popc(mask);
                __syncwarp();
                continue;
            }
        } else if (top > few) {
            const int take = top < 32 ? top : 32;
            top -= take;
            act = lane < take;
            const int p = top + (act ? lane : 0);
            const unsigned long long e = st.at[p];
            key = st.key[p];
            idx = (int)(e & 0xffffu);
            b = e >> 16;
        } else {
            break;
        }
        __syncwarp();                        // entries are read before this step's survivors overwrite them
        const Seen seen = see_bucket<KIND, BB, TOGETHER>(v, act, b, key);
        bool left = false;
        if (act) {
            if (seen.hit) {
                const bool won = cas_key<KIND>(Sl::key(v, b, __ffs(seen.hit) - 1), key, T::TOMB) == key;
                if (won) note_claim_key<KIND>(v.hdr, key, -1);
                ss[idx] = won ? (uint8_t)ST_ERASED : (uint8_t)ST_NOT_FOUND;
                cnts.del += won ? 1u : 0u;
            } else {
                b = next_bucket(v, b);
                left = !seen.empty && !came_round(v, (unsigned long long)key, b, reach);
                if (!left) ss[idx] = (uint8_t)ST_NOT_FOUND;
            }
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int p = top + __popc(mask & lanes_below());
            st.at[p] = b << 16 | (unsigned)idx;
            st.key[p] = key;
        }
        top += __popc(mask);
        __syncwarp();
    }
    while (top > 0) {
        const Drain d(top);
        const bool act = d.entry < top;
        const int p = act ? d.entry : 0;
        const unsigned long long e = st.at[p];
        const Key key = st.key[p];
        const int idx = (int)(e & 0xffffu);
        unsigned long long b = e >> 16;
        __syncwarp();
        const int unread = d.unread(v, (unsigned long long)key, b, reach);
        const unsigned long long mine = Drain::bucket(v, b, d.sub);
        const Seen seen = see_bucket<KIND, BB, TOGETHER>(v, act && d.sub < unread, mine, key);
        const unsigned stop = d.ballot(seen.hit || seen.empty);
        bool left = false;
        if (act && stop) {
            if (d.sub == __ffs(stop) - 1) {
                const bool won = seen.hit && cas_key<KIND>(Sl::key(v, mine, __ffs(seen.hit) - 1), key, T::TOMB) == key;
                if (won) note_claim_key<KIND>(v.hdr, key, -1);
                ss[idx] = won ? (uint8_t)ST_ERASED : (uint8_t)ST_NOT_FOUND;
                cnts.del += won ? 1u : 0u;
            }
        } else if (act && d.sub == 0) {
            left = unread == d.group;
            b = Drain::bucket(v, b, d.group);
            left = left && !(reach + d.group >= v.nb && b == first_bucket(v, (unsigned long long)key));
            if (!left) ss[idx] = (uint8_t)ST_NOT_FOUND;
        }
        const unsigned mask = __ballot_sync(0xffffffffu, left);
        if (left) {
            const int q = __popc(mask & lanes_below());
            st.at[q] = b << 16 | (unsigned)idx;
            st.key[q] = key;
        }
        top = __popc(mask);
        reach += d.group;
        __syncwarp();
    }
    __syncwarp();
}

// A run of the caller's arrays, in order.
template <int KIND>
struct ArraySrc {
    using Key = typename Traits<KIND>::Key;
    using Val = typename Traits<KIND>::Val;
    const Key *keys;
    const Val *vals;
    const uint8_t *skips;
    __device__ __forceinline__ Key key(int i) const { return ld_stream(keys + i); }
    __device__ __forceinline__ Val val(int i) const { return ld_stream(vals + i); }
    __device__ __forceinline__ bool skip(int i) const { return skips && ld_stream(skips + i); }
};

// Shared memory of one warp for runs of R keys.
template <int KIND, int OP, int R>
struct alignas(16) WarpRun {
    Stack<KIND, OP> stack;
    typename Traits<KIND>::Val vals[Traits<KIND>::MAP && OP == 1 ? R : 1];
    uint8_t st[R];
};

// The counts of a block's warps, added up in shared memory and moved to the
// header by the warp that finishes last.  Atomics on the one header line go one
// after another (1.5-3 ns each): with one per warp, 2^26 erases in runs of 64
// keys ran at 15.3 G/s instead of 21.4, and 10^6 L2-resident set erases at 21.6
// instead of 32.4.
struct BlockCounts {
    unsigned ins, new_slot, del, over, done;
    // by every thread of the block, before any flush
    __device__ __forceinline__ void init() {
        if (threadIdx.x == 0) ins = new_slot = del = over = done = 0u;
        __syncthreads();
    }
    // by all lanes of a warp; `warps` warps of the block do it
    __device__ __forceinline__ void flush(const View &v, const Counts &c, int warps) {
        __syncwarp();
        const uint32_t w_ins = __reduce_add_sync(0xffffffffu, c.ins);
        const uint32_t w_new = __reduce_add_sync(0xffffffffu, c.new_slot);
        const uint32_t w_del = __reduce_add_sync(0xffffffffu, c.del);
        const uint32_t w_over = __reduce_or_sync(0xffffffffu, c.over);
        if ((threadIdx.x & 31) == 0) {
            if (w_ins) atomicAdd(&ins, w_ins);
            if (w_new) atomicAdd(&new_slot, w_new);
            if (w_del) atomicAdd(&del, w_del);
            if (w_over) atomicOr(&over, 1u);
            __threadfence_block();
            if (atomicAdd(&done, 1u) == (unsigned)warps - 1u) {
                __threadfence_block();
                const long long d = (long long)atomicAdd(&ins, 0u) - (long long)atomicAdd(&del, 0u);
                const unsigned used = atomicAdd(&new_slot, 0u);
                if (d) atomicAdd(&v.hdr->live, (unsigned long long)d);
                if (used) atomicAdd(&v.hdr->used, (unsigned long long)used);
                if (atomicAdd(&over, 0u)) atomicOr(&v.hdr->err, ERR_OVERFLOW);
            }
        }
    }
};

// Blocks of 256 threads per SM that the probe loops are compiled for, by the
// key region that a key in flight holds in registers: 5 (51 registers) for 32
// bytes (at 6, 40 registers and 20-40 bytes spilled, lookups and inserts beyond
// L2 are 2-6 % slower, at 8, 32 registers, 10-20 %), 4 (64) for wider ones, 3
// where 128 bytes are read by lanes together.
constexpr int run_blocks(int krb, bool together) { return krb <= 32 ? 5 : krb == 128 && together ? 3 : 4; }

// The range kernels: warp w of the grid takes keys [w * run, w * run + run),
// run <= R.
template <int KIND, int BB, int OP, int R, bool TOGETHER>
__global__ void __launch_bounds__(256, run_blocks(Slots<KIND, BB>::KRB, TOGETHER))
k_run(View v, const typename Traits<KIND>::Key *keys, const typename Traits<KIND>::Val *vals, const uint8_t *skip,
      long long n, int run, uint8_t *out, typename Traits<KIND>::Val *vals_out) {
    using T = Traits<KIND>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ BlockCounts sum;
    WarpRun<KIND, OP, R> &w = reinterpret_cast<WarpRun<KIND, OP, R> *>(smem)[threadIdx.x >> 5];
    if constexpr (OP != 1) sum.init();
    const long long w0 = (long long)blockIdx.x * (blockDim.x >> 5);
    const long long c0 = (w0 + (threadIdx.x >> 5)) * run;
    if (c0 >= n) return;
    const int cnt = (int)(n - c0 < run ? n - c0 : run);
    debug_range(v, c0, cnt, n);
    ArraySrc<KIND> src{keys + c0, vals + c0, skip ? skip + c0 : nullptr};
    Counts cnts;
    if constexpr (OP == 0) insert_run<KIND, BB, TOGETHER>(v, src, cnt, w.stack, w.st, cnts);
    else if constexpr (OP == 1) find_run<KIND, BB, TOGETHER>(v, src, cnt, w.stack, w.st, w.vals, vals_out != nullptr);
    else erase_run<KIND, BB, TOGETHER>(v, src, cnt, w.stack, w.st, cnts);
    for (int i = threadIdx.x & 31; i < cnt; i += 32) {
        if (out) st_stream(out + c0 + i, w.st[i]);
        if constexpr (OP == 1 && T::MAP) {
            if (vals_out) st_stream(vals_out + c0 + i, w.vals[i]);
        }
    }
    if constexpr (OP != 1) {
        const long long busy = (n + run - 1) / run - w0;     // warps of this block with keys
        sum.flush(v, cnts, (int)(busy < (blockDim.x >> 5) ? busy : (blockDim.x >> 5)));
    }
}

// Streaming map lookup by lane pairs: the two lanes of a pair handle one key.
// The first probe reads the key's first bucket in one instruction, the even
// lane its key region (the first BB/2 bytes), the odd lane its values (the
// rest): one request for one line, and a match there (most present keys) has
// its value without a second, dependent request.  Later probes read the key
// regions of two consecutive buckets at once (even lane: b, odd lane: b + 1),
// so a probe chain advances two buckets per round; a match found there reads
// its value separately.  The pair keeps identical state and control flow and
// exchanges the comparison masks with shuffles.
template <int KIND, int BB, int KPT, int S>
__global__ void __launch_bounds__(256)
k_find_pair(View v, const typename Traits<KIND>::Key *keys, long long n, uint8_t *found,
            typename Traits<KIND>::Val *vals_out) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using Sl = Slots<KIND, BB>;
    constexpr int HB = BB / 2;                    // bytes per lane
    constexpr int SPL = Sl::SPB;
    static_assert(T::MAP && Sl::KRB == HB, "a pair splits a map bucket into keys and values");
    extern __shared__ __align__(16) unsigned char smem[];
    const int pairs = blockDim.x / 2;
    const int chunk = pairs * KPT;
    Key *sk = reinterpret_cast<Key *>(smem);
    Val *sv = reinterpret_cast<Val *>(smem + (size_t)chunk * sizeof(Key));
    uint8_t *sf = smem + (size_t)chunk * (sizeof(Key) + sizeof(Val));

    const long long c0 = (long long)blockIdx.x * chunk;
    const int m = (int)(n - c0 < chunk ? n - c0 : chunk);
    Stage<Key, KPT> gk;
    gk.load(keys + c0, m);
    gk.store(sk, m);
    __syncthreads();

    const unsigned lane = threadIdx.x & 31;
    const bool odd = lane & 1u;
    const unsigned pmask = 3u << (lane & 30u);
    const int pair = threadIdx.x >> 1;
    int idx[S];
    Key key[S];
    unsigned long long b[S];
    uint32_t probes[S];
    bool first[S];
    int next = 0;
    uint32_t active = 0;
    auto take = [&](int s) {
        while (next < KPT) {
            const int i = pair + (next++) * pairs;
            if (i >= m) { next = KPT; break; }
            const Key k = sk[i];
            const int side = side_index<KIND>(k);
            if (side >= 0) {
                if (!odd) {
                    const uint32_t pres = *((volatile unsigned int *)&v.hdr->side_present[side]);
                    sf[i] = pres ? 1 : 0;
                    sv[i] = pres ? (Val) * ((volatile unsigned long long *)&v.hdr->side_val[side]) : (Val)0;
                }
                continue;
            }
            idx[s] = i;
            key[s] = k;
            b[s] = first_bucket(v, (unsigned long long)k);
            probes[s] = 0;
            first[s] = true;
            active |= 1u << s;
            return;
        }
    };
#pragma unroll
    for (int s = 0; s < S; ++s) take(s);
    while (active) {
        LaneWords<HB> lw[S];
        // first probe of a key: keys (even lane) and values (odd lane) of its
        // first bucket; later probes: the key regions of two buckets, b (even
        // lane) and the next one (odd lane)
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if (!(active >> s & 1u)) continue;
            const unsigned long long bb = (odd && !first[s]) ? next_bucket(v, b[s]) : b[s];
            load_find<HB>(lw[s], bucket_at<BB>(v, bb) + ((odd && first[s]) ? HB : 0));
        }
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if (!(active >> s & 1u)) continue;
            uint32_t lm = 0, le = 0;
            if (!odd || !first[s]) {
#pragma unroll
                for (int q = 0; q < SPL; ++q) {
                    const Key ks = slot_key<KIND, HB>(lw[s], q);
                    lm |= (uint32_t)(ks == key[s]) << q;
                    le |= (uint32_t)(ks == T::EMPTY) << q;
                }
            }
            const uint32_t lm0 = __shfl_sync(pmask, lm, lane & 30u), le0 = __shfl_sync(pmask, le, lane & 30u);
            const uint32_t lm1 = __shfl_sync(pmask, lm, lane | 1u), le1 = __shfl_sync(pmask, le, lane | 1u);
            int hit = -1;                      // bucket offset (0 or 1) of a match
            bool absent = false;
            if (first[s]) {
                if (lm0) {
                    const int q = __ffs(lm0) - 1;
                    if (odd) {
                        Val val = 0;           // select the word without indexing registers at run time
#pragma unroll
                        for (int qq = 0; qq < SPL; ++qq) {
                            if constexpr (sizeof(Val) == 8) {
                                if (qq == q) val = (Val)lw[s].w[qq];
                            } else {
                                if (qq == q) val = (Val)(uint32_t)(lw[s].w[qq >> 1] >> ((qq & 1) * 32));
                            }
                        }
                        sv[idx[s]] = val;
                    } else {
                        sf[idx[s]] = 1;
                    }
                    hit = 2;                   // resolved with its value
                } else if (le0 || ++probes[s] >= v.nb) {
                    absent = true;
                } else {
                    b[s] = next_bucket(v, b[s]);
                    first[s] = false;
                }
            } else {
                if (lm0) hit = 0;
                else if (le0 || ++probes[s] >= v.nb) absent = true;
                else if (lm1) hit = 1;
                else if (le1 || ++probes[s] >= v.nb) absent = true;
                else b[s] = next_bucket(v, next_bucket(v, b[s]));
                if (hit >= 0 && !odd) {        // a later bucket: the value needs its own read
                    const unsigned long long hb = hit ? next_bucket(v, b[s]) : b[s];
                    sf[idx[s]] = 1;
                    sv[idx[s]] = (Val)load_find_val<KIND, BB>(v, hb, __ffs(hit ? lm1 : lm0) - 1);
                }
            }
            if (absent && !odd) {
                sf[idx[s]] = 0;
                sv[idx[s]] = (Val)0;
            }
            if (hit >= 0 || absent) {
                active &= ~(1u << s);
                take(s);
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        if (found) st_stream(found + c0 + i, sf[i]);
        if (vals_out) st_stream(vals_out + c0 + i, sv[i]);
    }
}

}  // namespace hc
