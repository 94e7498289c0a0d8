// hc_select.cu -- selection over the stored entries (Section 3.6): the
// library's predicates, a tile of buckets per block whose matches are appended
// with one atomic (user kernels have hcd::copy_if of the in-kernel header).
// hc_dump is the selection of every entry.
#include <algorithm>
#include <cstdint>

#include "hc.h"
#include "hc_device.cuh"
#include "hc_internal.h"

namespace hc {

namespace {

__device__ __forceinline__ long long coord21(unsigned long long key, int field) {
    const long long c = (long long)((key >> (21 * field)) & 0x1FFFFFull);
    return (c ^ 0x100000ll) - 0x100000ll;   // sign-extend 21 bits
}

template <int KIND>
struct Selector {
    using T = Traits<KIND>;
    SelectPred p;

    __device__ bool operator()(typename T::Key k, typename T::Val v) const {
        bool r = true;
        switch (p.kind) {
            case HC_PRED_KEY_RANGE:
                if constexpr (KIND == KIND_MAP_I64_I32) r = (long long)k >= p.lo && (long long)k <= p.hi;
                else if constexpr (KIND == KIND_SET_U32) r = k >= (uint32_t)p.lo && k <= (uint32_t)p.hi;
                else r = k >= (unsigned long long)p.lo && k <= (unsigned long long)p.hi;
                break;
            case HC_PRED_VALUE_RANGE:
                if constexpr (KIND == KIND_MAP_I64_I32) r = (long long)(int32_t)v >= p.lo && (long long)(int32_t)v <= p.hi;
                else r = (unsigned long long)v >= (unsigned long long)p.lo && (unsigned long long)v <= (unsigned long long)p.hi;
                break;
            case HC_PRED_KEY_MASK:
                r = ((unsigned long long)k & (unsigned long long)p.lo) == (unsigned long long)p.hi;
                break;
            case HC_PRED_BLOCK_BOX: {
                const long long x = coord21(k, 0), y = coord21(k, 1), z = coord21(k, 2);
                r = x >= p.box[0] && x <= p.box[1] && y >= p.box[2] && y <= p.box[3] && z >= p.box[4] && z <= p.box[5];
                break;
            }
            case HC_PRED_SHORT3_BOX: {
                const long long x = (short)((unsigned long long)k & 0xFFFFull);
                const long long y = (short)(((unsigned long long)k >> 16) & 0xFFFFull);
                const long long z = (short)(((unsigned long long)k >> 32) & 0xFFFFull);
                r = x >= p.box[0] && x <= p.box[1] && y >= p.box[2] && y <= p.box[3] && z >= p.box[4] && z <= p.box[5];
                break;
            }
            default: break;   // HC_PRED_ALL
        }
        return r != (p.negate != 0);
    }
};

// One block: a tile of kSelectThreads * NB consecutive buckets.  A thread reads
// the key region of a bucket with vector loads (and its values, where a slot
// is wanted), the tile's matches close ranks in shared memory, one atomic add
// takes their place in the output, and they leave in coalesced stores.  Bound
// by DRAM (70 % of the copy peak): 2^25 slots of 64-byte buckets at load factor
// 0.6, a sixteenth selected, 0.104 ms; every entry, 0.142 ms.  (A grid of blocks
// walking tiles with 8-byte loads and every thread storing its own matches: 0.19
// and 0.28 ms.)
constexpr int kSelectThreads = 256;

template <int KIND, int BB>
__global__ void __launch_bounds__(kSelectThreads)
k_select(View v, Selector<KIND> sel, typename Traits<KIND>::Key *keys_out, typename Traits<KIND>::Val *vals_out,
         unsigned long long cap, unsigned long long *count) {
    using T = Traits<KIND>;
    using Key = typename T::Key;
    using Val = typename T::Val;
    using S = Slots<KIND, BB>;
    constexpr int SPB = S::SPB, NT = kSelectThreads;
    constexpr int NB = SPB >= 8 ? 1 : 8 / SPB;               // buckets per thread: 8 slots or more
    __shared__ Key sk[NT * NB * SPB];
    __shared__ Val sv[T::MAP ? NT * NB * SPB : 1];
    __shared__ unsigned warp_sum[NT / 32];
    __shared__ unsigned long long tile_base;
    const int tid = threadIdx.x;
    const unsigned lane = tid & 31u, warp = tid >> 5;
    const unsigned long long b0 = (unsigned long long)blockIdx.x * (NT * NB) + tid;

    LaneWords<S::KRB> kw[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j)
        if (b0 + j * NT < v.nb) kw[j].load(bucket_at<BB>(v, b0 + j * NT));
    uint32_t hit[NB];
    Val val[T::MAP ? NB : 1][T::MAP ? SPB : 1];
    unsigned mine = 0;
#pragma unroll
    for (int j = 0; j < NB; ++j) {
        hit[j] = 0;
        if (b0 + j * NT >= v.nb) continue;
        uint32_t live = 0;
#pragma unroll
        for (int x = 0; x < SPB; ++x) {
            const Key k = slot_key<KIND, S::KRB>(kw[j], x);
            live |= (uint32_t)(k != T::EMPTY && k != T::TOMB) << x;
        }
        const bool by_value = sel.p.kind == HC_PRED_VALUE_RANGE;
        if (!by_value) {
#pragma unroll
            for (int x = 0; x < SPB; ++x)
                if (live >> x & 1u) hit[j] |= (uint32_t)sel(slot_key<KIND, S::KRB>(kw[j], x), Val()) << x;
        }
        if constexpr (T::MAP) {
            if (by_value ? live != 0 : hit[j] != 0 && vals_out) {
                constexpr int VRB = SPB * (int)sizeof(Val);  // value region: 8 to 64 bytes, aligned to its 16-byte pieces
                const unsigned char *p = bucket_at<BB>(v, b0 + j * NT) + S::KRB;
                if constexpr (VRB >= 16) {
#pragma unroll
                    for (int q = 0; q < VRB / 16; ++q) {
                        const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(p) + q);
                        memcpy(&val[j][q * 16 / (int)sizeof(Val)], &u, 16);
                    }
                } else {
                    const uint2 u = __ldcs(reinterpret_cast<const uint2 *>(p));
                    memcpy(&val[j][0], &u, 8);
                }
                if (by_value) {
#pragma unroll
                    for (int x = 0; x < SPB; ++x)
                        if (live >> x & 1u) hit[j] |= (uint32_t)sel(slot_key<KIND, S::KRB>(kw[j], x), val[j][x]) << x;
                }
            }
        }
        mine += __popc(hit[j]);
    }
    unsigned incl = mine;                                    // this thread's place among the tile's matches
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= (unsigned)d) incl += y;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    unsigned at = incl - mine, total = 0;
#pragma unroll
    for (unsigned w = 0; w < NT / 32; ++w) {
        if (w < warp) at += warp_sum[w];
        total += warp_sum[w];
    }
    if (tid == 0) tile_base = total ? atomicAdd(count, (unsigned long long)total) : 0ull;
#pragma unroll
    for (int j = 0; j < NB; ++j)
#pragma unroll
        for (int x = 0; x < SPB; ++x)
            if (hit[j] >> x & 1u) {
                sk[at] = slot_key<KIND, S::KRB>(kw[j], x);
                if constexpr (T::MAP) sv[at] = val[j][x];
                ++at;
            }
    __syncthreads();
    for (unsigned i = tid; i < total; i += NT) {
        const unsigned long long to = tile_base + i;
        if (to >= cap) break;
        keys_out[to] = sk[i];
        if constexpr (T::MAP) {
            if (vals_out) vals_out[to] = sv[i];
        }
    }
    if (blockIdx.x == 0 && tid == 0) {                       // the two side slots
        for (int side = 0; side < 2; ++side) {
            if (!*((volatile unsigned int *)&v.hdr->side_present[side])) continue;
            const Key k = side == 0 ? T::EMPTY : T::TOMB;
            const Val sval = T::MAP ? (Val) * ((volatile unsigned long long *)&v.hdr->side_val[side]) : Val();
            if (!sel(k, sval)) continue;
            const unsigned long long to = atomicAdd(count, 1ull);
            if (to < cap) {
                keys_out[to] = k;
                if constexpr (T::MAP) {
                    if (vals_out) vals_out[to] = sval;
                }
            }
        }
    }
}

template <int KIND, int BB>
void launch_bb(const View &v, const Selector<KIND> &sel, void *ko, void *vo, unsigned long long cap,
               unsigned long long *count, cudaStream_t s) {
    constexpr int SPB = Slots<KIND, BB>::SPB;
    constexpr unsigned long long tile = kSelectThreads * (SPB >= 8 ? 1 : 8 / SPB);
    k_select<KIND, BB><<<(unsigned)((v.nb + tile - 1) / tile), kSelectThreads, 0, s>>>(
        v, sel, (typename Traits<KIND>::Key *)ko, (typename Traits<KIND>::Val *)vo, cap, count);
}

template <int KIND>
cudaError_t launch(const hc_device_view &dv, const SelectPred &p, void *ko, void *vo, unsigned long long cap,
                   unsigned long long *count, cudaStream_t s) {
    const hcd::Table<KIND> t(dv);
    const Selector<KIND> sel{p};
    switch (dv.bucket_bytes) {
        case 32: launch_bb<KIND, 32>(t.view(), sel, ko, vo, cap, count, s); break;
        case 64: launch_bb<KIND, 64>(t.view(), sel, ko, vo, cap, count, s); break;
        default: launch_bb<KIND, 128>(t.view(), sel, ko, vo, cap, count, s); break;
    }
    return cudaGetLastError();
}

}  // namespace

namespace {

__global__ void __launch_bounds__(256) k_pack_short3(const int16_t *xyz, long long n, long long *keys) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned long long x = (uint16_t)xyz[3 * i], y = (uint16_t)xyz[3 * i + 1], z = (uint16_t)xyz[3 * i + 2];
        keys[i] = (long long)(x | (y << 16) | (z << 32));
    }
}

__global__ void __launch_bounds__(256) k_unpack_short3(const long long *keys, long long n, int16_t *xyz) {
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const unsigned long long k = (unsigned long long)keys[i];
        xyz[3 * i] = (int16_t)(k & 0xFFFFull);
        xyz[3 * i + 1] = (int16_t)((k >> 16) & 0xFFFFull);
        xyz[3 * i + 2] = (int16_t)((k >> 32) & 0xFFFFull);
    }
}

unsigned grid_for_items(long long n, int sms) {
    const long long g = (n + 255) / 256;
    return (unsigned)std::max<long long>(1, std::min<long long>(g, (long long)sms * 8));
}

}  // namespace

cudaError_t pack_short3(const int16_t *xyz, long long n, long long *keys, int sms, cudaStream_t s) {
    k_pack_short3<<<grid_for_items(n, sms), 256, 0, s>>>(xyz, n, keys);
    return cudaGetLastError();
}

cudaError_t unpack_short3(const long long *keys, long long n, int16_t *xyz, int sms, cudaStream_t s) {
    k_unpack_short3<<<grid_for_items(n, sms), 256, 0, s>>>(keys, n, xyz);
    return cudaGetLastError();
}

cudaError_t select_entries(const hc_device_view &dv, const SelectPred &p, void *ko, void *vo, unsigned long long cap,
                           unsigned long long *count, cudaStream_t s) {
    switch (dv.kind) {
        case HC_SET_U32: return launch<KIND_SET_U32>(dv, p, ko, vo, cap, count, s);
        case HC_SET_U64: return launch<KIND_SET_U64>(dv, p, ko, vo, cap, count, s);
        case HC_MAP_I64_I32: return launch<KIND_MAP_I64_I32>(dv, p, ko, vo, cap, count, s);
        default: return launch<KIND_MAP_U64_U64>(dv, p, ko, vo, cap, count, s);
    }
}

}  // namespace hc
