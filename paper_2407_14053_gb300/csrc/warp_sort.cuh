// Sort of one tile list by one warp in its own shared memory, shared by the
// compositing kernels (composite.cu) and the ray-order renderer (raycast.cu).
#pragma once

#include <cstdint>

namespace dl {

// largest bucket whose keys the odd-even phases order; a larger one sends the
// list to a bitonic sort
constexpr int kBucketSortLimit = 64;

template <int CAP>
struct WarpSort {
    // at least one bucket a key up to 384 (or 320) keys: the passes that
    // order keys inside buckets grow with the most crowded bucket, and depths
    // cluster; for CAP = 512 the buckets fill the space the stream phase
    // needs anyway, for CAP = 1024 the sort phase sets the size (six blocks
    // per SM)
    static constexpr int kBuckets = CAP <= 512 ? 384 : 320;
    unsigned long long sk[CAP];
    uint32_t bstart[kBuckets];  // bucket sizes, starts, then (after the scatter) ends
};
// Warp-level version of block_sort (len <= CAP).  The first KPL * 32 keys
// (256 in the 512-key class, whose registers are held to 64 for eight blocks
// per SM; 512 in the 1024-key class) are held in registers; the rest of a
// longer list is re-read from global memory (L2) per pass.
template <int CAP>
__device__ void warp_sort(const unsigned long long* __restrict__ keys, uint32_t start, int len,
                          WarpSort<CAP>& W) {
    const int lane = threadIdx.x & 31;
    constexpr int kWarpBuckets = WarpSort<CAP>::kBuckets;
    constexpr int KPL = CAP <= 512 ? 8 : 16;
    unsigned long long kr[KPL];
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    const bool in_regs = len <= KPL * 32;
#pragma unroll
    for (int j = 0; j < KPL; ++j) {
        const int i = j * 32 + lane;
        kr[j] = i < len ? keys[start + i] : ~0ull;
        if (i < len) {
            lo = min(lo, uint32_t(kr[j] >> 32));
            hi = max(hi, uint32_t(kr[j] >> 32));
        }
    }
    for (int i = KPL * 32 + lane; i < len; i += 32) {
        lo = min(lo, uint32_t(keys[start + i] >> 32));
        hi = max(hi, uint32_t(keys[start + i] >> 32));
    }
    if (len <= 1) {
        if (len == 1 && lane == 0) W.sk[0] = kr[0];
        __syncwarp();
        return;
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    int NB = 1;
    while (NB < len) NB <<= 1;
    if (NB > kWarpBuckets) NB = kWarpBuckets;
    // Depths cluster (a dense core in front of a sparse background), so
    // buckets spread evenly over [lo, hi] crowd where the keys are.  With 64
    // buckets or more the mapping is equi-depth at a coarse grain: a first
    // count over kCoarse even bins of [lo, hi] gives bin c a share of the
    // buckets in proportion to its keys (at least one when it has any), and
    // a key takes the bucket of its position within its bin.  The bucket is
    // non-decreasing in the depth word (t is; so is the bin; within a bin so
    // are t - c, exact, and its scaled integer part; the bins' bucket ranges
    // are disjoint and in order), which is all the phases below need.  The
    // bins' table takes the last kCoarse bucket words.
    constexpr int kCoarse = 32;
    const bool equi = NB >= 2 * kCoarse;
    if (equi && NB > kWarpBuckets - kCoarse) NB = kWarpBuckets - kCoarse;
    uint32_t* const table = W.bstart + (kWarpBuckets - kCoarse);
    for (int b = lane; b < NB; b += 32) W.bstart[b] = 0u;
    const float scale = float(equi ? kCoarse : NB) / (float(hi - lo) + 1.0f);
    if (equi) {
        auto bin = [&](unsigned long long k) {
            return min(kCoarse - 1, int(float(uint32_t(k >> 32) - lo) * scale));
        };
        table[lane] = 0u;
        __syncwarp();
#pragma unroll
        for (int j = 0; j < KPL; ++j)
            if (j * 32 + lane < len) atomicAdd(&table[bin(kr[j])], 1u);
        if (!in_regs)
            for (int i = KPL * 32 + lane; i < len; i += 32) atomicAdd(&table[bin(keys[start + i])], 1u);
        __syncwarp();
        const uint32_t nc = table[lane];  // keys in bin `lane`
        const uint32_t nb = nc * uint32_t(NB - kCoarse) / uint32_t(len) + (nc ? 1u : 0u);
        uint32_t inc = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        __syncwarp();
        table[lane] = (inc - nb) | (nb << 16);  // first bucket | buckets << 16
    }
    __syncwarp();
    auto bucket = [&](unsigned long long k) {
        const float t = float(uint32_t(k >> 32) - lo) * scale;
        if (!equi) return min(NB - 1, int(t));
        const int c = min(kCoarse - 1, int(t));
        const uint32_t q = table[c];
        const int nb = int(q >> 16);
        return int(q & 0xFFFFu) + min(nb - 1, int((t - float(c)) * float(nb)));
    };
    // the first KPL * 32 keys are in registers, the rest are re-read
#pragma unroll
    for (int j = 0; j < KPL; ++j)
        if (j * 32 + lane < len) atomicAdd(&W.bstart[bucket(kr[j])], 1u);
    if (!in_regs)
        for (int i = KPL * 32 + lane; i < len; i += 32)
            atomicAdd(&W.bstart[bucket(keys[start + i])], 1u);
    __syncwarp();
    uint32_t most = 0u;  // the most crowded bucket's size
    {  // exclusive scan of bstart[0..NB)
        const int per = (NB + 31) / 32, b0 = lane * per;
        uint32_t sum = 0;
        for (int b = b0; b < b0 + per && b < NB; ++b) {
            const uint32_t c = W.bstart[b];
            sum += c;
            most = max(most, c);
        }
        most = __reduce_max_sync(0xffffffffu, most);
        uint32_t inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        uint32_t run = inc - sum;
        __syncwarp();
        for (int b = b0; b < b0 + per && b < NB; ++b) {
            const uint32_t c = W.bstart[b];
            W.bstart[b] = run;
            run += c;
        }
    }
    __syncwarp();
    // scatter: bstart[b] serves as bucket b's cursor, so afterwards it holds
    // the bucket's end (= the start of bucket b + 1)
#pragma unroll
    for (int j = 0; j < KPL; ++j)
        if (j * 32 + lane < len) W.sk[atomicAdd(&W.bstart[bucket(kr[j])], 1u)] = kr[j];
    if (!in_regs)
        for (int i = KPL * 32 + lane; i < len; i += 32) {
            const unsigned long long k = keys[start + i];
            W.sk[atomicAdd(&W.bstart[bucket(k)], 1u)] = k;
        }
    __syncwarp();
    if (most > uint32_t(kBucketSortLimit)) {
        int P = 1;
        while (P < len) P <<= 1;
        for (int i = len + lane; i < P; i += 32) W.sk[i] = ~0ull;
        __syncwarp();
        for (int k = 2; k <= P; k <<= 1)
            for (int jj = k >> 1; jj > 0; jj >>= 1) {
                for (int i = lane; i < (P >> 1); i += 32) {
                    const int a = ((i & ~(jj - 1)) << 1) | (i & (jj - 1));
                    const int c = a + jj;
                    const bool up = (a & k) == 0;
                    const unsigned long long x = W.sk[a], y = W.sk[c];
                    if ((x > y) == up) {
                        W.sk[a] = y;
                        W.sk[c] = x;
                    }
                }
                __syncwarp();
            }
    } else {
        // The buckets are in order, so only keys within a bucket are out of
        // place, and no compared pair that straddles two buckets is ever
        // swapped: odd-even transposition phases over the whole list (even
        // pairs (2i, 2i + 1) as one 16-byte access, odd pairs (2i + 1,
        // 2i + 2)) sort every bucket at once, and s phases sort s keys
        // whichever phase comes first, so the most crowded bucket's size is
        // the phase count (none when every bucket holds at most one key).
        // Every lane has work in every phase, unlike a lane-per-bucket
        // insertion sort, where the warp waits for the most crowded of each
        // 32 buckets.
        ulonglong2* const pairs = reinterpret_cast<ulonglong2*>(W.sk);
        for (uint32_t ph = 0; ph < most; ++ph) {
            if ((ph & 1u) == 0u) {
                for (int i = lane; 2 * i + 1 < len; i += 32) {
                    const ulonglong2 q = pairs[i];
                    if (q.x > q.y) pairs[i] = make_ulonglong2(q.y, q.x);
                }
            } else {
                for (int i = 2 * lane + 1; i + 1 < len; i += 64) {
                    const unsigned long long x = W.sk[i], y = W.sk[i + 1];
                    if (x > y) {
                        W.sk[i] = y;
                        W.sk[i + 1] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
}

}  // namespace dl
