// Front-to-back alpha compositing (Sec. 3.2 Eq. (5), Sec. 3.3 Eq. (10)) and
// the standard paradigm's interweave (Alg. 1).
//
// Both compositing kernels stream one (view, tile) list of depth-sorted
// Gaussian records through shared memory in batches.  Each warp first tests
// 32 records at a time against the bounding box of its own rays (one ballot)
// and then composites only the records whose alpha >= 1/255 box touches it,
// in list order, so the per-ray sequence of composited Gaussians is exactly
// the depth-sorted one.  A block stops once every ray's transmittance would
// fall below 1e-4 (block-wide vote).
//  - composite_rays_kernel (DirectL): one block per work item, i.e. up to
//    kRayThreads required rays of one (view, tile), ordered along a Morton
//    curve so that a warp's rays are close together; each ray writes its
//    colour, and reorder_kernel gathers the encoded image by the ray table
//    (Sec. 4 step (3): the channel reorder by precomputed indices).
//  - composite_full_kernel (standard paradigm): one block per (view, tile),
//    one thread per pixel, every pixel of every view into M_m.
#include <algorithm>
#include <climits>

#include "dl_internal.cuh"
#include "warp_sort.cuh"

namespace dl {
namespace {

constexpr int kRayThreads = 128;
constexpr float kLog2MinAlpha = -7.99435343685886f;  // log2(1/255)

struct Acc {
    float T, c0, c1, c2;
    uint32_t blended;
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Asynchronous 16-byte global -> shared copies (Ampere-and-later cp.async),
// used to fetch the next batch of records while the current one is blended.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// log2 alpha = A dx^2 + B dx dy + C dy^2 + log2 o at pixel offset (dx, dy)
// from the record's mean.  Every caller evaluates exactly this expression, so
// a pre-test and the blend below always agree bit for bit.
__device__ __forceinline__ float log2_alpha(float px, float py, float u, float v, float A, float B,
                                            float C, float L) {
    const float dx = px - u, dy = py - v;
    return fmaf(dx, fmaf(A, dx, B * dy), fmaf(C * dy, dy, L));
}

// One record against one ray.  Returns false once the ray is finished.
// alpha = min(0.99, 2^log2_alpha); skip alpha < 1/255 (CHECK_L2: tested
// first on log2 alpha, which spares the ex2 for records that miss the ray,
// then on alpha itself); stop before T (1 - alpha) = T - alpha T would drop
// below 1e-4.  After the log2 test the steps are selects, not branches: a
// skipped record adds 0 alpha T = 0 to the colour and leaves T (>= 1e-4) as
// it is.  COUNT keeps the composited-pair statistic.  The colour is
// (q1.z, q1.w, b): kernels that load a batch thread by thread decode the
// packed colour once per record when they store it in shared memory (the
// standard paradigm blends tens of times per record); blend_rec below takes
// a record as stored.
template <bool CHECK_L2 = true, bool COUNT = true>
__device__ __forceinline__ bool blend(Acc& a, float px, float py, const float4& q0,
                                      const float4& q1, float b) {
    const float l2 = log2_alpha(px, py, q0.x, q0.y, q0.z, q0.w, q1.x, q1.y);
    if (CHECK_L2 && l2 < kLog2MinAlpha) return true;
    float alpha = fminf(0.99f, ex2_approx(l2));
    alpha = alpha < (1.0f / 255.0f) ? 0.f : alpha;
    const float w0 = alpha * a.T;
    const float Tn = a.T - w0;
    const bool go = Tn >= 1e-4f;
    const float w = go ? w0 : 0.f;
    a.c0 = fmaf(w, q1.z, a.c0);
    a.c1 = fmaf(w, q1.w, a.c1);
    a.c2 = fmaf(w, b, a.c2);
    a.T = go ? Tn : a.T;
    if (COUNT && go && alpha > 0.f) ++a.blended;
    return go;
}

// blend() on a record as the projection stored it (packed colour).
template <bool CHECK_L2 = true, bool COUNT = true>
__device__ __forceinline__ bool blend_rec(Acc& a, float px, float py, const float4& q0,
                                          const float4& q1) {
    float r, g, b;
    unpack_rgb(q1.z, q1.w, r, g, b);
    return blend<CHECK_L2, COUNT>(a, px, py, q0, make_float4(q1.x, q1.y, r, g), b);
}

// blend() of two candidates in list order, their alphas formed together
// (`two` false: the second is none).  The arithmetic and its order are
// blend()'s on each candidate in turn; false once the ray is finished.
template <bool COUNT>
__device__ __forceinline__ bool blend2(Acc& a, float px, float py, const float4& p0,
                                       const float4& p1, float pb, const float4& q0,
                                       const float4& q1, float qb, bool two) {
    const float la = log2_alpha(px, py, p0.x, p0.y, p0.z, p0.w, p1.x, p1.y);
    const float lb = log2_alpha(px, py, q0.x, q0.y, q0.z, q0.w, q1.x, q1.y);
    float alpha_a = fminf(0.99f, ex2_approx(la));
    float alpha_b = fminf(0.99f, ex2_approx(lb));
    alpha_a = alpha_a < (1.0f / 255.0f) ? 0.f : alpha_a;
    alpha_b = (alpha_b < (1.0f / 255.0f) || !two) ? 0.f : alpha_b;
    const float wa0 = alpha_a * a.T;
    const float Ta = a.T - wa0;
    const bool goa = Ta >= 1e-4f;
    const float wa = goa ? wa0 : 0.f;
    a.c0 = fmaf(wa, p1.z, a.c0);
    a.c1 = fmaf(wa, p1.w, a.c1);
    a.c2 = fmaf(wa, pb, a.c2);
    a.T = goa ? Ta : a.T;
    const float wb0 = alpha_b * a.T;
    const float Tb = a.T - wb0;
    const bool gob = goa && Tb >= 1e-4f;
    const float wb = gob ? wb0 : 0.f;
    a.c0 = fmaf(wb, q1.z, a.c0);
    a.c1 = fmaf(wb, q1.w, a.c1);
    a.c2 = fmaf(wb, qb, a.c2);
    a.T = gob ? Tb : a.T;
    if (COUNT) a.blended += (goa && alpha_a > 0.f) + (gob && alpha_b > 0.f);
    return gob;
}

// A record and its pixel box in the shared-memory layout of the batch
// loaders: s0 = (u, v, A, B), s1 = (C, L, r, g), s2 = (b, -, rect_c, rect_r).
__device__ __forceinline__ void store_decoded(const float4& q0, const float4& q1, uint2 rect,
                                              float4& s0, float4& s1, float4& s2) {
    float r, g, b;
    unpack_rgb(q1.z, q1.w, r, g, b);
    s0 = q0;
    s1 = make_float4(q1.x, q1.y, r, g);
    s2 = make_float4(b, 0.f, __uint_as_float(rect.x), __uint_as_float(rect.y));
}

// Adds the block's evaluated and composited pair counts to pairs[0..1].
__device__ __forceinline__ void count_pairs(unsigned long long* pairs, uint32_t evals,
                                            uint32_t blended) {
    unsigned long long e = evals, b = blended;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_down_sync(0xffffffffu, e, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(pairs, e);
        atomicAdd(pairs + 1, b);
    }
}

// Transposed evaluation of up to 32 records (indices wbuf[0..n)) for the
// warp's rays: each lane holds one record, tests it against every ray that is
// still compositing (ray position by shuffle, one ballot per ray), and keeps
// the mask of records that may reach alpha >= 1/255 for its own ray.  Then
// every lane blends its own candidates in list order.  Finished rays drop out
// of the ray loop, so they cost nothing.
__device__ __forceinline__ void warp_group(Acc& a, bool& done, uint32_t& evals, float px, float py,
                                           const int* wbuf, int n, const float4* s0,
                                           const float4* s1, const float4* s2) {
    const int lane = threadIdx.x & 31;
    const int j = lane < n ? wbuf[lane] : -1;
    float u = 0.f, v = 0.f, A = 0.f, B = 0.f, C = 0.f, L = -1e30f;
    if (j >= 0) {
        const float4 q0 = s0[j];
        const float2 q1 = *reinterpret_cast<const float2*>(s1 + j);
        u = q0.x; v = q0.y; A = q0.z; B = q0.w; C = q1.x; L = q1.y;
    }
    unsigned act = __ballot_sync(0xffffffffu, !done);
    unsigned mine = 0;
    while (act) {
        const int r = __ffs(act) - 1;
        act &= act - 1;
        const float rx = __shfl_sync(0xffffffffu, px, r);
        const float ry = __shfl_sync(0xffffffffu, py, r);
        const bool pass = log2_alpha(rx, ry, u, v, A, B, C, L) >= kLog2MinAlpha;
        const unsigned m = __ballot_sync(0xffffffffu, pass);
        if (lane == r) mine = m;
    }
    if (!done) evals += uint32_t(n);
    while (mine && !done) {
        const int sidx = __ffs(mine) - 1;
        mine &= mine - 1;
        const int jj = wbuf[sidx];
        if (!blend(a, px, py, s0[jj], s1[jj], s2[jj].x)) done = true;
    }
}

// Composites a shared-memory batch of nb records for this lane's ray.  Records
// whose pixel box misses the warp's box [bx0,bx1] x [by0,by1] are dropped; the
// rest are compacted, in list order, into the warp's buffer (64 ints) and
// evaluated 32 at a time.
__device__ __forceinline__ void warp_batch(Acc& a, bool& done, uint32_t& evals, float px, float py,
                                           int bx0, int bx1, int by0, int by1, const float4* s0,
                                           const float4* s1, const float4* s2, int nb, int* wbuf) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1;
    int cnt = 0;
    for (int j0 = 0; j0 < nb; j0 += 32) {
        if (__all_sync(0xffffffffu, done)) return;
        bool hit = false;
        if (j0 + lane < nb) {
            const float4 q2 = s2[j0 + lane];
            const uint32_t rc = __float_as_uint(q2.z), rr = __float_as_uint(q2.w);
            hit = int(rc & 0xFFFFu) <= bx1 && int(rc >> 16) >= bx0 && int(rr & 0xFFFFu) <= by1 &&
                  int(rr >> 16) >= by0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (hit) wbuf[cnt + __popc(m & lt)] = j0 + lane;
        cnt += __popc(m);
        __syncwarp();
        if (cnt >= 32) {
            warp_group(a, done, evals, px, py, wbuf, 32, s0, s1, s2);
            __syncwarp();
            const int rest = cnt - 32;
            const int t = lane < rest ? wbuf[32 + lane] : 0;
            __syncwarp();
            if (lane < rest) wbuf[lane] = t;
            __syncwarp();
            cnt = rest;
        }
    }
    if (cnt > 0 && !__all_sync(0xffffffffu, done)) {
        warp_group(a, done, evals, px, py, wbuf, cnt, s0, s1, s2);
    }
    __syncwarp();
}

// Direct evaluation: every lane walks the culled records in list order and
// evaluates each one for its own ray (record fields by shared-memory broadcast).
__device__ __forceinline__ void warp_batch_direct(Acc& a, bool& done, uint32_t& evals, float px,
                                                  float py, int bx0, int bx1, int by0, int by1,
                                                  const float4* s0, const float4* s1,
                                                  const float4* s2, int nb) {
    const int lane = threadIdx.x & 31;
    for (int j0 = 0; j0 < nb; j0 += 32) {
        if (__all_sync(0xffffffffu, done)) return;
        bool hit = false;
        if (j0 + lane < nb) {
            const float4 q2 = s2[j0 + lane];
            const uint32_t rc = __float_as_uint(q2.z), rr = __float_as_uint(q2.w);
            hit = int(rc & 0xFFFFu) <= bx1 && int(rc >> 16) >= bx0 && int(rr & 0xFFFFu) <= by1 &&
                  int(rr >> 16) >= by0;
        }
        unsigned m = __ballot_sync(0xffffffffu, hit);
        while (m) {
            const int j = j0 + __ffs(m) - 1;
            m &= m - 1;
            if (!done) {
                ++evals;
                if (!blend(a, px, py, s0[j], s1[j], s2[j].x)) done = true;
            }
        }
    }
}

template <bool TRANSPOSED>
__device__ __forceinline__ void eval_batch(Acc& a, bool& done, uint32_t& evals, float px, float py,
                                           int bx0, int bx1, int by0, int by1, const float4* s0,
                                           const float4* s1, const float4* s2, int nb, int* wbuf) {
    if (TRANSPOSED)
        warp_batch(a, done, evals, px, py, bx0, bx1, by0, by1, s0, s1, s2, nb, wbuf);
    else
        warp_batch_direct(a, done, evals, px, py, bx0, bx1, by0, by1, s0, s1, s2, nb);
}

__device__ __forceinline__ void warp_box(bool active, int col, int row, int& bx0, int& bx1, int& by0,
                                         int& by1) {
    bx0 = __reduce_min_sync(0xffffffffu, active ? col : INT_MAX);
    bx1 = __reduce_max_sync(0xffffffffu, active ? col : INT_MIN);
    by0 = __reduce_min_sync(0xffffffffu, active ? row : INT_MAX);
    by1 = __reduce_max_sync(0xffffffffu, active ? row : INT_MIN);
}

__global__ void __launch_bounds__(kRayThreads)
composite_rays_kernel(CompositeParams p, const int4* __restrict__ work,
                      const int2* __restrict__ grouped, const uint2* __restrict__ ranges,
                      const uint32_t* __restrict__ vals, const float4* __restrict__ rec,
                      float* __restrict__ raycol, unsigned long long* __restrict__ pairs) {
    __shared__ float4 s0[kRayThreads];
    __shared__ float4 s1[kRayThreads];
    __shared__ float4 s2[kRayThreads];
    const int4 wi = work[blockIdx.x];
    const int v = wi.x / p.ntiles;
    const int rid = wi.y + int(threadIdx.x);
    const bool active = rid < wi.z;
    const int2 ray = active ? grouped[rid] : make_int2(0, -1);
    const int col = int(uint32_t(ray.x) & 0xFFFFu), row = int(uint32_t(ray.x) >> 16);
    const float px = float(col) - p.half_w;
    const float py = float(row) - p.half_h;
    int bx0, bx1, by0, by1;
    warp_box(active, col, row, bx0, bx1, by0, by1);
    const uint2 rg = ranges[wi.x];
    const int64_t vbase = int64_t(v) * p.n;
    Acc a{1.f, 0.f, 0.f, 0.f, 0u};
    uint32_t evals = 0;
    bool done = !active;
    for (uint32_t b = rg.x; b < rg.y; b += kRayThreads) {
        const uint32_t i = b + threadIdx.x;
        if (i < rg.y) {
            const int64_t e = vbase + vals[i];
            const float4 q0 = rec[kRecordFloat4 * e], q1 = rec[kRecordFloat4 * e + 1];
            const uint4 m = p.meta[e];
            store_decoded(q0, q1, make_uint2(m.x, m.y), s0[threadIdx.x], s1[threadIdx.x],
                          s2[threadIdx.x]);
        }
        __syncthreads();
        const int nb = int(rg.y - b < kRayThreads ? rg.y - b : kRayThreads);
        warp_batch_direct(a, done, evals, px, py, bx0, bx1, by0, by1, s0, s1, s2, nb);
        if (__syncthreads_count(done) == int(blockDim.x)) break;
    }
    if (pairs) count_pairs(pairs, evals, a.blended);
    if (active) {
        float* o = raycol + 3 * int64_t(rid);  // grouped order
        o[0] = a.c0;
        o[1] = a.c1;
        o[2] = a.c2;
    }
}

// A thread per pixel, so blocks of up to 1024 threads (the largest tile): 40
// registers a thread, and 48 bytes of shared memory a thread are exactly the
// 48 KB that a block has without asking for more.
__global__ void composite_full_kernel(CompositeParams p, const uint2* __restrict__ ranges,
                                      const uint32_t* __restrict__ vals,
                                      const float4* __restrict__ rec, float* __restrict__ Mm,
                                      unsigned long long* __restrict__ pairs) {
    extern __shared__ float4 sm[];
    const int nthr = blockDim.x;
    float4* s0 = sm;
    float4* s1 = sm + nthr;
    float4* s2 = sm + 2 * nthr;
    const int group = blockIdx.x;
    const int v = group / p.ntiles;
    const int tile = group - v * p.ntiles;
    const int tx = tile % p.ntx, ty = tile / p.ntx;
    const int col = tx * p.tile_w + int(threadIdx.x) % p.tile_w;
    const int row = ty * p.tile_h + int(threadIdx.x) / p.tile_w;
    const bool inside = col < p.width && row < p.height;
    const float px = float(col) - p.half_w, py = float(row) - p.half_h;
    int bx0, bx1, by0, by1;
    warp_box(inside, col, row, bx0, bx1, by0, by1);
    const uint2 rg = ranges[group];
    const int64_t vbase = int64_t(v) * p.n;
    Acc a{1.f, 0.f, 0.f, 0.f, 0u};
    uint32_t evals = 0;
    bool done = !inside;
    for (uint32_t b = rg.x; b < rg.y; b += nthr) {
        const uint32_t i = b + threadIdx.x;
        if (i < rg.y) {
            const int64_t e = vbase + vals[i];
            const float4 q0 = rec[kRecordFloat4 * e], q1 = rec[kRecordFloat4 * e + 1];
            const uint4 m = p.meta[e];
            store_decoded(q0, q1, make_uint2(m.x, m.y), s0[threadIdx.x], s1[threadIdx.x],
                          s2[threadIdx.x]);
        }
        __syncthreads();
        const int nb = int(rg.y - b < uint32_t(nthr) ? rg.y - b : uint32_t(nthr));
        warp_batch_direct(a, done, evals, px, py, bx0, bx1, by0, by1, s0, s1, s2, nb);
        if (__syncthreads_count(done) == nthr) break;
    }
    if (pairs) count_pairs(pairs, evals, a.blended);
    if (inside) {
        float* o = Mm + ((int64_t(v) * p.height + row) * p.width + col) * 3;
        o[0] = a.c0;
        o[1] = a.c1;
        o[2] = a.c2;
    }
}

// ---------------------------------------------------------- binned path ---
// Ascending bitonic sort of n unique keys in shared memory, for any n: every
// compared pair puts the larger key at the higher index, so positions past
// the end act as larger than any key and are left out.
__device__ void bitonic_sort(unsigned long long* s, int n) {
    int P = 1;
    while (P < n) P <<= 1;
    auto order = [&](int lo, int hi) {
        if (hi >= n) return;
        const unsigned long long a = s[lo], b = s[hi];
        if (a > b) {
            s[lo] = b;
            s[hi] = a;
        }
    };
    for (int k = 2; k <= P; k <<= 1) {
        for (int i = threadIdx.x; i < (P >> 1); i += blockDim.x) {  // mirrored pairs
            const int off = i & ((k >> 1) - 1), base = (i - off) << 1;
            order(base + off, base + k - 1 - off);
        }
        __syncthreads();
        for (int j = k >> 2; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < (P >> 1); i += blockDim.x) {
                const int lo = ((i & ~(j - 1)) << 1) | (i & (j - 1));
                order(lo, lo + j);
            }
            __syncthreads();
        }
    }
}

// Exclusive scan, in place, of n <= blockDim.x * 64 counters in shared memory.
__device__ void block_scan_counts(uint32_t* c, int n) {
    __shared__ uint32_t s_w[32];
    const int nthr = blockDim.x, tid = threadIdx.x;
    const int per = (n + nthr - 1) / nthr;
    const int b0 = tid * per;
    uint32_t sum = 0;
    for (int i = b0; i < b0 + per && i < n; ++i) sum += c[i];
    const int lane = tid & 31, wid = tid >> 5, nw = (nthr + 31) >> 5;
    uint32_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) s_w[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        const uint32_t x = lane < nw ? s_w[lane] : 0;
        uint32_t xi = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, xi, o);
            if (lane >= o) xi += t;
        }
        if (lane < nw) s_w[lane] = xi - x;
    }
    __syncthreads();
    uint32_t run = s_w[wid] + inc - sum;
    for (int i = b0; i < b0 + per && i < n; ++i) {
        const uint32_t v = c[i];
        c[i] = run;
        run += v;
    }
    __syncthreads();
}

// Sorts the group's keys (depth << 32 | Gaussian, all distinct) into sk: a
// counting sort into depth buckets (monotone in the depth), then as many
// odd-even transposition phases over the whole list as the most crowded
// bucket holds keys (as in warp_sort below).  From 256 buckets on they are
// equi-depth at a coarse grain: a first count over kBlockBins even bins gives
// each bin a share of the buckets in proportion to its keys, since depths
// cluster and crowded buckets set the number of phases.  If a bucket still
// holds more than kBucketSortLimit keys (many equal depths), the whole list is
// bitonic-sorted instead.  The keys are re-read (from L2) by every pass.  sk
// holds cap keys and cnt cap / 2 counters, cap >= len being the class capacity
// (a multiple of 512, at least 1024): ten bytes a key.  What bounds the block
// classes is resident warps, which shared memory sets: 10 bytes a key of a
// capacity in steps of 512, reused by the stream phase, against 12 of the next
// power of two beside it, took 11,189 lists of up to 1862 keys (7.9-inch
// panel) from 1.23 to 0.65 ms and 21,885 of up to 3072 (800 x 450 views) from
// 3.4 to 2.5 ms.
constexpr int kBlockBins = 128;
__device__ void block_sort(const unsigned long long* __restrict__ keys, uint32_t start, int len,
                           int cap, unsigned long long* sk, uint32_t* cnt) {
    __shared__ uint32_t s_lo, s_hi, s_most;
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (tid == 0) {
        s_lo = 0xFFFFFFFFu;
        s_hi = 0u;
        s_most = 0u;
    }
    __syncthreads();
    if (len <= 1) {
        if (len == 1 && tid == 0) sk[0] = keys[start];
        __syncthreads();
        return;
    }
    uint32_t lo = 0xFFFFFFFFu, hi = 0u;
    for (int i = tid; i < len; i += nthr) {
        const uint32_t d = uint32_t(keys[start + i] >> 32);
        lo = min(lo, d);
        hi = max(hi, d);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((tid & 31) == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    // up to a bucket a key; the bins' table (kBlockBins + 1 words) ends the counters
    constexpr int kTable = kBlockBins + 8;
    int NB = 1;
    while (NB < len) NB <<= 1;
    if (NB > cap / 2 - kTable) NB = cap / 2 - kTable;
    const bool equi = NB >= 2 * kBlockBins;
    uint32_t* const bstart = cnt;
    uint32_t* const table = cnt + (cap / 2 - kTable);
    for (int i = tid; i < NB; i += nthr) bstart[i] = 0u;
    if (equi)
        for (int i = tid; i <= kBlockBins; i += nthr) table[i] = 0u;
    __syncthreads();
    const uint32_t dmin = s_lo;
    const float scale = float(equi ? kBlockBins : NB) / (float(s_hi - dmin) + 1.0f);
    if (equi) {
        for (int i = tid; i < len; i += nthr) {
            const float t = float(uint32_t(keys[start + i] >> 32) - dmin) * scale;
            atomicAdd(&table[min(kBlockBins - 1, int(t))], 1u);
        }
        __syncthreads();
        for (int c = tid; c < kBlockBins; c += nthr) {
            const uint32_t n = table[c];
            table[c] = n ? uint32_t(uint64_t(n) * uint32_t(NB - kBlockBins) / uint32_t(len)) + 1u : 0u;
        }
        __syncthreads();
        block_scan_counts(table, kBlockBins + 1);  // bin c: buckets [table[c], table[c + 1])
    }
    auto bucket = [&](unsigned long long k) {
        const float t = float(uint32_t(k >> 32) - dmin) * scale;
        if (!equi) return min(NB - 1, int(t));
        const int c = min(kBlockBins - 1, int(t));
        const int first = int(table[c]), nb = int(table[c + 1]) - first;
        return first + min(nb - 1, int((t - float(c)) * float(nb)));
    };
    for (int i = tid; i < len; i += nthr) atomicAdd(&bstart[bucket(keys[start + i])], 1u);
    __syncthreads();
    uint32_t most = 0u;
    for (int b = tid; b < NB; b += nthr) most = max(most, bstart[b]);
    most = __reduce_max_sync(0xffffffffu, most);
    if ((tid & 31) == 0) atomicMax(&s_most, most);
    __syncthreads();
    block_scan_counts(bstart, NB);
    most = s_most;
    for (int i = tid; i < len; i += nthr) {  // bstart[b]: the bucket's cursor
        const unsigned long long k = keys[start + i];
        sk[atomicAdd(&bstart[bucket(k)], 1u)] = k;
    }
    __syncthreads();
    if (most > uint32_t(kBucketSortLimit)) {
        bitonic_sort(sk, len);
    } else {
        ulonglong2* const two = reinterpret_cast<ulonglong2*>(sk);
        for (uint32_t ph = 0; most > 1u && ph < most; ++ph) {
            if ((ph & 1u) == 0u) {
                for (int i = tid; 2 * i + 1 < len; i += nthr) {
                    const ulonglong2 q = two[i];
                    if (q.x > q.y) two[i] = make_ulonglong2(q.y, q.x);
                }
            } else {
                for (int i = 2 * tid + 1; i + 1 < len; i += 2 * nthr) {
                    const unsigned long long x = sk[i], y = sk[i + 1];
                    if (x > y) {
                        sk[i] = y;
                        sk[i + 1] = x;
                    }
                }
            }
            __syncthreads();
        }
    }
}

// Keeps the low words of a block's sorted keys (Gaussian index << 4 | nibble)
// in place of the keys, as narrow_keys below; returns them.
__device__ __forceinline__ uint32_t* block_narrow(unsigned long long* sk, int len) {
    uint32_t* const idx = reinterpret_cast<uint32_t*>(sk);
    for (int base = 0; base < len; base += blockDim.x) {
        const int i = base + int(threadIdx.x);
        const uint32_t lo = i < len ? uint32_t(sk[i]) : 0u;
        __syncthreads();
        if (i < len) idx[i] = lo;
        __syncthreads();
    }
    return idx;
}

// Streams the sorted list's records through two shared-memory batches of
// blockDim.x records (cp.async prefetch of batch b+1 while batch b is
// blended) until every ray of the block is finished.
template <bool TRANSPOSED>
__device__ __forceinline__ void stream_list(const CompositeParams& p, const unsigned long long* sk,
                                            int len, int64_t vbase, const float4* __restrict__ rec,
                                            float4* buf, int* wbuf, Acc& a, bool& done,
                                            uint32_t& evals, float px, float py, int bx0, int bx1,
                                            int by0, int by1) {
    const int nthr = blockDim.x, t = threadIdx.x;
    // single shared batch: load (the record and, from the tile metadata, its
    // pixel box), barrier, blend, vote
    for (int b = 0; b < len; b += nthr) {
        const int i = b + t;
        if (i < len) {
            const int64_t e = vbase + (uint32_t(sk[i]) >> 4);
            const float4 q0 = rec[kRecordFloat4 * e], q1 = rec[kRecordFloat4 * e + 1];
            const uint4 m = p.meta[e];
            store_decoded(q0, q1, make_uint2(m.x, m.y), buf[t], buf[nthr + t], buf[2 * nthr + t]);
        }
        __syncthreads();
        const int nb = len - b < nthr ? len - b : nthr;
        eval_batch<TRANSPOSED>(a, done, evals, px, py, bx0, bx1, by0, by1, buf, buf + nthr,
                               buf + 2 * nthr, nb, wbuf);
        if (__syncthreads_count(done) == nthr) break;
    }
}

// Shared memory of a binned block: keys (cap), bucket counters (cap / 2),
// a record batch (3 x nthr float4), compaction buffers (64 ints per warp).
struct BinnedSmem {
    unsigned long long* sk;
    uint32_t* cnt;
    float4* buf;
    int* wbuf;
};

// Bytes of the key array (cap keys) and the bucket counters (cap / 2) of
// block_sort; a multiple of 16.
__host__ __device__ __forceinline__ size_t block_sort_bytes(int cap) { return 10 * size_t(cap); }

__device__ __forceinline__ BinnedSmem carve_binned(unsigned char* base, int cap, int nthr) {
    BinnedSmem m;
    m.sk = reinterpret_cast<unsigned long long*>(base);
    m.cnt = reinterpret_cast<uint32_t*>(base + 8 * size_t(cap));
    m.buf = reinterpret_cast<float4*>(base + block_sort_bytes(cap));
    m.wbuf = reinterpret_cast<int*>(m.buf + 3 * nthr) + 64 * (threadIdx.x >> 5);
    return m;
}

template <bool TRANSPOSED>
__global__ void __launch_bounds__(kBinnedThreads)
composite_rays_binned_kernel(CompositeParams p, const int4* __restrict__ gwork,
                             const int32_t* __restrict__ list, int cap,
                             const int2* __restrict__ grouped, const uint32_t* __restrict__ gstart,
                             const unsigned long long* __restrict__ keys,
                             const float4* __restrict__ rec, float* __restrict__ raycol,
                             unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char smb[];
    const int nthr = blockDim.x;
    const BinnedSmem S = carve_binned(smb, cap, nthr);
    const int4 wi = gwork[list[blockIdx.x]];
    const int v = wi.x / p.ntiles;
    const uint32_t start = gstart[wi.x];
    const int len = int(gstart[wi.x + 1] - start);
    block_sort(keys, start, len, cap, S.sk, S.cnt);
    const int64_t vbase = int64_t(v) * p.n;
    uint32_t evals = 0, blended = 0;
    for (int r0 = wi.y; r0 < wi.z; r0 += nthr) {
        const int rid = r0 + int(threadIdx.x);
        const bool active = rid < wi.z;
        const int2 ray = active ? grouped[rid] : make_int2(0, -1);
        const int col = int(uint32_t(ray.x) & 0xFFFFu), row = int(uint32_t(ray.x) >> 16);
        const float px = float(col) - p.half_w, py = float(row) - p.half_h;
        int bx0, bx1, by0, by1;
        warp_box(active, col, row, bx0, bx1, by0, by1);
        Acc a{1.f, 0.f, 0.f, 0.f, 0u};
        bool done = !active;
        stream_list<TRANSPOSED>(p, S.sk, len, vbase, rec, S.buf, S.wbuf, a, done, evals, px, py,
                                bx0, bx1, by0, by1);
        if (active) {
            float* o = raycol + 3 * int64_t(rid);  // grouped order
            o[0] = a.c0;
            o[1] = a.c1;
            o[2] = a.c2;
        }
        blended += a.blended;
    }
    if (pairs) count_pairs(pairs, evals, blended);
}

// The standard paradigm under DL_EVAL_TRANSPOSED: a block per (view, tile), a
// thread per pixel.  (Direct evaluation, the default: composite_views_*.)
__global__ void __launch_bounds__(1024, 1)
composite_full_binned_kernel(CompositeParams p, const int32_t* __restrict__ list, int cap,
                             const uint32_t* __restrict__ gstart,
                             const unsigned long long* __restrict__ keys,
                             const float4* __restrict__ rec, float* __restrict__ Mm,
                             unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char smb[];
    const int nthr = blockDim.x;
    const BinnedSmem S = carve_binned(smb, cap, nthr);
    const int group = list[blockIdx.x];
    const int v = group / p.ntiles;
    const int tile = group - v * p.ntiles;
    const int tx = tile % p.ntx, ty = tile / p.ntx;
    const int col = tx * p.tile_w + int(threadIdx.x) % p.tile_w;
    const int row = ty * p.tile_h + int(threadIdx.x) / p.tile_w;
    const bool inside = col < p.width && row < p.height;
    const float px = float(col) - p.half_w, py = float(row) - p.half_h;
    const uint32_t start = gstart[group];
    const int len = int(gstart[group + 1] - start);
    block_sort(keys, start, len, cap, S.sk, S.cnt);
    int bx0, bx1, by0, by1;
    warp_box(inside, col, row, bx0, bx1, by0, by1);
    const int64_t vbase = int64_t(v) * p.n;
    Acc a{1.f, 0.f, 0.f, 0.f, 0u};
    uint32_t evals = 0;
    bool done = !inside;
    stream_list<true>(p, S.sk, len, vbase, rec, S.buf, S.wbuf, a, done, evals, px, py, bx0,
                            bx1, by0, by1);
    if (pairs) count_pairs(pairs, evals, a.blended);
    if (inside) {
        float* o = Mm + ((int64_t(v) * p.height + row) * p.width + col) * 3;
        o[0] = a.c0;
        o[1] = a.c1;
        o[2] = a.c2;
    }
}

// ------------------------------------------------- one warp per tile ----
// DirectL tiles hold few rays (tens) and a few hundred Gaussians, so each
// warp owns one (view, tile) group: it sorts the group's keys in its own
// shared memory (warp-level bucket sort), streams the records in batches of
// 32 with cp.async (up to three batches ahead), and evaluates them transposed
// against its rays.  Only __syncwarp is used, so warps never wait on each
// other.
constexpr int kWarpsPerBlock = 4;

// Positions of the warp's rays about their box centre (x, y), written per
// ray chunk, the per-ray candidate masks of one batch and the third colour
// channel of its records (the other two are decoded in place).  Coordinates
// are stored apart, so four rays' x (or y) are one 16-byte read.
struct RayTable {
    float4 x[8], y[8];
    uint4 mask[8];
    float blue[32];
};

// A warp's shared memory holds its group's keys while it sorts them and,
// once sorted, only their low words (Gaussian index << 4 | quadrant nibble)
// beside the record batches and the ray table: the two phases share the
// space, which keeps the 1024-key class at six blocks per SM.
template <int CAP>
struct WarpStream {
    // record batch slots (one being composited, the rest in flight): as many
    // 32-record batches of 32-byte records as fit in the space the sort phase
    // needs anyway (the 512-key class at eight blocks per SM, the 1024-key
    // class at six)
    static constexpr int kSlots = CAP <= 512 ? 3 : 4;
    uint32_t idx[CAP];
    float4 buf[kSlots][kRecordFloat4][32];
    RayTable rays;
};
template <int CAP>
union WarpSmem {
    WarpSort<CAP> s;
    WarpStream<CAP> c;
};
static_assert(sizeof(WarpSort<512>) <= sizeof(WarpStream<512>), "sort phase fits the stream's space");
static_assert(sizeof(WarpStream<1024>) <= sizeof(WarpSort<1024>), "stream phase fits the sort's space");
// blocks of kWarpsPerBlock warps per SM: eight (512-key class, 64
// registers a thread) and six (1024-key class, 80 registers); 228 KB of
// shared memory an SM, 1 KB of it reserved per block
template <int CAP>
constexpr int warp_class_blocks() { return CAP <= 512 ? 8 : 6; }
static_assert(warp_class_blocks<1024>() * (kWarpsPerBlock * sizeof(WarpSmem<1024>) + 1024) <=
                  228 * 1024, "1024-key class: 6 blocks");
static_assert(warp_class_blocks<512>() * (kWarpsPerBlock * sizeof(WarpSmem<512>) + 1024) <=
                  228 * 1024, "512-key class: 8 blocks");

// Keeps the low words of the warp's sorted keys (Gaussian index << 4 |
// nibble) in place of the keys: chunk by chunk, each chunk read whole before
// it is written, and a chunk's 32 words land on keys already read (the words
// of chunk c take bytes [128 c, 128 c + 128), below the chunk's own keys).
template <int CAP>
__device__ __forceinline__ void narrow_keys(WarpSmem<CAP>& W, int len) {
    const int lane = threadIdx.x & 31;
    for (int base = 0; base < len; base += 32) {
        const int i = base + lane;
        const uint32_t lo = i < len ? uint32_t(W.s.sk[i]) : 0u;
        __syncwarp();
        if (i < len) W.c.idx[i] = lo;
        __syncwarp();
    }
}

// Margin of the batch test below: the expanded quadratic is rounded
// differently from log2_alpha, by less than 0.05 for tiles up to 256 x 256
// pixels (its terms are bounded by lambda_max(conic) <= 1/0.3 times the
// squared distance from the box centre), so a pair passes the test whenever
// log2_alpha reaches the threshold; blend() then decides exactly.
constexpr float kTestMargin = 0.05f;

// Transposed evaluation of a batch of n <= 32 records held in shared memory
// (c0, c1: the two halves of each record) for the warp's rays: lane j holds
// record j's conic (u, v, A, B, C, L) and packed colour (pc, pd) when `hit`
// (j < n).  The lane decodes the colour once for every ray that will blend
// the record (r, g over the packed words, b into T.blue), then expands the
// quadratic about the box centre (ox, oy) into
// l2(x, y) = x (A x + B y + D) + y (C y + E) + F and tests it against every
// ray (5 FMAs per pair, ray positions from the table), four rays per step
// with the FMAs paired over two rays (packed FP32x2 FMA: per component the
// same rounding as fmaf); ray r's mask of candidate records goes to
// T.mask[r].  Then every lane blends its candidates in list order.
template <bool COUNT>
__device__ __forceinline__ void eval32(const float4* c0, float4* c1, int n, bool hit, float u,
                                       float v, float A, float B, float C, float L, float pc,
                                       float pd, Acc& a, bool& done, uint32_t& evals, float px,
                                       float py, RayTable& T, float ox, float oy) {
    const int lane = threadIdx.x & 31;
    if (!__any_sync(0xffffffffu, hit)) return;
    if (hit) {
        float r, g, b;
        unpack_rgb(pc, pd, r, g, b);
        reinterpret_cast<float2*>(c1 + lane)[1] = make_float2(r, g);
        T.blue[lane] = b;
    }
    const unsigned act = __ballot_sync(0xffffffffu, !done);
    const float du = u - ox, dv = v - oy;
    const float D = -fmaf(2.f * A, du, B * dv);
    const float E = -fmaf(2.f * C, dv, B * du);
    const float F = hit ? fmaf(du, fmaf(A, du, B * dv), fmaf(C * dv, dv, L)) + kTestMargin : -1e30f;
    const float2 A2 = make_float2(A, A), B2 = make_float2(B, B), C2 = make_float2(C, C);
    const float2 D2 = make_float2(D, D), E2 = make_float2(E, E), F2 = make_float2(F, F);
#pragma unroll
    for (int g = 0; g < 8; ++g) {
        if (!((act >> (4 * g)) & 0xFu)) continue;
        const float4 qx = T.x[g], qy = T.y[g];
        unsigned m[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 x = h ? make_float2(qx.z, qx.w) : make_float2(qx.x, qx.y);
            const float2 y = h ? make_float2(qy.z, qy.w) : make_float2(qy.x, qy.y);
            const float2 t1 = __ffma2_rn(A2, x, __ffma2_rn(B2, y, D2));
            const float2 l2 = __ffma2_rn(x, t1, __ffma2_rn(y, __ffma2_rn(C2, y, E2), F2));
            m[2 * h] = __ballot_sync(0xffffffffu, l2.x >= kLog2MinAlpha);
            m[2 * h + 1] = __ballot_sync(0xffffffffu, l2.y >= kLog2MinAlpha);
        }
        if (lane == 0) T.mask[g] = make_uint4(m[0], m[1], m[2], m[3]);
    }
    __syncwarp();
    unsigned mine = (act >> lane) & 1u ? reinterpret_cast<const unsigned*>(T.mask)[lane] : 0u;
    if (COUNT && !done) evals += uint32_t(n);
    while (mine && !done) {  // candidates passed the (widened) test: alpha decides
        const int s1 = __ffs(mine) - 1;
        mine &= mine - 1;
        const bool two = mine != 0u;
        const int s2 = two ? __ffs(mine) - 1 : s1;
        mine &= mine - 1u;
        if (!blend2<COUNT>(a, px, py, c0[s1], c1[s1], T.blue[s1], c0[s2], c1[s2], T.blue[s2], two))
            done = true;
    }
    __syncwarp();
}

// Fills the ray table for the warp's current rays (box centre (ox, oy)).
__device__ __forceinline__ void ray_table(RayTable& T, bool active, float px, float py, float& ox,
                                          float& oy, int bx0, int bx1, int by0, int by1,
                                          float half_w, float half_h) {
    const int lane = threadIdx.x & 31;
    ox = 0.5f * float(bx0 + bx1) - half_w;
    oy = 0.5f * float(by0 + by1) - half_h;
    reinterpret_cast<float*>(T.x)[lane] = active ? px - ox : 1e18f;
    reinterpret_cast<float*>(T.y)[lane] = active ? py - oy : 1e18f;
    __syncwarp();
}

// Lane's record of a shared-memory batch: loads its conic and packed colour
// into registers (lanes past the batch hold a conic that no ray passes).  A
// tile list holds only records whose pixel box meets the tile, and the
// warp's rays spread over the tile, so no box pre-test is made: the widened
// test below sorts the records out at a few FMAs per pair.
__device__ __forceinline__ bool batch_conic(const float4* c0, const float4* c1, int n, float& u,
                                            float& v, float& A, float& B, float& C, float& L,
                                            float& pc, float& pd) {
    const int lane = threadIdx.x & 31;
    u = 0.f; v = 0.f; A = 0.f; B = 0.f; C = 0.f; L = -1e30f; pc = 0.f; pd = 0.f;
    if (lane >= n) return false;
    const float4 q0 = c0[lane];
    const float4 q1 = c1[lane];
    u = q0.x; v = q0.y; A = q0.z; B = q0.w; C = q1.x; L = q1.y; pc = q1.z; pd = q1.w;
    return true;
}

// Streams the warp's sorted list in batches of 32 records (cp.async, up to
// three batches ahead) and composites them, transposed, for the warp's rays.
template <int CAP, bool COUNT>
__device__ __forceinline__ void warp_stream(WarpSmem<CAP>& W, int len, int64_t vbase,
                                            const float4* __restrict__ rec, Acc& a, bool& done,
                                            uint32_t& evals, float px, float py, int bx0, int bx1,
                                            int by0, int by1, float ox, float oy) {
    const int lane = threadIdx.x & 31;
    const int nbatch = (len + 31) / 32;
    if (nbatch == 0) return;
    constexpr int S = WarpStream<CAP>::kSlots;
    // batch b goes to slot b mod S; S - 1 batches are in flight ahead of the
    // one being composited (one cp.async group per batch, empty past the end)
    auto issue = [&](int b, int slot) {
        const int i = b * 32 + lane;
        if (b < nbatch && i < len) {
            const int64_t e = vbase + (W.c.idx[i] >> 4);
            cp_async16(&W.c.buf[slot][0][lane], rec + kRecordFloat4 * e);
            cp_async16(&W.c.buf[slot][1][lane], rec + kRecordFloat4 * e + 1);
        }
        cp_async_commit();
    };
#pragma unroll
    for (int k = 0; k < S - 1; ++k) issue(k, k);
    int slot = 0;  // b mod S
    for (int b = 0; b < nbatch; ++b) {
        issue(b + S - 1, slot == 0 ? S - 1 : slot - 1);
        cp_async_wait<S - 1>();
        __syncwarp();
        const float4* c0 = W.c.buf[slot][0];
        float4* c1 = W.c.buf[slot][1];
        slot = slot + 1 == S ? 0 : slot + 1;
        const int n = len - b * 32 < 32 ? len - b * 32 : 32;
        float u, v, A, B, C, L, pc, pd;
        const bool hit = batch_conic(c0, c1, n, u, v, A, B, C, L, pc, pd);
        eval32<COUNT>(c0, c1, n, hit, u, v, A, B, C, L, pc, pd, a, done, evals, px, py, W.c.rays,
                      ox, oy);
        if (__all_sync(0xffffffffu, done)) break;
    }
    cp_async_wait<0>();
    __syncwarp();
}

// Per-warp shared memory of the quadrant block kernel: list positions
// selected for the warp's quadrant and not yet batched, and two batches of 32
// records in flight (cp.async double buffering).
struct QuadPipe {
    int stage[64];
    int idx[2][32];
    float4 buf[2][kRecordFloat4][32];
    RayTable rays;
};

// Streams the records of a block-sorted list whose key marks quadrant `q`
// (bit q of the key's low nibble) for the warp's rays, in list order: the
// selected positions are compacted 32 at a time and their records fetched
// with cp.async one batch ahead of the batch being evaluated (as in
// warp_stream).
__device__ void quadrant_stream(const uint32_t* idx, int len, int q, int64_t vbase,
                                const float4* __restrict__ rec, QuadPipe& Q, Acc& a, bool& done,
                                uint32_t& evals, float px, float py, int bx0, int bx1, int by0,
                                int by1, float ox, float oy) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int pos = 0, cnt = 0;  // scan position, staged positions (uniform)
    // next batch of up to 32 selected positions into Q.idx[slot], its records
    // requested; returns its size
    auto produce = [&](int slot) -> int {
        while (cnt < 32 && pos < len) {
            const int i = pos + lane;
            const bool sel = i < len && ((idx[i] >> q) & 1u);
            const unsigned m = __ballot_sync(0xffffffffu, sel);
            if (sel) Q.stage[cnt + __popc(m & lt)] = i;
            cnt += __popc(m);
            pos += 32;
            __syncwarp();
        }
        const int n = cnt < 32 ? cnt : 32;
        const int mine = lane < n ? Q.stage[lane] : 0;
        const int rest = lane + 32 < cnt ? Q.stage[lane + 32] : 0;
        __syncwarp();
        if (lane + 32 < cnt) Q.stage[lane] = rest;
        Q.idx[slot][lane] = mine;
        cnt -= n;
        if (lane < n) {
            const int64_t e = vbase + (idx[mine] >> 4);
            cp_async16(&Q.buf[slot][0][lane], rec + kRecordFloat4 * e);
            cp_async16(&Q.buf[slot][1][lane], rec + kRecordFloat4 * e + 1);
        }
        cp_async_commit();
        __syncwarp();
        return n;
    };
    int slot = 0;
    int n_cur = produce(0);
    while (n_cur > 0) {
        const int n_next = __all_sync(0xffffffffu, done) ? 0 : produce(slot ^ 1);
        if (n_next > 0) cp_async_wait<1>();
        else cp_async_wait<0>();
        __syncwarp();
        const float4* c0 = Q.buf[slot][0];
        float4* c1 = Q.buf[slot][1];
        float u, v, A, B, C, L, pc, pd;
        const bool hit = batch_conic(c0, c1, n_cur, u, v, A, B, C, L, pc, pd);
        eval32<true>(c0, c1, n_cur, hit, u, v, A, B, C, L, pc, pd, a, done, evals, px, py, Q.rays,
                     ox, oy);
        slot ^= 1;
        n_cur = __all_sync(0xffffffffu, done) ? 0 : n_next;
    }
    cp_async_wait<0>();
    __syncwarp();
}


// Index of the frame whose class range holds item i: the last f with
// prefix[f] <= i (prefix ascending, prefix[0] = 0).
__device__ __forceinline__ int frame_of(const int64_t* __restrict__ prefix, int n_frames, int64_t i) {
    int lo = 0, hi = n_frames - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(prefix + mid) <= i) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Item i of class cls (0: front of items, 1: back of items) across frames.
__device__ __forceinline__ int4 batch_item(const FrameDesc* __restrict__ F,
                                           const int64_t* __restrict__ prefix, int n_frames, int cls,
                                           int64_t i, int& f) {
    f = frame_of(prefix, n_frames, i);
    const int64_t j = i - __ldg(prefix + f);
    const int4* items = F[f].items;
    return cls == 0 ? items[j] : items[F[f].n_work - 1 - j];
}

// Persistent: resident warps take items until none is left (the first
// n_warps by warp id, the rest claimed from *cursor: groups differ widely in
// cost); an item is {group, first key, first ray, rays << 16 | keys} of
// frame f.  The next item is claimed and loaded before the current one is
// composited.  (Prefetching its keys and rays into L2 as well measured
// slower once eight blocks of the 512-key class were resident.)
template <int CAP, bool COUNT>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, warp_class_blocks<CAP>())
composite_rays_warp_kernel(const FrameDesc* __restrict__ F, const int64_t* __restrict__ prefix,
                           int n_frames, int cls, uint32_t* __restrict__ cursor,
                           unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char wsm_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WarpSmem<CAP>& W = reinterpret_cast<WarpSmem<CAP>*>(wsm_raw)[warp];
    const int64_t n_items = __ldg(prefix + n_frames);
    const int64_t n_warps = int64_t(gridDim.x) * kWarpsPerBlock;
    int64_t item = int64_t(blockIdx.x) * kWarpsPerBlock + warp;
    uint32_t evals = 0, blended = 0;
    int fcur = 0;
    int4 cur = item < n_items ? batch_item(F, prefix, n_frames, cls, item, fcur) : make_int4(0, 0, 0, 0);
    while (item < n_items) {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(cursor, 1u);
        const int64_t nxt = n_warps + int64_t(__shfl_sync(0xffffffffu, c, 0));
        int fnxt = 0;
        const int4 next = nxt < n_items ? batch_item(F, prefix, n_frames, cls, nxt, fnxt)
                                        : make_int4(0, 0, 0, 0);
        const FrameDesc& d = F[fcur];
        const int2* __restrict__ grouped = d.grouped;
        const float4* __restrict__ rec = d.rec;
        float* __restrict__ raycol = d.raycol;
        const int group = cur.x;
        const uint32_t start = uint32_t(cur.y);
        const int rbeg = cur.z, nrays = int(uint32_t(cur.w) >> 16), len = cur.w & 0xFFFF;
        const int v = group / d.cp.ntiles;
        const float half_w = d.cp.half_w, half_h = d.cp.half_h;
        warp_sort<CAP>(d.keys, start, len, W.s);
        narrow_keys<CAP>(W, len);
        const int64_t vbase = int64_t(v) * d.cp.n;
        for (int r0 = 0; r0 < nrays; r0 += 32) {
            const int rid = r0 + lane;
            const bool active = rid < nrays;
            const int2 ray = active ? grouped[rbeg + rid] : make_int2(0, -1);
            const int col = int(uint32_t(ray.x) & 0xFFFFu), row = int(uint32_t(ray.x) >> 16);
            const float px = float(col) - half_w, py = float(row) - half_h;
            int bx0, bx1, by0, by1;
            warp_box(active, col, row, bx0, bx1, by0, by1);
            float ox, oy;
            ray_table(W.c.rays, active, px, py, ox, oy, bx0, bx1, by0, by1, half_w, half_h);
            Acc a{1.f, 0.f, 0.f, 0.f, 0u};
            bool done = !active;
            warp_stream<CAP, COUNT>(W, len, vbase, rec, a, done, evals, px, py, bx0, bx1, by0, by1,
                                    ox, oy);
            if (active) {
                float* o = raycol + 3 * (int64_t(rbeg) + rid);  // grouped order
                o[0] = a.c0;
                o[1] = a.c1;
                o[2] = a.c2;
            }
            blended += a.blended;
        }
        item = nxt;
        cur = next;
        fcur = fnxt;
    }
    if (COUNT) count_pairs(pairs, evals, blended);
}

// Warp q's part of a group whose list a block has sorted: the rays in quadrant q
// of the tile, over the records marked for it.
__device__ __forceinline__ void composite_quadrant(const FrameDesc& d, const int4& wi, const uint32_t* idx,
                                                   int len, QuadPipe& pipe, uint32_t& evals,
                                                   uint32_t& blended) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int v = wi.x / d.cp.ntiles;
    const int tile = wi.x - v * d.cp.ntiles;
    const int xm = (tile % d.cp.ntx) * d.cp.tile_w + (d.cp.tile_w >> 1);
    const int ym = (tile / d.cp.ntx) * d.cp.tile_h + (d.cp.tile_h >> 1);
    const int qx = warp & 1, qy = warp >> 1;
    const int64_t vbase = int64_t(v) * d.cp.n;
    for (int r0 = wi.y; r0 < wi.z; r0 += 32) {
        const int rid = r0 + lane;
        const int2 ray = rid < wi.z ? d.grouped[rid] : make_int2(0, -1);
        const int col = int(uint32_t(ray.x) & 0xFFFFu), row = int(uint32_t(ray.x) >> 16);
        const bool mine = rid < wi.z && int(col >= xm) == qx && int(row >= ym) == qy;
        if (!__any_sync(0xffffffffu, mine)) continue;
        const float px = float(col) - d.cp.half_w, py = float(row) - d.cp.half_h;
        int bx0, bx1, by0, by1;
        warp_box(mine, col, row, bx0, bx1, by0, by1);
        float ox, oy;
        ray_table(pipe.rays, mine, px, py, ox, oy, bx0, bx1, by0, by1, d.cp.half_w, d.cp.half_h);
        Acc a{1.f, 0.f, 0.f, 0.f, 0u};
        bool done = !mine;
        quadrant_stream(idx, len, warp, vbase, d.rec, pipe, a, done, evals, px, py, bx0, bx1, by0, by1,
                        ox, oy);
        if (mine) {
            float* o = d.raycol + 3 * int64_t(rid);  // grouped order
            o[0] = a.c0;
            o[1] = a.c1;
            o[2] = a.c2;
        }
        blended += a.blended;
    }
}

// Block class across frames: one block of four warps per group list too long
// for a warp (sorted together in shared memory up to `cap` keys); warp q then
// composites the group's rays in quadrant q of the tile (x half + 2 * y half)
// over the records whose key marks that quadrant, so every warp has work and
// each streams only about half of the list.  Persistent like the warp
// classes.
__global__ void __launch_bounds__(kBinnedThreads)
composite_rays_block_kernel(const FrameDesc* __restrict__ F, const int64_t* __restrict__ prefix,
                            int n_frames, int2 caps, uint32_t* __restrict__ cursor,
                            unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char smb[];
    __shared__ int64_t s_item;
    const int cap = caps.x;  // keys in shared memory; caps.y: the longest list
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(smb);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smb + 8 * size_t(cap));
    QuadPipe* pipes = reinterpret_cast<QuadPipe*>(smb + 4 * size_t(cap));  // after the sort
    const int warp = threadIdx.x >> 5;
    const int64_t n_items = __ldg(prefix + n_frames);
    uint32_t evals = 0, blended = 0;
    int64_t item = blockIdx.x;
    while (item < n_items) {
        const int f = frame_of(prefix, n_frames, item);
        const FrameDesc& d = F[f];
        const int4 bi = d.block_items[item - __ldg(prefix + f)];
        const int4 wi = d.gwork[bi.z];
        const uint32_t start = uint32_t(bi.y);
        const int len = bi.w;
        if (len > caps.y) {
            if (threadIdx.x == 0) atomicOr(d.status, 2u);
        } else if (len <= cap) {  // (the ones between: composite_rays_long_kernel)
            // the keys carry the quadrant bits (bit q: the record's pixel
            // box overlaps quadrant q, x half + 2 * y half, of the tile)
            block_sort(d.keys, start, len, cap, sk, cnt);
            composite_quadrant(d, wi, block_narrow(sk, len), len, pipes[warp], evals, blended);
        }
        __syncthreads();  // shared memory reused by the next item
        if (threadIdx.x == 0) s_item = int64_t(gridDim.x) + int64_t(atomicAdd(cursor, 1u));
        __syncthreads();
        item = s_item;
    }
    if (pairs) count_pairs(pairs, evals, blended);
}

// One frame's block lists of more than caps.x and at most caps.y keys: lists
// that outgrew the shared memory their signature was sized for, sorted where
// they lie (a slice of the key buffer is its group's own).  Few frames hold any
// (the next one is sized again), so a block looks through its share of the items
// a thread each.  Within the block class's kernel it cost that 3 % (7.9-inch
// panel, whole frame 2.07 -> 2.11 ms).
__global__ void __launch_bounds__(kBinnedThreads)
composite_rays_long_kernel(const FrameDesc* __restrict__ F, const int64_t* __restrict__ prefix, int2 caps,
                           unsigned long long* __restrict__ pairs) {
    __shared__ QuadPipe pipes[kBinnedThreads / 32];
    __shared__ uint32_t s_long[kBinnedThreads / 32];
    const FrameDesc& d = *F;
    const int64_t n_items = prefix[1];
    const int warp = threadIdx.x >> 5;
    uint32_t evals = 0, blended = 0;
    for (int64_t i0 = 0; i0 * gridDim.x + blockIdx.x < n_items; i0 += kBinnedThreads) {
        const int64_t mine = (i0 + threadIdx.x) * gridDim.x + blockIdx.x;
        const int len = mine < n_items ? d.block_items[mine].w : 0;
        const uint32_t m = __ballot_sync(0xffffffffu, len > caps.x && len <= caps.y);
        if ((threadIdx.x & 31) == 0) s_long[warp] = m;
        __syncthreads();
        for (int w = 0; w < kBinnedThreads / 32; ++w) {
            for (uint32_t left = s_long[w]; left; left &= left - 1u) {
                const int t = 32 * w + __ffs(left) - 1;
                const int4 bi = d.block_items[(i0 + t) * gridDim.x + blockIdx.x];
                unsigned long long* const own =
                    const_cast<unsigned long long*>(d.keys) + uint32_t(bi.y);
                bitonic_sort(own, bi.w);
                composite_quadrant(d, d.gwork[bi.z], block_narrow(own, bi.w), bi.w, pipes[warp], evals,
                                   blended);
            }
        }
        __syncthreads();  // s_long is written again
    }
    if (pairs) count_pairs(pairs, evals, blended);
}

// ------------------------------------------------ standard paradigm ----
// Every pixel of every view.  A warp owns one (view, tile) group, sorts its
// keys in its own shared memory (warp_sort) and composites the tile one 8 x 8
// patch after another, two horizontally adjacent pixels a lane.  The stage is
// bound by issued instructions, so the work per (pixel, Gaussian) pair is
// what counts:
//  - a patch only walks the records whose alpha >= 1/255 ellipse reaches it:
//    one pass over the list, a record a lane, makes the masks of four patches
//    (a 16 x 16 quad) at once; a patch then gathers its records 32 at a time
//    into a shared-memory batch that the loop reads by broadcast;
//  - two pixels of a row share the row's terms of the quadratic (4 of its 7
//    operations), the record's loads and the loop, and their transmittance
//    and colour updates are packed FP32x2 operations (per component the
//    rounding of the scalar ones);
//  - a finished pixel is one whose alpha threshold is out of reach, so no
//    select guards the blend; whether a pixel finishes is asked once every
//    kBlendRun records, and the branch that finishes it is taken once.
// A larger patch culls worse and a smaller one shares less.  A warp per tile
// needs no block barrier for its sort.  Lists of more than 1024 keys:
// composite_views_block_kernel.
// Measured against a block per tile with one pixel a lane in 16 x 2 strips:
// 1080p (200k Gaussians, 45 views) 11.25 -> 4.07 ms, 4K (1M) 47.3 -> 17.0 ms,
// 4K panel with 800 x 450 views 9.17 -> 3.79 ms; of the 1080p stage the blend
// loop is about 2.7 ms (35 instructions for 64 pairs, then 30 with the runs),
// the sort 0.4 ms and the masks and batches the rest.
constexpr int kPatch = 8;
constexpr int kBlendRun = 4;  // records blended between two looks at the transmittance

// A patch's records, as the blend loop reads them: (u, v, A, B), (-r, -r, -g,
// -g), (-b, -b, C, L); the colours are negated and doubled for the packed
// update below.  stage: list positions selected and not yet batched.
struct PatchBatch {
    float4 geo[32], rg[32], bcl[32];
    uint32_t stage[64];
};

// Two pixels (x0, y), (x1, y) of a lane: transmittance and colour pairs, and
// per pixel the negated alpha a record has to reach (-1/255; -inf once the
// pixel is finished).
struct Px2 {
    float x0, x1, y, th0, th1;
    float2 T, r, g, b;
    uint32_t blended;
};

// Masks of the 32 records of a batch (lane i holds record i, `valid`) for the
// four patches of the quad at (qx, qy): bit i of component k is set when the
// record may reach alpha >= 1/255 at a pixel of patch k (x half + 2 * y
// half).  That is the largest value of its quadratic over the patch (pixel
// centres relative to the principal point) against the threshold: the
// quadratic is concave, so with its centre outside the patch the maximum is
// on one of the two edges that face the centre, at the best point of the
// nearest vertical edge (dy = -B dx / 2C, clamped) or of the nearest
// horizontal one.  The margin covers the rounding here and in log2_alpha:
// every term is below q = |A| dx^2 + |C| dy^2 at the quad's far corner (so is
// B dx dy, as B^2 <= 4 A C), and the two evaluations add less than 30
// roundings of 2^-24 q each.  A record that is not a number is kept.
__device__ __forceinline__ uint4 quad_masks(bool valid, float u, float v, float A, float B, float C,
                                            float L, const float (&x0)[2], const float (&x1)[2],
                                            const float (&y0)[2], const float (&y1)[2]) {
    const float hb = -0.5f * B, rc = hb * rcp_approx(C), ra = hb * rcp_approx(A);
    float lx[2], hx[2], ex[2], ly[2], hy[2], ey[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        lx[k] = x0[k] - u;
        hx[k] = x1[k] - u;
        ex[k] = fminf(fmaxf(0.f, lx[k]), hx[k]);
        ly[k] = y0[k] - v;
        hy[k] = y1[k] - v;
        ey[k] = fminf(fmaxf(0.f, ly[k]), hy[k]);
    }
    const float fx = fmaxf(-lx[0], hx[1]), fy = fmaxf(-ly[0], hy[1]);
    const float margin = fmaf(fmaf(-A * fx, fx, -C * fy * fy), 4e-6f, 0.01f);
    const float need = kLog2MinAlpha - L - margin;
    unsigned m[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = k & 1, j = k >> 1;
        const float oy = fminf(fmaxf(ex[i] * rc, ly[j]), hy[j]);
        const float ox = fminf(fmaxf(ey[j] * ra, lx[i]), hx[i]);
        const float f1 = fmaf(ex[i], fmaf(A, ex[i], B * oy), C * oy * oy);
        const float f2 = fmaf(ox, fmaf(A, ox, B * ey[j]), C * ey[j] * ey[j]);
        m[k] = __ballot_sync(0xffffffffu, valid && !(fmaxf(f1, f2) < need));
    }
    return make_uint4(m[0], m[1], m[2], m[3]);
}

// blend() of kBlendRun records (from `k` of the batch) on a lane's two
// pixels: the same operations in the same order per pixel (the signs of alpha
// and of the colour are both flipped, which changes no rounding).  blend()'s
// test of log2 alpha is implied by the one of alpha: one step below that
// threshold 2^x is 2.9e-7 below FP32's 1/255, more than ex2's error of 2^-22.
template <bool COUNT>
__device__ __forceinline__ void blend_run(Px2& p, const PatchBatch& S, int k) {
    float2 a[kBlendRun], w[kBlendRun];
    float2 T = p.T;
#pragma unroll
    for (int j = 0; j < kBlendRun; ++j) {
        const float4 geo = S.geo[k + j];
        const float2 cl = reinterpret_cast<const float2*>(S.bcl + k + j)[1];
        const float dy = p.y - geo.y, bdy = geo.w * dy, row = fmaf(cl.x * dy, dy, cl.y);
        const float dx0 = p.x0 - geo.x, dx1 = p.x1 - geo.x;
        const float l0 = fmaf(dx0, fmaf(geo.z, dx0, bdy), row);
        const float l1 = fmaf(dx1, fmaf(geo.z, dx1, bdy), row);
        const float a0 = fmaxf(-0.99f, -ex2_approx(l0)), a1 = fmaxf(-0.99f, -ex2_approx(l1));
        a[j] = make_float2(a0 <= p.th0 ? a0 : 0.f, a1 <= p.th1 ? a1 : 0.f);
        w[j] = __fmul2_rn(a[j], T);
        T = __fadd2_rn(T, w[j]);
    }
    // the transmittance only falls, so the last one tells whether a pixel
    // finishes inside the run; then the run is taken record by record
    if (fminf(T.x, T.y) < 1e-4f) {
        T = p.T;
        bool d0 = false, d1 = false;
#pragma unroll
        for (int j = 0; j < kBlendRun; ++j) {
            w[j] = __fmul2_rn(a[j], T);
            const float2 Tn = __fadd2_rn(T, w[j]);
            d0 = d0 || Tn.x < 1e-4f;
            d1 = d1 || Tn.y < 1e-4f;
            if (d0) { w[j].x = 0.f; a[j].x = 0.f; } else T.x = Tn.x;
            if (d1) { w[j].y = 0.f; a[j].y = 0.f; } else T.y = Tn.y;
        }
        if (d0) p.th0 = -INFINITY;
        if (d1) p.th1 = -INFINITY;
    }
    p.T = T;
#pragma unroll
    for (int j = 0; j < kBlendRun; ++j) {
        const float4 rg = S.rg[k + j];
        p.r = __ffma2_rn(w[j], make_float2(rg.x, rg.y), p.r);
        p.g = __ffma2_rn(w[j], make_float2(rg.z, rg.w), p.g);
        p.b = __ffma2_rn(w[j], reinterpret_cast<const float2*>(S.bcl + k + j)[0], p.b);
        if (COUNT) p.blended += (a[j].x < 0.f) + (a[j].y < 0.f);
    }
}

// A patch again, record by record as blend() takes them, for a lane's pixels
// (x0, y) and (x1, y), written to o (in0, in1: those inside the view); returns
// the records blended.  blend_run multiplies every record's colour, those below
// the threshold by an alpha of 0, which turns a colour that overflowed to
// infinity into NaN in every pixel of the patch, and nothing else does.  So a
// patch that ends with a NaN comes here.  (A vote a batch for infinite colours
// cost every frame 1.7 %: 1080p 4.72 -> 4.80 ms.  Not inlined, so that it
// takes no registers from the loop.)
template <bool COUNT, class Index>
__device__ __noinline__ uint32_t patch_by_records(const uint4* masks, int comp, Index index, int len,
                                                  const float4* __restrict__ base, float x0, float x1,
                                                  float y, bool in0, bool in1, float* o) {
    Acc a{1.f, 0.f, 0.f, 0.f, 0u}, b = a;
    bool open0 = in0, open1 = in1;
    for (int i0 = 0; i0 < len && __any_sync(0xffffffffu, open0 || open1); i0 += 32) {
        for (unsigned m = reinterpret_cast<const unsigned*>(masks + (i0 >> 5))[comp]; m; m &= m - 1u) {
            const float4* r = base + kRecordFloat4 * int64_t(index(i0 + __ffs(m) - 1));
            const float4 q0 = __ldg(r), q1 = __ldg(r + 1);
            if (open0) open0 = blend_rec<true, COUNT>(a, x0, y, q0, q1);
            if (open1) open1 = blend_rec<true, COUNT>(b, x1, y, q0, q1);
        }
    }
    if (in0) {
        o[0] = a.c0;
        o[1] = a.c1;
        o[2] = a.c2;
    }
    if (in1) {
        o[3] = b.c0;
        o[4] = b.c1;
        o[5] = b.c2;
    }
    return a.blended + b.blended;
}

// Composites one patch for the warp (columns from col0, rows from row0 of
// view v): the records index(0 .. len) that masks (component `comp` of a
// batch's uint4) select, in list order, and writes its pixels.
template <bool COUNT, class Index>
__device__ __forceinline__ void composite_patch(const CompositeParams& p, int v, int col0, int row0,
                                                const uint4* masks, int comp, Index index, int len,
                                                const float4* __restrict__ base, PatchBatch& S,
                                                float* __restrict__ Mm, uint32_t& evals,
                                                uint32_t& blended) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const int col = col0 + 2 * (lane & 3), row = row0 + (lane >> 2);
    const bool in0 = col < p.width && row < p.height, in1 = col + 1 < p.width && row < p.height;
    Px2 q;
    q.x0 = float(col) - p.half_w;
    q.x1 = float(col + 1) - p.half_w;
    q.y = float(row) - p.half_h;
    q.th0 = in0 ? -(1.0f / 255.0f) : -INFINITY;
    q.th1 = in1 ? -(1.0f / 255.0f) : -INFINITY;
    q.T = make_float2(1.f, 1.f);
    q.r = q.g = q.b = make_float2(0.f, 0.f);
    q.blended = 0u;
    const int nbatch = (len + 31) >> 5;
    int b = 0, cnt = 0;  // batches scanned, positions staged (uniform)
    float4 n0, n1;
    // the next up to 32 selected records, one a lane, requested; their number
    auto produce = [&]() -> int {
        for (; cnt < 32 && b < nbatch; ++b) {
            const unsigned m = reinterpret_cast<const unsigned*>(masks + b)[comp];
            if ((m >> lane) & 1u) S.stage[cnt + __popc(m & lt)] = index(32 * b + lane);
            cnt += __popc(m);
        }
        __syncwarp();
        const int n = cnt < 32 ? cnt : 32;
        if (lane < n) {
            const float4* r = base + kRecordFloat4 * int64_t(S.stage[lane]);
            n0 = __ldg(r);
            n1 = __ldg(r + 1);
        }
        const uint32_t rest = lane + 32 < cnt ? S.stage[lane + 32] : 0u;
        __syncwarp();
        if (lane + 32 < cnt) S.stage[lane] = rest;
        cnt -= n;
        return n;
    };
    int n = produce();
    while (n > 0) {
        if (lane < n) {
            float r, g, bl;
            unpack_rgb(n1.z, n1.w, r, g, bl);
            S.geo[lane] = n0;
            S.rg[lane] = make_float4(-r, -r, -g, -g);
            S.bcl[lane] = make_float4(-bl, -bl, n1.x, n1.y);
        } else {  // fills the last run: alpha 0
            S.geo[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
            S.rg[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
            S.bcl[lane] = make_float4(0.f, 0.f, 0.f, -1e30f);
        }
        const int n_next = produce();
        if (COUNT) evals += uint32_t(n) * ((q.th0 > -INFINITY) + (q.th1 > -INFINITY));
        for (int k = 0; k < n; k += kBlendRun) blend_run<COUNT>(q, S, k);
        if (__all_sync(0xffffffffu, q.th0 == -INFINITY && q.th1 == -INFINITY)) break;
        __syncwarp();  // the batch is written again
        n = n_next;
    }
    __syncwarp();
    float* o = Mm + ((int64_t(v) * p.height + row) * p.width + col) * 3;
    const float sum = ((q.r.x + q.r.y) + (q.g.x + q.g.y)) + (q.b.x + q.b.y);
    if (__any_sync(0xffffffffu, sum != sum)) {
        q.blended = patch_by_records<COUNT>(masks, comp, index, len, base, q.x0, q.x1, q.y, in0, in1, o);
        if (COUNT) blended += q.blended;
        return;
    }
    if (in0) {
        o[0] = q.r.x;
        o[1] = q.g.x;
        o[2] = q.b.x;
    }
    if (in1) {
        o[3] = q.r.y;
        o[4] = q.g.y;
        o[5] = q.b.y;
    }
    if (COUNT) blended += q.blended;
}

// A (view, tile) group's 16 x 16 quads, one after another: the masks of the
// quad's batches first, then its patches (those inside the tile and the
// view).  BLOCK: the warps of a block share the batches and then the patches
// (barriers between); otherwise one warp does both.
template <bool COUNT, bool BLOCK, class Index>
__device__ __forceinline__ void composite_quads(const CompositeParams& p, int group, Index index,
                                                int len, const float4* __restrict__ rec,
                                                uint4* masks, PatchBatch& S,
                                                float* __restrict__ Mm, uint32_t& evals,
                                                uint32_t& blended) {
    const int lane = threadIdx.x & 31, warp = BLOCK ? int(threadIdx.x >> 5) : 0;
    const int nwarps = BLOCK ? int(blockDim.x >> 5) : 1;
    const int v = group / p.ntiles;
    const int tile = group - v * p.ntiles;
    const int tx = (tile % p.ntx) * p.tile_w, ty = (tile / p.ntx) * p.tile_h;
    const int xe = min(tx + p.tile_w, p.width), ye = min(ty + p.tile_h, p.height);
    const float4* __restrict__ base = rec + kRecordFloat4 * (int64_t(v) * p.n);
    for (int qy = ty; qy < ye; qy += 2 * kPatch) {
        for (int qx = tx; qx < xe; qx += 2 * kPatch) {
            float x0[2], x1[2], y0[2], y1[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                x0[k] = float(qx + k * kPatch) - p.half_w;
                x1[k] = fmaxf(x0[k], float(min(qx + k * kPatch + kPatch, xe) - 1) - p.half_w);
                y0[k] = float(qy + k * kPatch) - p.half_h;
                y1[k] = fmaxf(y0[k], float(min(qy + k * kPatch + kPatch, ye) - 1) - p.half_h);
            }
            float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f);
            float2 n1 = make_float2(0.f, 0.f);
            auto fetch = [&](int i) {  // a batch ahead
                if (i < len) {
                    const float4* r = base + kRecordFloat4 * int64_t(index(i));
                    n0 = __ldg(r);
                    n1 = __ldg(reinterpret_cast<const float2*>(r + 1));
                }
            };
            fetch(32 * warp + lane);
            for (int b = 32 * warp; b < len; b += 32 * nwarps) {
                const float4 c0 = n0;
                const float2 c1 = n1;
                fetch(b + 32 * nwarps + lane);
                const uint4 m = quad_masks(b + lane < len, c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, x0, x1,
                                           y0, y1);
                if (lane == 0) masks[b >> 5] = m;
            }
            if (BLOCK) __syncthreads();
            else __syncwarp();
            for (int k = warp; k < 4; k += nwarps) {
                const int col0 = qx + (k & 1) * kPatch, row0 = qy + (k >> 1) * kPatch;
                if (col0 >= xe || row0 >= ye) continue;
                composite_patch<COUNT>(p, v, col0, row0, masks, k, index, len, base, S, Mm, evals,
                                       blended);
            }
            if (BLOCK) __syncthreads();  // the masks are written again
        }
    }
}

// The keys are sorted in the space that holds their indices, the masks and
// the batch afterwards.
template <int CAP>
union ViewSmem {
    WarpSort<CAP> s;
    struct {
        uint32_t idx[CAP];
        uint4 masks[CAP / 32];
        PatchBatch batch;
    } c;
};
template <int CAP>
constexpr int view_class_blocks() { return CAP <= 512 ? 8 : 5; }
static_assert(view_class_blocks<512>() * (kWarpsPerBlock * sizeof(ViewSmem<512>) + 1024) <=
                  228 * 1024, "512-key class: 8 blocks");
static_assert(view_class_blocks<1024>() * (kWarpsPerBlock * sizeof(ViewSmem<1024>) + 1024) <=
                  228 * 1024, "1024-key class: 5 blocks");

// Persistent, a warp per (view, tile) list of up to CAP keys: item
// {group, first key, -, keys} i of the class (BACK: from the end of `items`),
// the first by warp id, the rest claimed from *cursor.
template <int CAP, bool BACK, bool COUNT>
__global__ void __launch_bounds__(kWarpsPerBlock * 32, view_class_blocks<CAP>())
composite_views_warp_kernel(CompositeParams p, const int4* __restrict__ items, int64_t n_work,
                            uint32_t n_items, uint32_t* __restrict__ cursor,
                            const unsigned long long* __restrict__ keys,
                            const float4* __restrict__ rec, float* __restrict__ Mm,
                            unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char vsm_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    ViewSmem<CAP>& W = reinterpret_cast<ViewSmem<CAP>*>(vsm_raw)[warp];
    const uint32_t n_warps = gridDim.x * kWarpsPerBlock;
    uint32_t item = blockIdx.x * kWarpsPerBlock + warp;
    uint32_t evals = 0, blended = 0;
    while (item < n_items) {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(cursor, 1u);
        const int4 it = __ldg(items + (BACK ? n_work - 1 - int64_t(item) : int64_t(item)));
        const int len = it.w & 0xFFFF;
        warp_sort<CAP>(keys, uint32_t(it.y), len, W.s);
        for (int base = 0; base < len; base += 32) {  // as narrow_keys
            const int i = base + lane;
            const uint32_t lo = i < len ? uint32_t(W.s.sk[i]) >> 4 : 0u;
            __syncwarp();
            if (i < len) W.c.idx[i] = lo;
            __syncwarp();
        }
        composite_quads<COUNT, false>(p, it.x, [&](int i) { return W.c.idx[i]; }, len, rec,
                                      W.c.masks, W.c.batch, Mm, evals, blended);
        item = n_warps + __shfl_sync(0xffffffffu, c, 0);
    }
    if (COUNT) count_pairs(pairs, evals, blended);
}

// Lists too long for a warp (up to `cap` keys): a block of
// four warps sorts the list together, then its warps share the batches' tests
// and the patches.
template <bool COUNT>
__global__ void __launch_bounds__(kBinnedThreads)
composite_views_block_kernel(CompositeParams p, const int4* __restrict__ block_items, int cap,
                             const unsigned long long* __restrict__ keys,
                             const float4* __restrict__ rec, float* __restrict__ Mm,
                             unsigned long long* __restrict__ pairs) {
    extern __shared__ __align__(16) unsigned char smb[];
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(smb);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smb + 8 * size_t(cap));
    // after the sort: narrowed keys, batches, masks
    PatchBatch* batches = reinterpret_cast<PatchBatch*>(smb + 4 * size_t(cap));
    uint4* masks = reinterpret_cast<uint4*>(batches + kBinnedThreads / 32);
    const int4 it = block_items[blockIdx.x];  // {group, first key, -, keys}
    block_sort(keys, uint32_t(it.y), it.w, cap, sk, cnt);
    const uint32_t* idx = block_narrow(sk, it.w);
    uint32_t evals = 0, blended = 0;
    composite_quads<COUNT, true>(p, it.x, [idx](int i) { return idx[i] >> 4; }, it.w, rec, masks,
                                 batches[threadIdx.x >> 5], Mm, evals, blended);
    if (COUNT) count_pairs(pairs, evals, blended);
}

__global__ void batch_prefix_kernel(const FrameDesc* __restrict__ F, int n_frames,
                                    int64_t* __restrict__ prefix) {
    if (threadIdx.x != 0) return;
    int64_t a = 0, b = 0, c = 0;
    const int stride = n_frames + 1;
    for (int f = 0; f < n_frames; ++f) {
        prefix[f] = a;
        prefix[stride + f] = b;
        prefix[2 * stride + f] = c;
        a += F[f].meta[0];
        b += F[f].meta[4];
        c += F[f].meta[1];
    }
    prefix[n_frames] = a;
    prefix[stride + n_frames] = b;
    prefix[2 * stride + n_frames] = c;
}

// Items of the warp classes: DirectL groups with fewer than 65536 rays and
// at most cap1 keys become self-contained items at the front of `items`,
// those with cap1 < keys <= cap2 at the back (cap2 = 0: no second class); the
// rest become block items {group, first key, gwork index, keys}.
// meta = {n_items1, n_block, max keys, -, n_items2}.  Nothing is written
// when the frame's keys were not all emitted (*total_keys > key_cap, or
// status bit 0 already set).
__global__ void partition_warp_kernel(const int4* __restrict__ gwork, int64_t n_work,
                                      GroupSlices S, uint32_t cap1, uint32_t cap2,
                                      int4* __restrict__ items, int4* __restrict__ block_items,
                                      uint32_t* __restrict__ meta,
                                      const uint32_t* __restrict__ total_keys, uint32_t key_cap,
                                      uint32_t* __restrict__ status, SingleFrame single) {
    after_previous(gwork, S.start, S.start_alt, S.use_alt, S.cursor, total_keys, status);
    if (total_keys && *total_keys > key_cap) {  // keys were not emitted
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(status, 1u);
        return;
    }
    if (status && (*status & 1u)) return;
    const uint32_t* __restrict__ first = S.use_alt && *S.use_alt ? S.start_alt : S.start;
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    // one counter atomic a warp and class: the warp's items of a class stay
    // together and in group order (consecutive items share records in L2)
    auto slot = [&](unsigned am, bool mine, uint32_t* counter) -> uint32_t {
        const unsigned m = __ballot_sync(am, mine);
        uint32_t base = 0u;
        if (m) {
            const int leader = __ffs(m) - 1;
            if (int(threadIdx.x & 31) == leader) base = atomicAdd(counter, uint32_t(__popc(m)));
            base = __shfl_sync(am, base, leader);
        }
        return base + uint32_t(__popc(m & lt));
    };
    for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w < n_work;
         w += int64_t(gridDim.x) * blockDim.x) {
        const unsigned am = __activemask();
        const int4 wi = gwork ? gwork[w] : make_int4(int(w), 0, 0, 0);
        const uint32_t st = first[wi.x];
        const uint32_t len = (S.cursor ? S.cursor[wi.x] : S.start[wi.x + 1]) - st;
        const uint32_t nr = uint32_t(wi.z - wi.y);
        const int4 it = make_int4(wi.x, int(st), wi.y, int((nr << 16) | len));
        const int cls = nr < 65536u && len <= cap1 ? 0 : (nr < 65536u && len <= cap2 ? 1 : 2);
        const uint32_t s0 = slot(am, cls == 0, meta);
        const uint32_t s1 = slot(am, cls == 1, meta + 4);
        const uint32_t s2 = slot(am, cls == 2, meta + 1);
        if (cls == 0)
            items[s0] = it;
        else if (cls == 1)
            items[n_work - 1 - int64_t(s1)] = it;
        else
            block_items[s2] = make_int4(wi.x, int(st), int(w), int(len));
        const uint32_t longest = __reduce_max_sync(am, len);
        if (int(threadIdx.x & 31) == __ffs(am) - 1) atomicMax(meta + 2, longest);
    }
    if (!single.dst) return;
    // the last block to finish sees every block's counts
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(single.done, 1u) == gridDim.x - 1u;
    __syncthreads();
    if (s_last && threadIdx.x == 0) {
        *single.dst = single.fd;
        // one frame: {0, items} per class
        single.prefix[0] = single.prefix[2] = single.prefix[4] = 0;
        single.prefix[1] = int64_t(atomicAdd(meta, 0u));
        single.prefix[3] = int64_t(atomicAdd(meta + 4, 0u));
        single.prefix[5] = int64_t(atomicAdd(meta + 1, 0u));
    }
}

__global__ void partition_kernel(const int4* __restrict__ gwork, int64_t n_work,
                                 const uint32_t* __restrict__ gstart, uint32_t small_cap,
                                 int32_t* __restrict__ small_list, int32_t* __restrict__ large_list,
                                 uint32_t* __restrict__ meta) {
    for (int64_t w = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; w < n_work;
         w += int64_t(gridDim.x) * blockDim.x) {
        const int64_t g = gwork ? gwork[w].x : w;
        const uint32_t len = gstart[g + 1] - gstart[g];
        if (len <= small_cap) small_list[atomicAdd(meta, 1u)] = int32_t(w);
        else large_list[atomicAdd(meta + 1, 1u)] = int32_t(w);
        atomicMax(meta + 2, len);
    }
}

// out[i] = raycol[3 ray_of[i] + i mod 3], a block per kReorderCols x
// kReorderRows patch of subpixels (32 x 32 pixels).  Ray colours in grouped
// order lie together by tile, so a patch gathers from a few tens of kilobytes
// that its block's L1 keeps, and each 32-byte sector is fetched about once; a
// block that took 1024 consecutive subpixels of a row fetched a sector per
// subpixel from L2 (8K panel, 99.5 M subpixels: 1.12 -> 0.28 ms, 4K 0.095 ->
// 0.066 ms).  VEC: four subpixels a thread (16-byte index loads and stores),
// rows of a multiple of four subpixels and 16-byte aligned buffers.
constexpr int kReorderCols = 96, kReorderRows = 32;
template <bool VEC>
__global__ void __launch_bounds__(256)
reorder_kernel(const uint32_t* __restrict__ ray_of, const float* __restrict__ raycol, int32_t cols,
               int32_t rows, int32_t patches_x, float* __restrict__ out,
               const uint32_t* __restrict__ skip) {
    if (skip && *skip) return;  // the frame was not composited
    constexpr int V = VEC ? 4 : 1, W = kReorderCols / V;
    const int py = int(blockIdx.x) / patches_x, px = int(blockIdx.x) - py * patches_x;
    const int x0 = px * kReorderCols, y0 = py * kReorderRows;
#pragma unroll 3
    for (int t = threadIdx.x; t < W * kReorderRows; t += 256) {
        const int y = y0 + t / W, lx = (t % W) * V, x = x0 + lx;
        if (y >= rows || x >= cols) continue;
        const int64_t i = int64_t(y) * cols + x;
        const uint32_t k = uint32_t(lx) % 3u;  // channel of the first: patches start at 0
        if (VEC) {
            const uint4 r = *reinterpret_cast<const uint4*>(ray_of + i);
            const uint32_t k1 = k == 2u ? 0u : k + 1u, k2 = k == 0u ? 2u : k - 1u;
            float4 o;
            o.x = __ldg(raycol + 3 * int64_t(r.x) + k);
            o.y = __ldg(raycol + 3 * int64_t(r.y) + k1);
            o.z = __ldg(raycol + 3 * int64_t(r.z) + k2);
            o.w = __ldg(raycol + 3 * int64_t(r.w) + k);
            *reinterpret_cast<float4*>(out + i) = o;
        } else {
            out[i] = __ldg(raycol + 3 * int64_t(ray_of[i]) + k);
        }
    }
}

// The assembly kernels below take kGather subpixels a thread, so that as many
// gathers are in flight (one a thread, behind a 64-bit division, kept the
// memory system at a third: 4K interweave 0.41 ms, upsampling 0.22 ms).
// Indices inside one view or panel are 32-bit (16384^2 x 3 < 2^32).
constexpr int kGather = 4;

// M_e[x, y, k] = M_m[V(x, 3y + k), x, y, k] (Alg. 1, native resolution).
__global__ void interweave_kernel(int32_t w, int32_t h, const uint16_t* __restrict__ V,
                                  const float* __restrict__ Mm, float* __restrict__ out) {
    const uint32_t total = 3u * uint32_t(w) * uint32_t(h);  // = a view's values
    const uint32_t i0 = blockIdx.x * (256u * kGather) + threadIdx.x;
    float v[kGather];
#pragma unroll
    for (int j = 0; j < kGather; ++j) {
        const uint32_t i = i0 + 256u * j;
        v[j] = i < total ? __ldg(Mm + int64_t(V[i]) * total + i) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < kGather; ++j)
        if (i0 + 256u * j < total) out[i0 + 256u * j] = v[j];
}

// The paper's "HR w SR" assembly: subpixel (x, y, k) takes channel k of view
// V(x, 3y + k) at its repurposed source pixel src = (x' << 16 | y') (Sec. 5)
// rather than at (x, y); a source outside the panel (never produced by the
// repurposing) reads the subpixel's own pixel.
__global__ void repurposed_interweave_kernel(int32_t w, int32_t h, const uint16_t* __restrict__ V,
                                             const uint32_t* __restrict__ src,
                                             const float* __restrict__ Mm,
                                             float* __restrict__ out) {
    const uint32_t total = 3u * uint32_t(w) * uint32_t(h);
    const uint32_t i0 = blockIdx.x * (256u * kGather) + threadIdx.x;
    float v[kGather];
#pragma unroll
    for (int j = 0; j < kGather; ++j) {
        const uint32_t i = i0 + 256u * j;
        v[j] = 0.f;
        if (i < total) {
            const uint32_t sp = src[i], sr = sp >> 16, sc = sp & 0xFFFFu, own = i / 3u;
            const uint32_t p = (sr < uint32_t(h) && sc < uint32_t(w)) ? sr * uint32_t(w) + sc : own;
            v[j] = __ldg(Mm + int64_t(V[i]) * total + 3u * p + (i - 3u * own));
        }
    }
#pragma unroll
    for (int j = 0; j < kGather; ++j)
        if (i0 + 256u * j < total) out[i0 + 256u * j] = v[j];
}

// Alg. 1 with views rendered at rw x rh and upsampled while interweaving:
// subpixel (x, y, k) takes channel k of view V(x, 3y + k) bilinearly at
// column y rw / w, row x rh / h of that view (pixel (r, c) of a view samples
// its image point (c, r) about the principal point, so the panel's and the
// view's pixel grids share the corner), clamped at the border.  Positions
// are split into integer and fractional parts exactly (16384^2 < 2^32).
__global__ void resize_interweave_kernel(int32_t w, int32_t h, int32_t rw, int32_t rh,
                                         const uint16_t* __restrict__ V,
                                         const float* __restrict__ Mm, float* __restrict__ out) {
    const uint32_t total = 3u * uint32_t(w) * uint32_t(h);
    const uint32_t i0 = blockIdx.x * (256u * kGather) + threadIdx.x;
    float v[kGather];
#pragma unroll
    for (int j = 0; j < kGather; ++j) {
        const uint32_t i = i0 + 256u * j;
        v[j] = 0.f;
        if (i < total) {
            const uint32_t p = i / 3u, k = i - 3u * p, row = p / uint32_t(w), col = p - row * uint32_t(w);
            const uint32_t nx = col * uint32_t(rw), ny = row * uint32_t(rh);
            const uint32_t x0 = nx / uint32_t(w), y0 = ny / uint32_t(h);
            const float fx = float(nx - x0 * uint32_t(w)) / float(w);
            const float fy = float(ny - y0 * uint32_t(h)) / float(h);
            const uint32_t x1 = min(x0 + 1u, uint32_t(rw) - 1u), y1 = min(y0 + 1u, uint32_t(rh) - 1u);
            const float* img = Mm + int64_t(V[i]) * rh * rw * 3 + k;
            const float a = __ldg(img + 3u * (y0 * uint32_t(rw) + x0));
            const float b = __ldg(img + 3u * (y0 * uint32_t(rw) + x1));
            const float c = __ldg(img + 3u * (y1 * uint32_t(rw) + x0));
            const float d = __ldg(img + 3u * (y1 * uint32_t(rw) + x1));
            v[j] = (1.f - fy) * ((1.f - fx) * a + fx * b) + fy * ((1.f - fx) * c + fx * d);
        }
    }
#pragma unroll
    for (int j = 0; j < kGather; ++j)
        if (i0 + 256u * j < total) out[i0 + 256u * j] = v[j];
}

}  // namespace

cudaError_t launch_composite_rays(const CompositeParams& p, const int4* work, int64_t n_work,
                                  const int2* grouped, const uint2* ranges, const uint32_t* vals,
                                  const float4* rec, float* raycol, unsigned long long* pairs,
                                  cudaStream_t s) {
    if (n_work <= 0) return cudaSuccess;
    composite_rays_kernel<<<unsigned(n_work), kRayThreads, 0, s>>>(p, work, grouped, ranges, vals,
                                                                   rec, raycol, pairs);
    return cudaGetLastError();
}

cudaError_t launch_composite_full(const CompositeParams& p, int32_t nv, const uint2* ranges,
                                  const uint32_t* vals, const float4* rec, float* Mm,
                                  unsigned long long* pairs, cudaStream_t s) {
    const int nthr = p.tile_w * p.tile_h;
    const size_t smem = size_t(nthr) * 3 * sizeof(float4);
    const int64_t blocks = int64_t(nv) * p.ntiles;
    composite_full_kernel<<<unsigned(blocks), nthr, smem, s>>>(p, ranges, vals, rec, Mm, pairs);
    return cudaGetLastError();
}

size_t block_smem_bytes(int cap) {
    // the sort's keys and counters, then the narrowed keys and the pipes
    return std::max(block_sort_bytes(cap), 4 * size_t(cap) + (kBinnedThreads / 32) * sizeof(QuadPipe));
}

size_t binned_smem_bytes(int cap, int nthr) {
    return block_sort_bytes(cap) + size_t(nthr) * 3 * sizeof(float4) + size_t(nthr / 32) * 64 * sizeof(int);
}

cudaError_t launch_composite_rays_binned(const CompositeParams& p, const int4* gwork,
                                         const int32_t* list, int64_t n_list, int cap,
                                         const int2* grouped, const uint32_t* gstart,
                                         const unsigned long long* keys, const float4* rec,
                                         float* raycol, unsigned long long* pairs, int transposed,
                                         cudaStream_t s) {
    if (n_list <= 0) return cudaSuccess;
    const int nthr = kBinnedThreads;
    const size_t smem = binned_smem_bytes(cap, nthr);
    auto go = [&](auto kernel) -> cudaError_t {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             int(smem));
        if (e != cudaSuccess) return e;
        kernel<<<unsigned(n_list), nthr, smem, s>>>(p, gwork, list, cap, grouped, gstart, keys, rec,
                                                    raycol, pairs);
        return cudaGetLastError();
    };
    return transposed ? go(composite_rays_binned_kernel<true>) : go(composite_rays_binned_kernel<false>);
}

cudaError_t launch_composite_full_binned(const CompositeParams& p, const int32_t* list,
                                         int64_t n_list, int cap, const uint32_t* gstart,
                                         const unsigned long long* keys, const float4* rec,
                                         float* Mm, unsigned long long* pairs, cudaStream_t s) {
    if (n_list <= 0) return cudaSuccess;
    const int nthr = p.tile_w * p.tile_h;
    const size_t smem = binned_smem_bytes(cap, nthr);
    cudaError_t e = cudaFuncSetAttribute(composite_full_binned_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    composite_full_binned_kernel<<<unsigned(n_list), nthr, smem, s>>>(p, list, cap, gstart, keys, rec,
                                                                      Mm, pairs);
    return cudaGetLastError();
}

size_t views_block_smem_bytes(int cap) {
    return std::max(block_sort_bytes(cap), 4 * size_t(cap) +
                                               (kBinnedThreads / 32) * sizeof(PatchBatch) +
                                               size_t(cap / 32) * sizeof(uint4));
}

namespace {
template <int CAP, bool BACK, bool COUNT>
cudaError_t launch_views_warp(const CompositeParams& p, const int4* items, int64_t n_work, int64_t n,
                              uint32_t* cursor, const unsigned long long* keys, const float4* rec,
                              float* Mm, unsigned long long* pairs, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const auto kernel = composite_views_warp_kernel<CAP, BACK, COUNT>;
    const size_t smem = kWarpsPerBlock * sizeof(ViewSmem<CAP>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kWarpsPerBlock * 32, smem);
    if (e != cudaSuccess) return e;
    const int64_t need = (n + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int64_t fit = int64_t(num_sms()) * (per_sm > 0 ? per_sm : 1);
    kernel<<<unsigned(need < fit ? need : fit), kWarpsPerBlock * 32, smem, s>>>(
        p, items, n_work, uint32_t(n), cursor, keys, rec, Mm, pairs);
    return cudaGetLastError();
}

template <bool COUNT>
cudaError_t launch_views(const CompositeParams& p, const int4* items, const int4* block_items,
                         int64_t n_work, const int64_t n[3], int block_cap, uint32_t* const cursor[2],
                         const unsigned long long* keys, const float4* rec, float* Mm,
                         unsigned long long* pairs, cudaStream_t s) {
    // one after another on the one stream, the longest lists first
    if (n[2] > 0) {
        const size_t smem = views_block_smem_bytes(block_cap);
        cudaError_t e = cudaFuncSetAttribute(composite_views_block_kernel<COUNT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
        composite_views_block_kernel<COUNT><<<unsigned(n[2]), kBinnedThreads, smem, s>>>(
            p, block_items, block_cap, keys, rec, Mm, pairs);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const cudaError_t e = launch_views_warp<1024, true, COUNT>(p, items, n_work, n[1], cursor[1], keys,
                                                               rec, Mm, pairs, s);
    if (e != cudaSuccess) return e;
    return launch_views_warp<512, false, COUNT>(p, items, n_work, n[0], cursor[0], keys, rec, Mm,
                                                pairs, s);
}
}  // namespace

cudaError_t launch_composite_views(const CompositeParams& p, const int4* items,
                                   const int4* block_items, int64_t n_work, const int64_t n[3],
                                   int block_cap, uint32_t* const cursor[2],
                                   const unsigned long long* keys, const float4* rec, float* Mm,
                                   unsigned long long* pairs, cudaStream_t s) {
    return pairs ? launch_views<true>(p, items, block_items, n_work, n, block_cap, cursor, keys, rec,
                                      Mm, pairs, s)
                 : launch_views<false>(p, items, block_items, n_work, n, block_cap, cursor, keys, rec,
                                       Mm, pairs, s);
}

namespace {
template <class K, class Extra>
cudaError_t launch_persistent(K kernel, int threads, size_t smem, int64_t max_blocks,
                              const FrameDesc* frames, const int64_t* prefix, int32_t n_frames,
                              Extra extra, uint32_t* cursor, unsigned long long* pairs, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    int64_t blocks = int64_t(num_sms()) * (per_sm > 0 ? per_sm : 1);
    if (blocks > max_blocks) blocks = max_blocks;
    kernel<<<unsigned(blocks), threads, smem, s>>>(frames, prefix, n_frames, extra, cursor, pairs);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_batch_prefix(const FrameDesc* frames, int32_t n_frames, int64_t* prefix,
                                cudaStream_t s) {
    batch_prefix_kernel<<<1, 32, 0, s>>>(frames, n_frames, prefix);
    return cudaGetLastError();
}

cudaError_t launch_composite_rays_warp(int cap, int cls, const FrameDesc* frames,
                                       const int64_t* prefix, int32_t n_frames, int64_t max_items,
                                       uint32_t* cursor, unsigned long long* pairs, cudaStream_t s) {
    if (max_items <= 0 || n_frames <= 0) return cudaSuccess;
    const int64_t need = (max_items + kWarpsPerBlock - 1) / kWarpsPerBlock;
    const int64_t* pc = prefix + int64_t(cls) * (n_frames + 1);
    const int t = kWarpsPerBlock * 32;
    const size_t s1 = kWarpsPerBlock * sizeof(WarpSmem<512>), s2 = kWarpsPerBlock * sizeof(WarpSmem<1024>);
    if (cap == 1024)
        return pairs ? launch_persistent(composite_rays_warp_kernel<1024, true>, t, s2, need, frames,
                                         pc, n_frames, cls, cursor, pairs, s)
                     : launch_persistent(composite_rays_warp_kernel<1024, false>, t, s2, need, frames,
                                         pc, n_frames, cls, cursor, pairs, s);
    return pairs ? launch_persistent(composite_rays_warp_kernel<512, true>, t, s1, need, frames, pc,
                                     n_frames, cls, cursor, pairs, s)
                 : launch_persistent(composite_rays_warp_kernel<512, false>, t, s1, need, frames, pc,
                                     n_frames, cls, cursor, pairs, s);
}

cudaError_t launch_composite_rays_block(int block_cap, int longest, const FrameDesc* frames,
                                        const int64_t* prefix, int32_t n_frames, int64_t max_items,
                                        uint32_t* cursor, unsigned long long* pairs, cudaStream_t s) {
    if (max_items <= 0 || n_frames <= 0) return cudaSuccess;
    const size_t smem = block_smem_bytes(block_cap);
    return launch_persistent(composite_rays_block_kernel, kBinnedThreads, smem, max_items, frames,
                             prefix + 2 * (n_frames + 1), n_frames,
                             make_int2(block_cap, std::max(block_cap, longest)), cursor, pairs, s);
}

cudaError_t launch_composite_rays_long(int block_cap, int longest, const FrameDesc* frame,
                                       const int64_t* prefix, unsigned long long* pairs, cudaStream_t s) {
    if (longest <= block_cap) return cudaSuccess;
    composite_rays_long_kernel<<<unsigned(num_sms() * 4), kBinnedThreads, 0, s>>>(
        frame, prefix + 4, make_int2(block_cap, longest), pairs);
    return cudaGetLastError();
}

cudaError_t launch_partition_warp(const int4* gwork, int64_t n_work, const GroupSlices& slices,
                                  uint32_t cap1, uint32_t cap2, int4* items, int4* block_items,
                                  uint32_t* meta, const uint32_t* total_keys, uint32_t key_cap,
                                  uint32_t* status, const SingleFrame& single, cudaStream_t s) {
    if (n_work <= 0) return cudaSuccess;
    int64_t grid = (n_work + 255) / 256;
    const int64_t lim = int64_t(num_sms()) * 16;
    if (grid > lim) grid = lim;
    return launch_after(partition_warp_kernel, unsigned(grid), 256, 0, s, gwork, n_work, slices, cap1, cap2,
                        items, block_items, meta, total_keys, key_cap, status, single);
}

cudaError_t launch_partition(const int4* gwork, int64_t n_work, const uint32_t* gstart,
                             uint32_t small_cap, int32_t* small_list, int32_t* large_list,
                             uint32_t* meta, cudaStream_t s) {
    if (n_work <= 0) return cudaSuccess;
    int64_t grid = (n_work + 255) / 256;
    const int64_t cap = int64_t(num_sms()) * 16;
    if (grid > cap) grid = cap;
    partition_kernel<<<unsigned(grid), 256, 0, s>>>(gwork, n_work, gstart, small_cap, small_list,
                                                    large_list, meta);
    return cudaGetLastError();
}

cudaError_t launch_reorder(const uint32_t* ray_of, const float* raycol, int32_t w, int32_t h,
                           float* out, const uint32_t* skip, cudaStream_t s) {
    const int32_t cols = 3 * w;
    const int64_t px = (cols + kReorderCols - 1) / kReorderCols, py = (h + kReorderRows - 1) / kReorderRows;
    const bool vec = cols % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0 &&
                     (reinterpret_cast<uintptr_t>(ray_of) & 15u) == 0;
    if (vec)
        reorder_kernel<true><<<unsigned(px * py), 256, 0, s>>>(ray_of, raycol, cols, h, int32_t(px), out,
                                                               skip);
    else
        reorder_kernel<false><<<unsigned(px * py), 256, 0, s>>>(ray_of, raycol, cols, h, int32_t(px),
                                                                out, skip);
    return cudaGetLastError();
}

static unsigned gather_grid(int32_t w, int32_t h) {
    const int64_t n = 3 * int64_t(w) * h;
    return unsigned((n + 256 * kGather - 1) / (256 * kGather));
}

cudaError_t launch_resize_interweave(int32_t w, int32_t h, int32_t rw, int32_t rh,
                                     const uint16_t* V, const float* Mm, float* out,
                                     cudaStream_t s) {
    resize_interweave_kernel<<<gather_grid(w, h), 256, 0, s>>>(w, h, rw, rh, V, Mm, out);
    return cudaGetLastError();
}

cudaError_t launch_repurposed_interweave(int32_t w, int32_t h, const uint16_t* V, const uint32_t* src,
                                        const float* Mm, float* out, cudaStream_t s) {
    repurposed_interweave_kernel<<<gather_grid(w, h), 256, 0, s>>>(w, h, V, src, Mm, out);
    return cudaGetLastError();
}

cudaError_t launch_interweave(int32_t w, int32_t h, const uint16_t* V, const float* Mm, float* out,
                              cudaStream_t s) {
    interweave_kernel<<<gather_grid(w, h), 256, 0, s>>>(w, h, V, Mm, out);
    return cudaGetLastError();
}

}  // namespace dl
