// Offline display tables (Sec. 4 step (1)): the view-index map (Sec. 3.1,
// Eqs. (1)-(3)), subpixel repurposing (Sec. 5, Alg. 2) and the R-first ray
// table (Sec. 5, last part).  Integer arithmetic throughout, so the tables
// are exact.
#include <algorithm>
#include <mutex>

#include "../../include/directl.h"
#include "dl_internal.cuh"

namespace dl {
namespace {

constexpr int64_t kQ32 = int64_t(1) << 32;

__host__ __device__ __forceinline__ int64_t floor_div(int64_t a, int64_t b) {
    int64_t q = a / b;
    return (a % b != 0 && ((a < 0) != (b < 0))) ? q - 1 : q;
}
// d_offset (Eq. (1)) of subpixel column s in row x, Q32.
__host__ __device__ __forceinline__ int64_t d_offset(const DisplayQ& q, int64_t x, int64_t s) {
    return s * kQ32 + x * q.t3q - q.kq;
}

// ------------------------------------------------------------------ a1 ---
// v = floor(N_v (d mod L_x) / L_x), Eqs. (2)-(3), mod taken into [0, L_x).
// One thread writes 8 consecutive views (one 16-byte store).  N_v x_offset =
// v L_x + rem is kept as (v, rem): one subpixel on, N_v 2^32 = step_v L_x +
// step_rem is added, and a view past N_v wraps by N_v (x_offset by L_x), so
// only a thread's first subpixel and a row's first are divided out (with a
// division a subpixel the kernel was bound by it: 0.171 ms at 4K).
__global__ void view_map_kernel(DisplayQ q, int64_t step_v, int64_t step_rem,
                                uint16_t* __restrict__ V) {
    const int64_t S = 3 * int64_t(q.w);
    const int64_t total = S * q.h;
    const int64_t n8 = (total + 7) / 8;
    for (int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; t < n8;
         t += int64_t(gridDim.x) * blockDim.x) {
        const int64_t i0 = t * 8;
        int64_t x = i0 / S, s = i0 - x * S;
        int64_t v = 0, rem = 0;
        auto divide = [&]() {
            int64_t xo = d_offset(q, x, s) % q.lq;
            if (xo < 0) xo += q.lq;
            const int64_t n = int64_t(q.nv) * xo;
            v = n / q.lq;
            rem = n - v * q.lq;
        };
        divide();
        uint16_t out[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            out[j] = uint16_t(v);
            if (++s == S) {  // a new row restarts at s = 0
                s = 0;
                ++x;
                divide();
            } else {
                v += step_v;
                rem += step_rem;
                if (rem >= q.lq) {
                    rem -= q.lq;
                    ++v;
                }
                if (v >= q.nv) v -= q.nv;  // step_v < N_v: at most one wrap
            }
        }
        if (i0 + 8 <= total && ((reinterpret_cast<uintptr_t>(V + i0) & 15) == 0)) {
            uint4 pk;
            pk.x = out[0] | (uint32_t(out[1]) << 16);
            pk.y = out[2] | (uint32_t(out[3]) << 16);
            pk.z = out[4] | (uint32_t(out[5]) << 16);
            pk.w = out[6] | (uint32_t(out[7]) << 16);
            *reinterpret_cast<uint4*>(V + i0) = pk;
        } else {
            for (int j = 0; j < 8 && i0 + j < total; ++j) V[i0 + j] = out[j];
        }
    }
}

// ------------------------------------------------------------------ a2 ---
__device__ __forceinline__ uint32_t pack_px(int64_t x, int64_t y) {
    return (uint32_t(x) << 16) | uint32_t(y);
}

// ceil(x / 2^32); |x| < 2^54 here (panels end near 2^53), so it fits 32 bits
__device__ __forceinline__ int32_t ceil_q32(int64_t x) { return int32_t((x + (kQ32 - 1)) >> 32); }

// Alg. 2, four lanes per (area, view).  Areas are independent (Sec. 5), and
// inside an area so are the views: a chain (Eqs. (11)-(14)) starts at an
// empty subpixel of view v_i, parks and looks up idle channels in
// B_rgb(v_i, .) only, which is cleared when it ends, and fills only subpixels
// that show v_i.  So each view's chains run alone, in row-major order of
// their starts, and nothing they read is written by another group of lanes.
//
// Which subpixels of a row show view v follows from the map itself: those of
// grating unit u lie at d in [u L_x + vlo, u L_x + vhi) with vlo = ceil(v L_x
// / N_v), vhi = ceil((v + 1) L_x / N_v) in Q32 (v = floor(N_v x_offset / L_x)
// exactly then), i.e. at s from ceil((u L_x + vlo - base) / 2^32) on, base =
// x 3 tan - K.  Neither the walk nor the search reads V.
//
// A chain ends when the subpixel that the search finds (the first one in scan
// order: rows ascending, columns from y outward, channels 0..2, that shows v
// and whose channel has an idle subpixel parked) is outside the area or
// already filled.
//
// Bound by the latency of a chain's dependent steps, so the groups are many
// (35 thousand at 4K: 783 areas x 45 views, about 780 subpixels each) and take
// four rows at a time, of the walk as of the search.  The warp's eight groups
// advance together, one such look each an iteration, whatever the others do.
// 4.0 ms at 4K (6.1 with two lanes a group, 4.7 with eight).  As nested loops
// a thread per (area, view) took 30.8 ms, every lane waiting for each lane's
// chains, and a warp per area that took the views' chains in turn and
// searched V 32 candidates at a time 48.6 ms.
constexpr int kChainLanes = 4;

__global__ void __launch_bounds__(32)
repurpose_kernel(DisplayQ q, uint32_t* src) {
    const int64_t lq = q.lq;
    const int64_t far = 8 * lq;  // from here on a division is cheaper than steps
    const int lane = threadIdx.x, sub = lane % kChainLanes;
    const unsigned group = ((1u << kChainLanes) - 1u) << (lane - sub);
    const int32_t S = 3 * q.w, h = q.h;
    const int64_t most_u = (int64_t(1) << 53) / lq + 2;  // past every panel's units
    const int64_t total = int64_t(q.n_areas) * q.nv;
    constexpr int kGroups = 32 / kChainLanes;
    for (int64_t id0 = int64_t(blockIdx.x) * kGroups; id0 < total; id0 += int64_t(gridDim.x) * kGroups) {
        const int64_t id = id0 + lane / kChainLanes;
        bool done = id >= total;
        const int64_t a = q.area_min + (done ? 0 : id / q.nv), v = done ? 0 : id % q.nv;
        const int64_t vlo = (v * lq + q.nv - 1) / q.nv, vhi = ((v + 1) * lq + q.nv - 1) / q.nv;
        // the area's d range
        const int64_t u_lo = max(a * q.pw, -most_u) * lq, u_hi = min((a + 1) * q.pw, most_u) * lq;
        const int64_t span = vhi - vlo;
        int64_t wu = u_lo;            // unit of the lane's row of the search, at its first column
        int32_t x = 0;                // the walk's first row
        bool chain = false, fresh = false;  // a chain is running; it stands at a new subpixel
        int32_t cx = 0, cs = 0;       // the chain's subpixel
        uint32_t B0 = kEmpty, B1 = kEmpty, B2 = kEmpty;  // B_rgb(v_i, .)
        int32_t r_cur = 0, r_hi = 0, w0 = 0, w1 = 0;     // rows and subpixel columns left to search
        while (!__all_sync(0xffffffffu, done)) {
            // the walk: the first empty subpixel of view v of each lane's row
            int32_t at = -1;
            if (!done && !chain && x + sub < h) {
                const int64_t base = int64_t(x + sub) * q.t3q - q.kq, off = vlo - base;
                int64_t u = u_lo;  // or, in wide areas, the row's first unit
                if (base - u >= far) u += floor_div(base - u, lq) * lq;
                for (; u < u_hi && at < 0; u += lq) {
                    const int32_t s0 = ceil_q32(u + off), s1 = min(ceil_q32(u + off + span), S);
                    if (s0 >= S) break;
                    for (int32_t s = max(s0, 0); s < s1; ++s)
                        if (src[int64_t(x + sub) * S + s] == kEmpty) {
                            at = s;
                            break;
                        }
                }
            }
            const unsigned hit = __ballot_sync(0xffffffffu, at >= 0) & group;
            const int32_t start = __shfl_sync(0xffffffffu, at, hit ? __ffs(hit) - 1 : lane);
            if (!done && !chain) {
                if (hit) {
                    x += (__ffs(hit) - 1) % kChainLanes;
                    cx = x;
                    cs = start;
                    B0 = B1 = B2 = kEmpty;
                    chain = fresh = true;
                } else {
                    x += kChainLanes;
                    done = x >= h;
                }
            }
            if (fresh) {
                fresh = false;
                const int32_t cy = cs / 3, ck = cs - 3 * cy;
                const uint32_t Bk = ck == 0 ? B0 : (ck == 1 ? B1 : B2);
                const bool idle = Bk != kEmpty;
                const uint32_t own = pack_px(cx, cy);
                if (sub == 0) src[int64_t(cx) * S + cs] = idle ? Bk : own;  // Eq. (13) / (11)
                // Eq. (12); used channels are cleared
                B0 = ck == 0 ? kEmpty : (idle ? B0 : own);
                B1 = ck == 1 ? kEmpty : (idle ? B1 : own);
                B2 = ck == 2 ? kEmpty : (idle ? B2 : own);
                // Eq. (14): rows [x + 2, x + win_dx], columns from y outward
                r_cur = min(cx + 2, h - 1);
                r_hi = min(cx + q.win_dx, h - 1);
                w0 = 3 * (q.slant_neg ? cy : max(cy - q.win_dy, 0));
                w1 = 3 * (q.slant_neg ? min(cy + q.win_dy, q.w - 1) : cy) + 2;
            }
            // the search: the first candidate of each lane's row
            int32_t found = -1;
            bool inside = false;  // in the chain's area
            if (chain && r_cur + sub <= r_hi) {
                const int64_t rb = int64_t(r_cur + sub) * q.t3q - q.kq, off = vlo - rb;
                // the first unit whose subpixels of view v end past column w0
                const int64_t t0 = int64_t(w0) * kQ32 + rb - wu;
                if (t0 < -far || t0 >= far) wu += floor_div(t0, lq) * lq;
                while (ceil_q32(wu + off + span) > w0) wu -= lq;
                do wu += lq;
                while (ceil_q32(wu + off + span) <= w0);
                int32_t fcol = -1;
                for (int64_t t = wu;; t += lq) {
                    const int32_t a0 = ceil_q32(t + off);
                    if (a0 > w1) break;
                    const int32_t a1 = min(ceil_q32(t + off + span) - 1, w1);
                    for (int32_t j = max(a0, w0); j <= a1; ++j) {
                        const int32_t c = j / 3, ch = j - 3 * c;
                        if ((ch == 0 ? B0 : (ch == 1 ? B1 : B2)) == kEmpty) continue;
                        // the nearest column first, then the lowest channel
                        if (found < 0 || (!q.slant_neg && c > fcol)) {
                            found = j;
                            fcol = c;
                            inside = t >= u_lo && t < u_hi;
                        }
                    }
                    if (q.slant_neg && found >= 0) break;
                }
            }
            const unsigned fb = __ballot_sync(0xffffffffu, found >= 0) & group;
            const unsigned ib = __ballot_sync(0xffffffffu, inside) & group;
            const int32_t next = __shfl_sync(0xffffffffu, found, fb ? __ffs(fb) - 1 : lane);
            if (chain) {
                if (fb) {
                    // while condition of Alg. 2: inside the area and still empty
                    const int32_t fr = r_cur + (__ffs(fb) - 1) % kChainLanes;
                    chain = ((ib >> (__ffs(fb) - 1)) & 1u) && src[int64_t(fr) * S + next] == kEmpty;
                    fresh = chain;
                    cx = fr;
                    cs = next;
                } else {
                    r_cur += kChainLanes;
                    chain = r_cur <= r_hi;  // no position left for view v_i
                }
            }
            __syncwarp();  // the group's lanes read what its first lane wrote
        }
    }
}

// Alg. 2, a warp per area, which takes the area's chains in turn and searches V
// 32 candidates at a time.  It does not depend on how many views an area shows
// nor on how many units a window holds, and is the better one where the
// kernel above has few groups of lanes to run or many units to look at:
//  - a pitch below a subpixel.  Panel set-up at 1080p with 45 views and an
//    irregular slant: pitch 0.31 6.2 ms (50.8 with the kernel above), 0.52 5.2
//    (14.6), 0.71 6.9 (12.0), 0.96 9.3 (10.2); 480 x 270 at 0.01 1.8 (662);
//  - a pitch below 3.5 subpixels that, with the slant, repeats after a few
//    subpixels, so that few of the views are shown.  Slant 1/6: pitch 1.05 45 ms
//    (81), 1.5 26 (101), 2 21 (45), 3 16.0 (16.3); 200 views, 3 174 (226); slant
//    1/3, 3 16.0 (20.7).  From 3.5 on the kernel above wins (4: 8.2 against
//    18.6, slant 1/3 13.3 against 18.5), as it does where most views are shown
//    (1.37: 7.2 against 13.9, 3.17: 4.3 against 19.2).
__global__ void __launch_bounds__(128)
repurpose_area_kernel(DisplayQ q, const uint16_t* __restrict__ V, uint32_t* src) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5;
    if (warp >= q.n_areas) return;
    const int64_t a = q.area_min + warp;
    const int64_t S = 3 * int64_t(q.w);
    const int64_t most_u = (int64_t(1) << 53) / q.lq + 2;  // past every panel's units
    // the area covers d in [lo_d, hi_d)
    const int64_t lo_d = max(a * q.pw, -most_u) * q.lq, hi_d = min((a + 1) * q.pw, most_u) * q.lq;
    for (int64_t x = 0; x < q.h; ++x) {
        const int64_t base = x * q.t3q - q.kq;
        const int64_t s_lo = max(ceil_q32(lo_d - base), 0), s_hi = min(int64_t(ceil_q32(hi_d - base)), S);
        for (int64_t s = s_lo; s < s_hi; ++s) {
            int64_t ci = x * S + s;
            uint32_t cur = 0;
            if (lane == 0) cur = src[ci];
            cur = __shfl_sync(0xffffffffu, cur, 0);
            if (cur != kEmpty) continue;
            const uint16_t vi = V[ci];
            uint32_t B0 = kEmpty, B1 = kEmpty, B2 = kEmpty;  // B_rgb(v_i, .)
            int64_t cx = x, cy = s / 3;
            int ck = int(s % 3);
            while (true) {
                const uint32_t Bk = ck == 0 ? B0 : (ck == 1 ? B1 : B2);
                const bool idle = Bk != kEmpty;
                const uint32_t own = pack_px(cx, cy);
                if (lane == 0) src[ci] = idle ? Bk : own;  // Eq. (13) / (11)
                // Eq. (12); used channels are cleared
                B0 = ck == 0 ? kEmpty : (idle ? B0 : own);
                B1 = ck == 1 ? kEmpty : (idle ? B1 : own);
                B2 = ck == 2 ? kEmpty : (idle ? B2 : own);
                // Eq. (14): rows [x + 2, x + win_dx], columns from y outward
                const int64_t r0 = min(cx + 2, int64_t(q.h) - 1), r1 = min(cx + q.win_dx, int64_t(q.h) - 1);
                const int64_t step = q.slant_neg ? 1 : -1;
                const int64_t last = q.slant_neg ? min(cy + q.win_dy, int64_t(q.w) - 1)
                                                 : max(cy - q.win_dy, int64_t(0));
                const int64_t row = 3 * ((last - cy) * step + 1);  // candidates a row
                const int64_t ncand = r1 >= r0 ? (r1 - r0 + 1) * row : 0;
                int64_t found = -1;
                for (int64_t b = 0; b < ncand; b += 32) {
                    const int64_t j = b + lane;
                    bool match = false;
                    if (j < ncand) {
                        const int64_t r = j / row, rem = j - r * row;
                        const int ch = int(rem % 3);
                        match = (ch == 0 ? B0 : (ch == 1 ? B1 : B2)) != kEmpty &&
                                V[(r0 + r) * S + 3 * (cy + step * (rem / 3)) + ch] == vi;
                    }
                    const unsigned hit = __ballot_sync(0xffffffffu, match);
                    if (hit) {
                        found = b + (__ffs(hit) - 1);
                        break;
                    }
                }
                if (found < 0) break;  // no position left for view v_i
                const int64_t r = found / row, rem = found - r * row;
                cx = r0 + r;
                cy += step * (rem / 3);
                ck = int(rem % 3);
                ci = cx * S + 3 * cy + ck;
                // while condition of Alg. 2: inside the area and still empty
                const int64_t d = d_offset(q, cx, 3 * cy + ck);
                uint32_t next = 0;
                if (lane == 0) next = src[ci];
                next = __shfl_sync(0xffffffffu, next, 0);
                if (d < lo_d || d >= hi_d || next != kEmpty) break;
            }
        }
    }
}

// Whether x_offset takes few values (so few of the views are shown), by 64 runs
// of 64 subpixels spread over the panel: fewer than half of four bins a view
// (finer than the views, as values that lie on the border of two views show
// both).
bool few_offsets(const DisplayQ& q) {
    constexpr int kRuns = 64, kRun = 64;
    const int64_t S = 3 * int64_t(q.w), bins = std::min(4 * q.nv, kRuns * kRun / 4);
    bool seen[kRuns * kRun / 4] = {};
    int64_t filled = 0;
    for (int i = 0; i < kRuns; ++i) {
        const int64_t x = int64_t(q.h) * i / kRuns, s0 = (S * i / kRuns) * 7;
        for (int j = 0; j < kRun; ++j) {
            const int64_t d = d_offset(q, x, (s0 + j) % S);
            const int64_t xo = d - floor_div(d, q.lq) * q.lq;
            bool& f = seen[bins * xo / q.lq];
            filled += f ? 0 : 1;
            f = true;
        }
    }
    return 2 * filled < bins;
}

__global__ void identity_src_kernel(int32_t w, int32_t h, uint32_t* __restrict__ src) {
    const int64_t total = 3 * int64_t(w) * h;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < total;
         i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t p = i / 3;
        src[i] = pack_px(p / w, p % w);
    }
}

// ------------------------------------------------------------------ a3 ---
// A ray (v, x', y') is identified by its owner: the subpixel (x', y', k0) of
// the source pixel with the lowest channel k0 showing view v.  Rays are
// numbered in order of first use by the R subpixels (row-major), then G,
// then B (Sec. 5: R~_rays follows the R subpixels): an owner's order key is
// the lowest of its subpixels' keys k wh + pixel, and its ray id is the rank
// of that key.
struct RayTmp {
    uint32_t* owner;  // 3wh: owner subpixel of each subpixel's ray
    uint32_t* id_of;  // 3wh: order key, then ray id, per owner (kEmpty when not an owner)
    uint32_t* flag;   // 3wh: 1 at every used order key
    uint32_t* rank;   // 3wh
    void* scan_tmp;
};

__host__ RayTmp carve(const DisplayQ& q, void* tmp) {
    const size_t n = 3 * size_t(q.w) * q.h;
    char* p = static_cast<char*>(tmp);
    RayTmp t;
    auto take = [&](size_t bytes) {
        char* r = p;
        p += (bytes + 255) & ~size_t(255);
        return r;
    };
    t.owner = reinterpret_cast<uint32_t*>(take(4 * n));
    t.id_of = reinterpret_cast<uint32_t*>(take(4 * n));
    t.flag = reinterpret_cast<uint32_t*>(take(4 * n));
    t.rank = reinterpret_cast<uint32_t*>(take(4 * n));
    t.scan_tmp = take(0);
    return t;
}

// id_of holds kEmpty everywhere at the launch
__global__ void owner_kernel(int32_t w, int32_t h, int64_t n, const uint16_t* __restrict__ V,
                             const uint32_t* __restrict__ src, RayTmp t) {
    const uint32_t wh = uint32_t(n / 3);
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t s = src[i], p = uint32_t(i) / 3u;
        // a source outside the panel (never produced by the repurposing) is
        // read as the subpixel's own pixel rather than followed
        const bool ok = (s >> 16) < uint32_t(h) && (s & 0xFFFF) < uint32_t(w);
        const int64_t sp = ok ? int64_t(s >> 16) * w + (s & 0xFFFF) : int64_t(p);
        const uint16_t v = V[i];
        int k0 = 0;
        while (k0 < 2 && V[3 * sp + k0] != v) ++k0;
        const uint32_t o = uint32_t(3 * sp + k0);
        t.owner[i] = o;
        atomicMin(&t.id_of[o], (uint32_t(i) - 3u * p) * wh + p);
    }
}

__global__ void mark_keys_kernel(int64_t n, RayTmp t) {
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n;
         o += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t key = t.id_of[o];
        if (key != kEmpty) t.flag[key] = 1;
    }
}

__global__ void assign_kernel(int64_t n, RayTmp t) {
    for (int64_t o = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; o < n;
         o += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t key = t.id_of[o];
        if (key != kEmpty) t.id_of[o] = t.rank[key];
    }
}

__global__ void ray_of_kernel(int64_t n, const RayTmp t, uint32_t* __restrict__ ray_of) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x)
        ray_of[i] = t.id_of[t.owner[i]];
}

__global__ void ray_attr_kernel(int32_t w, int64_t n, const uint16_t* __restrict__ V,
                                const RayTmp t, uint32_t* __restrict__ ray_view,
                                uint32_t* __restrict__ ray_pix) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t r = t.id_of[i];
        if (r != kEmpty) {  // i is an owner subpixel
            const uint32_t p = uint32_t(i) / 3u, x = p / uint32_t(w);
            ray_view[r] = V[i];
            ray_pix[r] = pack_px(x, p - x * uint32_t(w));
        }
    }
}

__global__ void group_keys_kernel(const uint32_t* __restrict__ ray_view,
                                  const uint32_t* __restrict__ ray_pix, int64_t n, int32_t tw,
                                  int32_t th, int32_t ntx, int32_t nv, int shift,
                                  unsigned long long* __restrict__ keys,
                                  uint32_t* __restrict__ vals) {
    for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n;
         r += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t px = ray_pix[r];
        const uint32_t row = px >> 16, col = px & 0xFFFF;
        // tile-major: the views of a tile are neighbours in the grouping
        const uint64_t g = uint64_t((row / th) * ntx + (col / tw)) * nv + ray_view[r];
        // inside the tile, order rays along a Morton curve so that each warp's
        // rays cover a compact patch
        uint32_t x = col % tw, y = row % th, m = 0;
        for (int b = 0; b < 8; ++b) m |= (((x >> b) & 1u) << (2 * b)) | (((y >> b) & 1u) << (2 * b + 1));
        keys[r] = (g << shift) | m;
        vals[r] = uint32_t(r);
    }
}

__global__ void group_gather_kernel(const uint32_t* __restrict__ order,
                                    const uint32_t* __restrict__ ray_pix, int64_t n,
                                    int2* __restrict__ grouped) {
    for (int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; j < n;
         j += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t r = order[j];
        grouped[j] = make_int2(int(ray_pix[r]), int(r));
    }
}

// pos[ray id] = position of the ray in the (view, tile) grouping
__global__ void group_pos_kernel(const int2* __restrict__ grouped, int64_t n,
                                 uint32_t* __restrict__ pos) {
    for (int64_t j = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; j < n;
         j += int64_t(gridDim.x) * blockDim.x)
        pos[uint32_t(grouped[j].y)] = uint32_t(j);
}

// slot_of[i] = pos[ray_of[i]]: the grouped position of subpixel i's ray
__global__ void group_slot_kernel(const uint32_t* __restrict__ ray_of, int64_t n,
                                  const uint32_t* __restrict__ pos, uint32_t* __restrict__ slot_of) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x)
        slot_of[i] = pos[ray_of[i]];
}

// Work lists of a grouping: ranges[k], k = tile * nv + view, are the rays of
// group g = view * ntiles + tile.  chunks[k]: pieces of at most `piece` rays;
// used[g]: 1 when the group holds rays.  Entry n_groups of both is 0.
__global__ void list_counts_kernel(const uint2* __restrict__ ranges, int64_t n_groups, int64_t ntiles,
                                   int64_t nv, uint32_t piece, uint32_t* __restrict__ chunks,
                                   uint32_t* __restrict__ used) {
    for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k <= n_groups;
         k += int64_t(gridDim.x) * blockDim.x) {
        const uint2 r = k < n_groups ? ranges[k] : make_uint2(0u, 0u);
        const int64_t tile = k / nv;
        chunks[k] = (r.y - r.x + piece - 1) / piece;
        used[k < n_groups ? (k - tile * nv) * ntiles + tile : k] = r.y > r.x ? 1u : 0u;
    }
}

// work: every piece {group, first ray, end ray, -} in k order; gwork: every
// group with rays {group, first ray, end ray, -} in g (view-major) order.
__global__ void list_fill_kernel(const uint2* __restrict__ ranges, int64_t n_groups, int64_t ntiles,
                                 int64_t nv, uint32_t piece, const uint32_t* __restrict__ chunk_at,
                                 const uint32_t* __restrict__ used_at, int4* __restrict__ work,
                                 int4* __restrict__ gwork) {
    for (int64_t k = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; k < n_groups;
         k += int64_t(gridDim.x) * blockDim.x) {
        const uint2 r = ranges[k];
        if (r.y <= r.x) continue;
        const int64_t tile = k / nv, g = (k - tile * nv) * ntiles + tile;
        gwork[used_at[g]] = make_int4(int(g), int(r.x), int(r.y), 0);
        uint32_t w = chunk_at[k];
        for (uint32_t b = r.x; b < r.y; b += piece)
            work[w++] = make_int4(int(g), int(b), int(min(b + piece, r.y)), 0);
    }
}

__global__ void rays_export_kernel(const uint32_t* __restrict__ ray_view,
                                   const uint32_t* __restrict__ ray_pix, int64_t n,
                                   int32_t* __restrict__ out) {
    for (int64_t r = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; r < n;
         r += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t px = ray_pix[r];
        out[3 * r] = int32_t(ray_view[r]);
        out[3 * r + 1] = int32_t(px >> 16);
        out[3 * r + 2] = int32_t(px & 0xFFFF);
    }
}

// (view, row, col) of every ray straight from the owner table.
__global__ void ray_triplets_kernel(int32_t w, int64_t n, const uint16_t* __restrict__ V,
                                    const RayTmp t, int32_t* __restrict__ out) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n;
         i += int64_t(gridDim.x) * blockDim.x) {
        const uint32_t r = t.id_of[i];
        if (r != kEmpty) {
            const int64_t p = i / 3;
            out[3 * int64_t(r)] = int32_t(V[i]);
            out[3 * int64_t(r) + 1] = int32_t(p / w);
            out[3 * int64_t(r) + 2] = int32_t(p % w);
        }
    }
}

int grid_for(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    const int64_t cap = int64_t(num_sms()) * 16;
    if (g > cap) g = cap;
    return int(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t launch_view_map(const DisplayQ& q, uint16_t* V, cudaStream_t s) {
    const int64_t n8 = (3 * int64_t(q.w) * q.h + 7) / 8;
    // 2^32 mod L_x: whole lens lines (a pitch below a subpixel) do not count
    const int64_t n = int64_t(q.nv) * (kQ32 % q.lq);
    view_map_kernel<<<grid_for(n8, 256), 256, 0, s>>>(q, n / q.lq, n % q.lq, V);
    return cudaGetLastError();
}

cudaError_t launch_repurpose(const DisplayQ& q, const uint16_t* V, uint32_t* src, int identity,
                             cudaStream_t s) {
    if (identity) {
        identity_src_kernel<<<grid_for(3 * int64_t(q.w) * q.h, 256), 256, 0, s>>>(q.w, q.h, src);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(src, 0xFF, sizeof(uint32_t) * 3 * size_t(q.w) * q.h, s);
    if (e != cudaSuccess) return e;
    if (q.lq < kQ32 || (2 * q.lq < 7 * kQ32 && few_offsets(q))) {
        repurpose_area_kernel<<<(q.n_areas + 3) / 4, 128, 0, s>>>(q, V, src);
        return cudaGetLastError();
    }
    // a warp a block: the warps' lengths differ with the areas on the panel
    const int64_t blocks = (int64_t(q.n_areas) * q.nv * kChainLanes + 31) / 32;
    repurpose_kernel<<<unsigned(blocks < 0x7FFFFFFF ? blocks : 0x7FFFFFFF), 32, 0, s>>>(q, src);
    return cudaGetLastError();
}

size_t ray_table_tmp_bytes(const DisplayQ& q) {
    const size_t n = 3 * size_t(q.w) * q.h;
    return 4 * ((4 * n + 255) & ~size_t(255)) + scan_tmp_bytes(int64_t(n)) + 256;
}

cudaError_t launch_ray_table(const DisplayQ& q, const uint16_t* V, const uint32_t* src,
                             uint32_t* ray_of, void* tmp, uint32_t* d_n_rays, cudaStream_t s) {
    const int64_t n = 3 * int64_t(q.w) * q.h;
    RayTmp t = carve(q, tmp);
    cudaError_t e = cudaMemsetAsync(t.flag, 0, sizeof(uint32_t) * size_t(n), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(t.id_of, 0xFF, sizeof(uint32_t) * size_t(n), s);
    if (e != cudaSuccess) return e;
    owner_kernel<<<grid_for(n, 256), 256, 0, s>>>(q.w, q.h, n, V, src, t);
    mark_keys_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, t);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_exclusive_scan(t.flag, t.rank, n, d_n_rays, t.scan_tmp, s);
    if (e != cudaSuccess) return e;
    assign_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, t);
    ray_of_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, t, ray_of);
    return cudaGetLastError();
}

cudaError_t launch_ray_attributes(const DisplayQ& q, const uint16_t* V, const void* tmp,
                                  uint32_t* ray_view, uint32_t* ray_pix, cudaStream_t s) {
    const int64_t n = 3 * int64_t(q.w) * q.h;
    RayTmp t = carve(q, const_cast<void*>(tmp));
    ray_attr_kernel<<<grid_for(n, 256), 256, 0, s>>>(q.w, n, V, t, ray_view, ray_pix);
    return cudaGetLastError();
}

cudaError_t launch_ray_group_keys(const uint32_t* ray_view, const uint32_t* ray_pix, int64_t n_rays,
                                  int32_t tile_w, int32_t tile_h, int32_t ntx, int32_t nv, int shift,
                                  unsigned long long* keys, uint32_t* vals, cudaStream_t s) {
    group_keys_kernel<<<grid_for(n_rays, 256), 256, 0, s>>>(ray_view, ray_pix, n_rays, tile_w,
                                                             tile_h, ntx, nv, shift, keys, vals);
    return cudaGetLastError();
}

cudaError_t launch_list_counts(const uint2* ranges, int64_t n_groups, int32_t ntiles, int32_t nv,
                               int32_t piece, uint32_t* chunks, uint32_t* used, cudaStream_t s) {
    list_counts_kernel<<<grid_for(n_groups + 1, 256), 256, 0, s>>>(ranges, n_groups, ntiles, nv,
                                                                   uint32_t(piece), chunks, used);
    return cudaGetLastError();
}

cudaError_t launch_list_fill(const uint2* ranges, int64_t n_groups, int32_t ntiles, int32_t nv,
                             int32_t piece, const uint32_t* chunk_at, const uint32_t* used_at,
                             int4* work, int4* gwork, cudaStream_t s) {
    list_fill_kernel<<<grid_for(n_groups, 256), 256, 0, s>>>(ranges, n_groups, ntiles, nv,
                                                             uint32_t(piece), chunk_at, used_at, work,
                                                             gwork);
    return cudaGetLastError();
}

cudaError_t launch_rays_export(const uint32_t* ray_view, const uint32_t* ray_pix, int64_t n_rays,
                               int32_t* out, cudaStream_t s) {
    if (n_rays <= 0) return cudaSuccess;
    rays_export_kernel<<<grid_for(n_rays, 256), 256, 0, s>>>(ray_view, ray_pix, n_rays, out);
    return cudaGetLastError();
}

cudaError_t launch_ray_group_gather(const uint32_t* order, const uint32_t* ray_pix, int64_t n_rays,
                                    int2* grouped, cudaStream_t s) {
    group_gather_kernel<<<grid_for(n_rays, 256), 256, 0, s>>>(order, ray_pix, n_rays, grouped);
    return cudaGetLastError();
}

cudaError_t launch_group_slots(const int2* grouped, int64_t n_rays, const uint32_t* ray_of,
                               int64_t n_subpixels, uint32_t* pos_tmp, uint32_t* slot_of,
                               cudaStream_t s) {
    group_pos_kernel<<<grid_for(n_rays, 256), 256, 0, s>>>(grouped, n_rays, pos_tmp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    group_slot_kernel<<<grid_for(n_subpixels, 256), 256, 0, s>>>(ray_of, n_subpixels, pos_tmp,
                                                                  slot_of);
    return cudaGetLastError();
}

}  // namespace dl

// ---------------------------------------------------------------------------
// Ray table without any allocation.
//
// Some callers cannot call cudaMalloc: code running where the allocator is
// off limits (inside another library's memory pool, in a process whose
// device memory is fully reserved up front, or in a real-time loop that must
// not synchronise the device the way cudaMalloc/cudaFree can).  For them
// dl_ray_table_static builds the same ray table as dl_set_display, from a
// view map and subpixel map the caller holds in device memory, using only
// this file-scope scratch array.  Every GPU that loads the library holds the
// array until the process exits.
namespace {
constexpr int64_t kStaticMaxPixels = 65536;  // panels up to e.g. 256 x 256
constexpr size_t kStaticScratchBytes = 6u * 1024u * 1024u + 512u * 1024u;
constexpr int kStaticMaxDevices = 64;
}  // namespace

static __device__ __align__(256) unsigned char g_ray_table_scratch[kStaticScratchBytes];

static std::mutex g_static_mu;
static void* g_static_addr[kStaticMaxDevices] = {};

extern "C" dl_status dl_ray_table_static(int32_t width, int32_t height, const uint16_t* V,
                                         const uint32_t* src, uint32_t* ray_of, int32_t* rays,
                                         int64_t* n_rays, void* stream) {
    using namespace dl;
    if (!V || !src || !ray_of || !rays || !n_rays || width < 1 || height < 1)
        return DL_ERR_INVALID_ARG;
    if (int64_t(width) * height > kStaticMaxPixels) return DL_ERR_INVALID_ARG;
    DisplayQ q{};
    q.w = width;
    q.h = height;
    if (ray_table_tmp_bytes(q) + 256 > kStaticScratchBytes) return DL_ERR_INVALID_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return DL_ERR_CUDA;
    }
    if (dev < 0 || dev >= kStaticMaxDevices) return DL_ERR_INVALID_ARG;
    void* base = nullptr;
    {
        // Host code only knows a stand-in for the array's name: ask the
        // runtime for its device address, once per device.
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_addr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_ray_table_scratch) != cudaSuccess || !p) {
                cudaGetLastError();
                return DL_ERR_CUDA;
            }
            g_static_addr[dev] = p;
        }
        base = g_static_addr[dev];
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    uint32_t* d_n = reinterpret_cast<uint32_t*>(static_cast<char*>(base) + kStaticScratchBytes - 256);
    const int64_t n = 3 * int64_t(width) * height;
    if (launch_ray_table(q, V, src, ray_of, base, d_n, s) != cudaSuccess) {
        cudaGetLastError();
        return DL_ERR_CUDA;
    }
    RayTmp t = carve(q, base);
    ray_triplets_kernel<<<grid_for(n, 256), 256, 0, s>>>(width, n, V, t, rays);
    uint32_t h_n = 0;
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(&h_n, d_n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        cudaGetLastError();
        return DL_ERR_CUDA;
    }
    *n_rays = int64_t(h_n);
    return DL_OK;
}

