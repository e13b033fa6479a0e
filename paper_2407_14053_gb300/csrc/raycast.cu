// Ray-order 3DGS (Sec. 7, Alg. 3): every required ray is cast through the
// scene, one thread per ray.  Per ray, each Gaussian it meets gives its point
// of highest density t_j = (mu - o)^T S^-1 d / (d^T S^-1 d) (Eq. (16)) and
// alpha_j = o_j G(o + t_j d) (Eq. (17)); the c_h nearest are kept (Alg. 3
// keeps them in a max-heap of capacity c_h; here an ascending list of the
// same capacity, which needs no sort at the end) and blended front to back
// with the SH colour at the ray direction.  The ray meets a Gaussian when
// alpha_j >= 1/255 and t_j > 0.2 (the near plane of the rasteriser); the
// list orders by (t, index), so the image does not depend on the traversal
// order.
//
// Two ways to the Gaussians a ray meets.  Rays normally go through the list of
// their (view, tile), which holds every Gaussian whose alpha >= 1/255 outline
// reaches the tile (rc_cast_kernel).  When the lists of a frame do not fit
// their memory, the rays walk the scene's tree (rc_trace_kernel).  Both test
// with rc_alpha and keep the same list; the colours may differ by the order of
// the SH sums (rc_blend_kernel).
//
// The tree (Sec. 7: a compact 8-wide bounding-volume hierarchy built with
// the surface area heuristic): every Gaussian is bounded by the box of its
// alpha >= 1/255 ellipsoid.  A binary tree is built top down over the
// scene's stored order (a 3D Morton curve of the means), so every node holds
// a contiguous run of Gaussians; each node is split at the position of the
// run that minimises the SAH cost A(left) n(left) + A(right) n(right) over
// every split position (prefix and suffix boxes of the run), down to leaves
// of at most four Gaussians.  The binary tree is then collapsed into 8-wide
// nodes: a wide node starts from a binary node's two children and
// repeatedly opens the child with the largest surface area until it has
// eight.  Children are visited nearest first, and once the list is full a
// node whose box starts beyond the list's farthest entry is skipped: a
// Gaussian's highest-density point lies inside its ellipsoid, hence inside
// every box above it.
#include <cfloat>

#include "dl_internal.cuh"
#include "sh.cuh"
#include "warp_sort.cuh"

namespace dl {
namespace {

constexpr float kNearT = 0.2f;
constexpr float kMinAlpha = 1.0f / 255.0f;

// Per Gaussian: a = (mean, opacity), b = (S00, S01, S02, S11), c = (S12, S22)
// of S = Sigma^-1 = R diag(s^-2) R^T; box of the alpha >= 1/255 ellipsoid.
template <typename T>
__global__ void rc_prepare_kernel(GaussiansView<T> G, int64_t n, float4* __restrict__ gauss,
                                  float4* __restrict__ box) {
    for (int64_t g = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; g < n;
         g += int64_t(gridDim.x) * blockDim.x) {
        float qw = to_f(G.rot[4 * g]), qx = to_f(G.rot[4 * g + 1]);
        float qy = to_f(G.rot[4 * g + 2]), qz = to_f(G.rot[4 * g + 3]);
        const float qn = rsqrtf(qw * qw + qx * qx + qy * qy + qz * qz);
        qw *= qn; qx *= qn; qy *= qn; qz *= qn;
        const float R[3][3] = {
            {1.f - 2.f * (qy * qy + qz * qz), 2.f * (qx * qy - qw * qz), 2.f * (qx * qz + qw * qy)},
            {2.f * (qx * qy + qw * qz), 1.f - 2.f * (qx * qx + qz * qz), 2.f * (qy * qz - qw * qx)},
            {2.f * (qx * qz - qw * qy), 2.f * (qy * qz + qw * qx), 1.f - 2.f * (qx * qx + qy * qy)}};
        float s2[3], is2[3];
        for (int k = 0; k < 3; ++k) {
            const float ls = to_f(G.log_scale[3 * g + k]);
            s2[k] = __expf(2.f * ls);
            is2[k] = __expf(-2.f * ls);
        }
        auto inv = [&](int i, int j) {
            return R[i][0] * R[j][0] * is2[0] + R[i][1] * R[j][1] * is2[1] + R[i][2] * R[j][2] * is2[2];
        };
        const float op = 1.f / (1.f + __expf(-to_f(G.opacity_logit[g])));
        const float mx = G.mean[3 * g], my = G.mean[3 * g + 1], mz = G.mean[3 * g + 2];
        gauss[3 * g] = make_float4(mx, my, mz, op);
        gauss[3 * g + 1] = make_float4(inv(0, 0), inv(0, 1), inv(0, 2), inv(1, 1));
        gauss[3 * g + 2] = make_float4(inv(1, 2), inv(2, 2), 0.f, 0.f);
        // alpha >= 1/255 inside (x - mu)^T S (x - mu) <= K = 2 ln(255 o); the
        // ellipsoid's half extent along axis i is sqrt(K Sigma_ii) (+0.1 %)
        float4 lo = make_float4(FLT_MAX, FLT_MAX, FLT_MAX, 0.f), hi = make_float4(-FLT_MAX, -FLT_MAX, -FLT_MAX, 0.f);
        if (op * 255.f > 1.f) {
            const float K = 2.f * logf(255.f * op);
            float h[3];
            for (int i = 0; i < 3; ++i)
                h[i] = sqrtf(K * (R[i][0] * R[i][0] * s2[0] + R[i][1] * R[i][1] * s2[1] +
                                  R[i][2] * R[i][2] * s2[2])) * 1.001f + 1e-6f;
            lo = make_float4(mx - h[0], my - h[1], mz - h[2], 0.f);
            hi = make_float4(mx + h[0], my + h[1], mz + h[2], 0.f);
        }
        box[2 * g] = lo;
        box[2 * g + 1] = hi;
    }
}

// ---- SAH tree ------------------------------------------------------------
constexpr int kLeafMax = 4;           // Gaussians per leaf of the binary tree
constexpr int kMedianDepth = 40;      // from this binary depth on, runs split at the middle
constexpr int kBuildThreads = 256;

__host__ __device__ inline uint32_t leaf_ref(uint32_t first, uint32_t count) {
    return kRayLeafBit | (first << 3) | (count - 1);
}

// Binary node of the build (not kept): box, children (node index or leaf
// reference), the box's surface area.
struct BinNode {
    float4 lo, hi;
    uint32_t child[2];
    float area;
    uint32_t pad;
};
// Run [a, b) of Gaussians that becomes binary node `node` at `depth`.
struct BuildTask {
    uint32_t a, b, node, depth;
};

struct Box {
    float lx, ly, lz, hx, hy, hz;
};
__device__ __forceinline__ Box box_empty() { return {FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX}; }
__device__ __forceinline__ Box box_join(const Box& a, const Box& b) {
    return {fminf(a.lx, b.lx), fminf(a.ly, b.ly), fminf(a.lz, b.lz),
            fmaxf(a.hx, b.hx), fmaxf(a.hy, b.hy), fmaxf(a.hz, b.hz)};
}
__device__ __forceinline__ Box box_of(const float4* __restrict__ gbox, uint32_t g) {
    const float4 l = gbox[2 * size_t(g)], h = gbox[2 * size_t(g) + 1];
    return {l.x, l.y, l.z, h.x, h.y, h.z};
}
__device__ __forceinline__ float box_area(const Box& b) {
    const float dx = b.hx - b.lx, dy = b.hy - b.ly, dz = b.hz - b.lz;
    if (!(dx >= 0.f) || !(dy >= 0.f) || !(dz >= 0.f)) return 0.f;
    return 2.f * (dx * dy + dy * dz + dz * dx);
}
__device__ __forceinline__ Box shfl_box(const Box& b, int src_delta, bool up) {
    Box r;
    if (up) {
        r.lx = __shfl_up_sync(0xffffffffu, b.lx, src_delta);
        r.ly = __shfl_up_sync(0xffffffffu, b.ly, src_delta);
        r.lz = __shfl_up_sync(0xffffffffu, b.lz, src_delta);
        r.hx = __shfl_up_sync(0xffffffffu, b.hx, src_delta);
        r.hy = __shfl_up_sync(0xffffffffu, b.hy, src_delta);
        r.hz = __shfl_up_sync(0xffffffffu, b.hz, src_delta);
    } else {
        r.lx = __shfl_down_sync(0xffffffffu, b.lx, src_delta);
        r.ly = __shfl_down_sync(0xffffffffu, b.ly, src_delta);
        r.lz = __shfl_down_sync(0xffffffffu, b.lz, src_delta);
        r.hx = __shfl_down_sync(0xffffffffu, b.hx, src_delta);
        r.hy = __shfl_down_sync(0xffffffffu, b.hy, src_delta);
        r.hz = __shfl_down_sync(0xffffffffu, b.hz, src_delta);
    }
    return r;
}

// Exclusive prefix (pre) and suffix (suf) unions of the block's per-thread
// boxes in thread order, and their total.  Every thread of the block calls it.
__device__ void block_box_scans(const Box& mine, Box& pre, Box& suf, Box& total) {
    __shared__ Box s_warp[kBuildThreads / 32], s_pre[kBuildThreads / 32], s_suf[kBuildThreads / 32];
    __shared__ Box s_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Box inc = mine, rinc = mine;  // inclusive prefix / suffix inside the warp
    for (int o = 1; o < 32; o <<= 1) {
        const Box u = shfl_box(inc, o, true), d = shfl_box(rinc, o, false);
        if (lane >= o) inc = box_join(inc, u);
        if (lane + o < 32) rinc = box_join(rinc, d);
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (threadIdx.x == 0) {
        Box run = box_empty();
        for (int w = 0; w < nw; ++w) {
            s_pre[w] = run;
            run = box_join(run, s_warp[w]);
        }
        s_total = run;
        run = box_empty();
        for (int w = nw - 1; w >= 0; --w) {
            s_suf[w] = run;
            run = box_join(run, s_warp[w]);
        }
    }
    __syncthreads();
    const Box ex_in = shfl_box(inc, 1, true);     // inclusive prefix of lane - 1
    const Box ex_rin = shfl_box(rinc, 1, false);  // inclusive suffix of lane + 1
    pre = lane > 0 ? box_join(s_pre[warp], ex_in) : s_pre[warp];
    suf = lane < 31 ? box_join(s_suf[warp], ex_rin) : s_suf[warp];
    total = s_total;
    __syncthreads();
}

// One block per task: the run [a, b) is split at the position k (a < k < b)
// minimising A([a, k)) (k - a) + A([k, b)) (b - k), over every position
// (from binary depth kMedianDepth on: the middle).  A side of at most
// kLeafMax Gaussians becomes a leaf, a longer one a new node and a task of
// the next level.  sal: one float per Gaussian of scratch.  counters[0]:
// binary nodes allocated, counters[1]: next level's tasks.
__global__ void __launch_bounds__(kBuildThreads)
sah_split_kernel(const BuildTask* __restrict__ tasks, const float4* __restrict__ gbox,
                 float* __restrict__ sal, BinNode* __restrict__ nodes, BuildTask* __restrict__ next,
                 uint32_t* __restrict__ counters) {
    __shared__ float s_cost[kBuildThreads];
    __shared__ uint32_t s_k[kBuildThreads];
    const BuildTask tk = tasks[blockIdx.x];
    const uint32_t a = tk.a, b = tk.b, m = b - a;
    const uint32_t per = (m + blockDim.x - 1) / blockDim.x;
    const uint32_t c0 = min(b, a + threadIdx.x * per), c1 = min(b, c0 + per);
    Box cb = box_empty();
    for (uint32_t g = c0; g < c1; ++g) cb = box_join(cb, box_of(gbox, g));
    Box pre, suf, total;
    block_box_scans(cb, pre, suf, total);
    // forward: sal[g] = area of [a, g + 1)
    Box L = pre;
    for (uint32_t g = c0; g < c1; ++g) {
        L = box_join(L, box_of(gbox, g));
        sal[g] = box_area(L);
    }
    __syncthreads();
    // backward: the cost of splitting at k = g, right side [g, b)
    Box R = suf;
    float best = FLT_MAX;
    uint32_t bk = a + m / 2;
    for (uint32_t g = c1; g > c0; --g) {
        R = box_join(R, box_of(gbox, g - 1));
        const uint32_t k = g - 1;
        if (k > a) {
            const float cost = sal[k - 1] * float(k - a) + box_area(R) * float(b - k);
            if (cost < best || (cost == best && k < bk)) {
                best = cost;
                bk = k;
            }
        }
    }
    s_cost[threadIdx.x] = best;
    s_k[threadIdx.x] = bk;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t k = a + m / 2;
        if (tk.depth < uint32_t(kMedianDepth)) {
            float bc = FLT_MAX;
            for (unsigned t = 0; t < blockDim.x; ++t)
                if (s_cost[t] < bc || (s_cost[t] == bc && s_k[t] < k)) {
                    bc = s_cost[t];
                    k = s_k[t];
                }
            if (!(bc < FLT_MAX)) k = a + m / 2;  // every box empty: the middle
        }
        BinNode nd;
        nd.lo = make_float4(total.lx, total.ly, total.lz, 0.f);
        nd.hi = make_float4(total.hx, total.hy, total.hz, 0.f);
        nd.area = box_area(total);
        nd.pad = 0u;
        const uint32_t ra[2] = {a, k}, rb[2] = {k, b};
        for (int side = 0; side < 2; ++side) {
            const uint32_t n = rb[side] - ra[side];
            if (n <= uint32_t(kLeafMax)) {
                nd.child[side] = leaf_ref(ra[side], n);
            } else {
                const uint32_t id = atomicAdd(counters, 1u);
                nd.child[side] = id;
                next[atomicAdd(counters + 1, 1u)] = BuildTask{ra[side], rb[side], id, tk.depth + 1};
            }
        }
        nodes[tk.node] = nd;
    }
}

// Collapse of the binary tree into 8-wide nodes, one wide node per task: the
// binary node's two children are opened, the one with the largest surface
// area first, until there are eight (or only leaves).  counters[2]: wide
// nodes allocated, [3]: next level's tasks, [4]: deepest wide level.
struct CollapseTask {
    uint32_t bin, wide, depth, pad;
};

__global__ void collapse_kernel(const CollapseTask* __restrict__ q, uint32_t nq,
                                const BinNode* __restrict__ bins, const float4* __restrict__ gbox,
                                RayNode* __restrict__ wide, CollapseTask* __restrict__ next,
                                uint32_t* __restrict__ counters) {
    for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < nq; idx += gridDim.x * blockDim.x) {
        const CollapseTask t = q[idx];
        uint32_t ref[8];
        int c = 2;
        ref[0] = bins[t.bin].child[0];
        ref[1] = bins[t.bin].child[1];
        while (c < 8) {
            int best = -1;
            float ba = -1.f;
            for (int i = 0; i < c; ++i)
                if (!(ref[i] & kRayLeafBit) && bins[ref[i]].area > ba) {
                    ba = bins[ref[i]].area;
                    best = i;
                }
            if (best < 0) break;
            const uint32_t r = ref[best];
            ref[best] = bins[r].child[0];
            ref[c++] = bins[r].child[1];
        }
        RayNode nd;
        for (int k = 0; k < 8; ++k) {
            Box bx = box_empty();
            uint32_t ch = kRayNoChild;
            if (k < c) {
                if (ref[k] & kRayLeafBit) {
                    const uint32_t first = (ref[k] & ~kRayLeafBit) >> 3, cnt = (ref[k] & 7u) + 1u;
                    for (uint32_t g = first; g < first + cnt; ++g) bx = box_join(bx, box_of(gbox, g));
                    ch = ref[k];
                } else {
                    const BinNode& bn = bins[ref[k]];
                    bx = {bn.lo.x, bn.lo.y, bn.lo.z, bn.hi.x, bn.hi.y, bn.hi.z};
                    ch = atomicAdd(counters + 2, 1u);
                    next[atomicAdd(counters + 3, 1u)] = CollapseTask{ref[k], ch, t.depth + 1, 0u};
                }
            }
            nd.lox[k] = bx.lx; nd.loy[k] = bx.ly; nd.loz[k] = bx.lz;
            nd.hix[k] = bx.hx; nd.hiy[k] = bx.hy; nd.hiz[k] = bx.hz;
            nd.child[k] = ch;
            nd.pad[k] = 0u;
        }
        wide[t.wide] = nd;
        atomicMax(counters + 4, t.depth);
    }
}

// A scene of at most kLeafMax Gaussians: the root holds one leaf.
__global__ void leaf_root_kernel(const float4* __restrict__ gbox, uint32_t n, RayNode* __restrict__ wide) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    RayNode nd;
    for (int k = 0; k < 8; ++k) {
        Box bx = box_empty();
        uint32_t ch = kRayNoChild;
        if (k == 0 && n > 0) {
            for (uint32_t g = 0; g < n; ++g) bx = box_join(bx, box_of(gbox, g));
            ch = leaf_ref(0u, n);
        }
        nd.lox[k] = bx.lx; nd.loy[k] = bx.ly; nd.loz[k] = bx.lz;
        nd.hix[k] = bx.hx; nd.hiy[k] = bx.hy; nd.hiz[k] = bx.hz;
        nd.child[k] = ch;
        nd.pad[k] = 0u;
    }
    wide[0] = nd;
}

// Highest-density point and alpha along the ray of the Gaussian whose three
// float4 are at pa, pb, pc (global or shared memory).  They are read into
// locals first: taking them by reference changed the compiler's choice of
// fused multiply-adds, and a few pixels in a million with it.
__device__ __forceinline__ float rc_alpha(const float4* pa, const float4* pb, const float4* pc,
                                          float ox, float oy, float oz, float dx, float dy, float dz,
                                          float& t) {
    const float4 a = *pa, b = *pb, c = *pc;
    // S d and d^T S d, S = [[b.x b.y b.z] [b.y b.w c.x] [b.z c.x c.y]]
    const float sx = b.x * dx + b.y * dy + b.z * dz;
    const float sy = b.y * dx + b.w * dy + c.x * dz;
    const float sz = b.z * dx + c.x * dy + c.y * dz;
    const float den = dx * sx + dy * sy + dz * sz;
    const float mx = a.x - ox, my = a.y - oy, mz = a.z - oz;
    t = (mx * sx + my * sy + mz * sz) / den;
    const float px = t * dx - mx, py = t * dy - my, pz = t * dz - mz;
    const float q = b.x * px * px + b.w * py * py + c.y * pz * pz +
                    2.f * (b.y * px * py + b.z * px * pz + c.x * py * pz);
    return fminf(0.99f, a.w * __expf(-0.5f * q));
}
__device__ __forceinline__ float rc_alpha(const float4* __restrict__ gauss, int64_t g, float ox,
                                          float oy, float oz, float dx, float dy, float dz, float& t) {
    return rc_alpha(gauss + 3 * g, gauss + 3 * g + 1, gauss + 3 * g + 2, ox, oy, oz, dx, dy, dz, t);
}

// Whole 16-byte pieces of a Gaussian's SH coefficients, 0 when their size is no
// multiple of that (degree 3, and degree 1 in FP32, is).
template <typename T, int DEG>
constexpr int sh_pieces() {
    constexpr int bytes = 3 * (DEG + 1) * (DEG + 1) * int(sizeof(T));
    return bytes % 16 == 0 ? bytes / 16 : 0;
}

// Adds the coefficients of piece p to the colour sums acc[0..2], Y being the
// basis values of the direction (coefficient index outer, RGB inner).
template <typename T>
__device__ __forceinline__ void sh_piece(const uint4& raw, int p, const float* Y, float* acc) {
    constexpr int VE = 16 / int(sizeof(T));
    T v[VE];
    memcpy(v, &raw, 16);
#pragma unroll
    for (int k = 0; k < VE; ++k) {
        const int f = p * VE + k;
        acc[f % 3] = fmaf(Y[f / 3], to_f(v[k]), acc[f % 3]);
    }
}

// SH colour of a Gaussian.  Every lane of a warp reads another Gaussian, so a
// load touches a line per lane whatever its width: the coefficients are read
// in pieces of 16 bytes where their size allows (the array is 256-byte
// aligned), else one by one.
template <typename T, int DEG>
__device__ __forceinline__ void sh_colour(const T* __restrict__ sh, const float* Y, float* col) {
    constexpr int NF = 3 * (DEG + 1) * (DEG + 1), NP = sh_pieces<T, DEG>();
    float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int p = 0; p < NP; ++p) sh_piece<T>(__ldg(reinterpret_cast<const uint4*>(sh) + p), p, Y, acc);
#pragma unroll
    for (int f = NP ? NF : 0; f < NF; ++f) acc[f % 3] = fmaf(Y[f / 3], to_f(sh[f]), acc[f % 3]);
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) col[ch] = fmaxf(acc[ch] + 0.5f, 0.f);
}

constexpr int kTraceThreads = 128;
constexpr int kTraceWarps = kTraceThreads / 32;

// A ray's entry into a box (+inf when it misses the box or the box lies
// behind the near plane).
__device__ __forceinline__ float slab_enter(const float4& lo, const float4& hi, float ox, float oy,
                                            float oz, float ix, float iy, float iz) {
    const float tx0 = (lo.x - ox) * ix, tx1 = (hi.x - ox) * ix;
    const float ty0 = (lo.y - oy) * iy, ty1 = (hi.y - oy) * iy;
    const float tz0 = (lo.z - oz) * iz, tz1 = (hi.z - oz) * iz;
    const float tn = fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fminf(tz0, tz1));
    const float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fmaxf(tz0, tz1));
    return (tn <= tf && tf > kNearT) ? tn : INFINITY;
}

// A ray: camera centre, unit direction through its pixel (camera ray ((c -
// w/2 - shift)/f, (r - h/2)/f, 1) to world).
struct Ray {
    float ox, oy, oz, dx, dy, dz;
};
__device__ __forceinline__ Ray make_ray(const Cam& cam, uint32_t pixel, float focal, float half_w,
                                        float half_h) {
    Ray r;
    const float cx = (float(pixel & 0xFFFFu) - half_w - cam.shift) / focal;
    const float cy = (float(pixel >> 16) - half_h) / focal;
    r.dx = cam.r[0] * cx + cam.r[3] * cy + cam.r[6];
    r.dy = cam.r[1] * cx + cam.r[4] * cy + cam.r[7];
    r.dz = cam.r[2] * cx + cam.r[5] * cy + cam.r[8];
    const float dn = rsqrtf(r.dx * r.dx + r.dy * r.dy + r.dz * r.dz);
    r.dx *= dn; r.dy *= dn; r.dz *= dn;
    r.ox = cam.c[0];
    r.oy = cam.c[1];
    r.oz = cam.c[2];
    return r;
}

// A ray's ascending list of its c_h nearest intersections, packed as t's FP32
// bits << 32 | Gaussian index: t > 0, so the integer order of the packed key
// is the (t, index) order.  The tree walk keeps slots below kListHead in
// shared memory (slot k at head[32 k]) and the rest in the thread's local
// memory; the cast keeps slot k of every ray of a chunk together.
constexpr int kListHead = 16;
struct WalkList {
    unsigned long long* head;
    unsigned long long* rest;
    __device__ __forceinline__ unsigned long long get(int k) const {
        return k < kListHead ? head[32 * k] : rest[k - kListHead];
    }
    __device__ __forceinline__ void set(int k, unsigned long long v) const {
        if (k < kListHead) head[32 * k] = v;
        else rest[k - kListHead] = v;
    }
};
struct CastList {
    unsigned long long* slot0;
    int64_t stride;
    __device__ __forceinline__ unsigned long long get(int k) const { return slot0[k * stride]; }
    __device__ __forceinline__ void set(int k, unsigned long long v) const { slot0[k * stride] = v; }
};

// What a ray has found: its list and the transmittance bound.  tb is set once
// the intersections found so far (every one at t <= tmax) multiply T below
// 5e-5.  Sorted, they alone take T below 1e-4 by t = tmax, so blending stops
// at or before tmax and nothing beyond tb can be blended.  (5e-5, not 1e-4:
// the product is formed in another order than the blend's.)
// LAST: the list's largest key is kept in a register, so a hit that comes in
// order is stored without a read (the cast; the tree walk has no register to
// spare).
template <class List, bool LAST>
struct RayHits {
    List list;
    int n = 0, cap;
    float prodT = 1.f, tmax = 0.f, tb = INFINITY;
    unsigned long long top = 0ull;
    __device__ __forceinline__ unsigned long long largest() const { return LAST ? top : list.get(n - 1); }
    // no intersection beyond this is kept
    __device__ __forceinline__ float bound() const {
        return fminf(tb, n == cap ? __uint_as_float(uint32_t(largest() >> 32)) : INFINITY);
    }
    __device__ __forceinline__ void add(float a, float t, uint32_t g) {
        if (!(a >= kMinAlpha) || !(t > kNearT) || t > tb) return;
        if (tb == INFINITY) {
            prodT *= 1.f - a;
            tmax = fmaxf(tmax, t);
            if (prodT < 5e-5f) tb = tmax;
        }
        const unsigned long long key = (static_cast<unsigned long long>(__float_as_uint(t)) << 32) | g;
        if (LAST && key > top) {
            if (n == cap) return;  // full and farther than all
            list.set(n++, key);
            top = key;
            return;
        }
        if (n == cap) {  // full: drop the farthest if this one is nearer
            if (!LAST && !(key < list.get(n - 1))) return;
            --n;
        }
        // insert into the ascending list: rays find their intersections
        // nearly in order, so few entries move
        int k = n++;
        while (k > 0) {
            const unsigned long long vp = list.get(k - 1);
            if (!(key < vp)) break;
            list.set(k, vp);
            --k;
        }
        list.set(k, key);
        if (LAST && n == cap) top = list.get(n - 1);
    }
};

// Blends a ray's list of n front to back, colour from the SH at the ray direction,
// into o[0..2].
template <typename T, int DEG, class List>
__device__ __forceinline__ void blend_hits(const List& list, int n, const float4* __restrict__ gauss,
                                           const T* __restrict__ sh, const Ray& r, float* o) {
    constexpr int NC = (DEG + 1) * (DEG + 1);
    float Y[16];
    sh_basis<DEG>(r.dx, r.dy, r.dz, Y);
    float tr = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;  // transmittance, colour
    for (int k = 0; k < n; ++k) {
        float t;
        const int64_t g = int64_t(uint32_t(list.get(k)));
        const float a = rc_alpha(gauss, g, r.ox, r.oy, r.oz, r.dx, r.dy, r.dz, t);
        const float tn = tr * (1.f - a);
        if (tn < 1e-4f) break;
        float col[3];
        sh_colour<T, DEG>(sh + g * (3 * NC), Y, col);
        const float w = a * tr;
        c0 = fmaf(w, col[0], c0);
        c1 = fmaf(w, col[1], c1);
        c2 = fmaf(w, col[2], c2);
        tr = tn;
    }
    o[0] = c0;
    o[1] = c1;
    o[2] = c2;
}

// Traversal of the 8-wide tree is by the whole warp: its rays share a camera
// centre and nearly a direction, so they need nearly the same nodes.  A
// warp-shared stack holds {node or leaf reference, the lanes whose ray hit
// its box}; a popped node is loaded once for the warp, every lane tests its
// ray against the eight child boxes (a child beyond the lane's full list does
// not count as hit), and the children hit by any lane are pushed farthest
// first by their nearest entry over those lanes.  A leaf is tested by the
// lanes that hit it.  At most 7 entries a level plus 8 are pending (the
// tree's depth is checked against kMaxWideDepth when it is built; the guard
// only keeps the stack in bounds).  Every lane reaches every warp-wide
// synchronisation point: the loop's trip count and the branch between leaf
// and node are the same for the whole warp.
template <typename T, int DEG>
__global__ void __launch_bounds__(kTraceThreads)
rc_trace_kernel(const float4* __restrict__ gauss, const RayNode* __restrict__ nodes,
                int64_t n, const T* __restrict__ sh, const uint32_t* __restrict__ ray_view,
                const uint32_t* __restrict__ ray_pix, const int2* __restrict__ order,
                int64_t n_rays, const Cam* __restrict__ cams, float focal, float half_w,
                float half_h, int heap_cap, float* __restrict__ raycol,
                const uint32_t* __restrict__ gate) {
    if (gate && *gate == 0u) return;
    __shared__ uint32_t s_ref[kTraceWarps][kRayStack];
    __shared__ uint32_t s_lanes[kTraceWarps][kRayStack];
    __shared__ unsigned long long s_head[kTraceWarps][kListHead][32];  // [slot][lane]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const bool valid = i0 < n_rays;
    const int64_t i = valid ? i0 : n_rays - 1;  // lanes past the end follow the last ray, unwritten
    // thread i casts ray order[i].y: the rays grouped by (view, tile) and
    // Morton-ordered inside a tile
    const int64_t r = order ? int64_t(order[i].y) : i;
    const Ray ray = make_ray(cams[ray_view[r]], ray_pix[r], focal, half_w, half_h);
    const float dx = ray.dx, dy = ray.dy, dz = ray.dz;
    const float ox = ray.ox, oy = ray.oy, oz = ray.oz;
    const float ix = 1.f / dx, iy = 1.f / dy, iz = 1.f / dz;
    unsigned long long rest[kMaxHeap - kListHead];
    RayHits<WalkList, false> hits;
    hits.list = {&s_head[warp][0][lane], rest};
    hits.cap = heap_cap;
    uint32_t* const st_ref = s_ref[warp];
    uint32_t* const st_lanes = s_lanes[warp];
    const unsigned all = __ballot_sync(0xffffffffu, valid);
    if (lane == 0) {
        st_ref[0] = 0u;  // the root
        st_lanes[0] = all;
    }
    int sp = all ? 1 : 0;
    __syncwarp();
    while (sp > 0) {
        --sp;
        const uint32_t e = st_ref[sp];
        const bool mine = (st_lanes[sp] >> lane) & 1u;
        __syncwarp();
        const float bound = hits.bound();
        if (e & kRayLeafBit) {  // leaf: Gaussians first .. first + count - 1
            if (mine) {
                const uint32_t first = (e & ~kRayLeafBit) >> 3, cnt = (e & 7u) + 1u;
                // the leaf's Gaussians evaluated together (their loads in
                // flight at once), then taken in order
                for (uint32_t base = 0; base < cnt; base += kLeafMax) {
                    float al[kLeafMax], tl[kLeafMax];
#pragma unroll
                    for (int q = 0; q < kLeafMax; ++q) {
                        al[q] = 0.f;
                        tl[q] = 0.f;
                        if (base + q < cnt)
                            al[q] = rc_alpha(gauss, first + base + q, ox, oy, oz, dx, dy, dz, tl[q]);
                    }
#pragma unroll
                    for (int q = 0; q < kLeafMax; ++q) {
                        if (base + q >= cnt) break;
                        hits.add(al[q], tl[q], first + base + q);
                    }
                }
            }
        } else {  // wide node: its children, nearest first
            const float4* nf = reinterpret_cast<const float4*>(nodes + e);
            float te[8];
            uint32_t chv[8];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float4 a0 = __ldg(nf + q), a1 = __ldg(nf + 2 + q), a2 = __ldg(nf + 4 + q);
                const float4 a3 = __ldg(nf + 6 + q), a4 = __ldg(nf + 8 + q), a5 = __ldg(nf + 10 + q);
                const uint4 c4 = __ldg(reinterpret_cast<const uint4*>(nf + 12 + q));
                const float lxa[4] = {a0.x, a0.y, a0.z, a0.w}, lya[4] = {a1.x, a1.y, a1.z, a1.w};
                const float lza[4] = {a2.x, a2.y, a2.z, a2.w}, hxa[4] = {a3.x, a3.y, a3.z, a3.w};
                const float hya[4] = {a4.x, a4.y, a4.z, a4.w}, hza[4] = {a5.x, a5.y, a5.z, a5.w};
                const uint32_t ca[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    chv[4 * q + k] = ca[k];
                    float t = INFINITY;
                    if (mine && ca[k] != kRayNoChild) {
                        t = slab_enter(make_float4(lxa[k], lya[k], lza[k], 0.f),
                                       make_float4(hxa[k], hya[k], hza[k], 0.f), ox, oy, oz, ix, iy,
                                       iz);
                        if (t > bound) t = INFINITY;  // beyond a full list
                    }
                    te[4 * q + k] = t;
                }
            }
            // children hit by any lane, with their nearest entry (t >= 0:
            // the bits order like the values)
            uint32_t hit[8], near[8];
            int m = 0;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const bool h = te[c] < INFINITY;
                hit[c] = __ballot_sync(0xffffffffu, h);
                near[c] = __reduce_min_sync(0xffffffffu,
                                            h ? __float_as_uint(fmaxf(te[c], 0.f)) : 0xFFFFFFFFu);
                m += hit[c] ? 1 : 0;
            }
            if (sp + m > kRayStack) m = 0;  // cannot happen (depth checked); keeps the stack in bounds
            if (lane < 8 && m > 0) {
                // farthest first: lane c places child c by its rank in
                // descending entry (ties by child position)
                uint32_t my_hit = 0u, my_near = 0u, my_ref = 0u;
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    if (c == lane) {
                        my_hit = hit[c];
                        my_near = near[c];
                        my_ref = chv[c];
                    }
                }
                if (my_hit) {
                    int rank = 0;
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        rank += (hit[c] && (near[c] > my_near || (near[c] == my_near && c < lane)));
                    st_ref[sp + rank] = my_ref;
                    st_lanes[sp + rank] = my_hit;
                }
            }
            sp += m;
            __syncwarp();
        }
    }
    // colours in thread order: the grouped order when `order` is given
    if (valid) blend_hits<T, DEG>(hits.list, hits.n, gauss, sh, ray, raycol + 3 * i);
}

// ---- rays cast through tile lists ------------------------------------------
// The rays of a (view, tile) group against the Gaussians whose alpha >= 1/255
// outline reaches the tile (launch_project_outline), which is the set the
// tree's walk would find, without the walk.  A warp owns a group: it sorts
// the list by the hits' least depth, up to kCastCap keys at a time, streams
// the records 32 at a time (cp.async, one batch ahead), tests each record's
// outline against all of the warp's rays (a lane a record, as in the
// compositing kernels: packed FMAs and ballots), and each lane takes its own
// candidates through the exact rc_alpha into its list.  In depth order a ray
// finds its hits nearly sorted, and a list ends for the warp once every ray's
// bound lies before the next record's least depth.  The lists only say which
// Gaussians are tested and in which order, so a ray's intersections are the
// tree walk's.  (Gaussians thinner than about 400 : 1 apart: the FP32 test then
// also passes points that 64 bits put below 1/255, and of those the lists hold
// what lies inside the outline.)
//
// Bound by the latency of the candidates' evaluation and insertion at half the
// lanes (rays have different numbers of candidates in a batch).  1080p frame,
// 200k Gaussians, c_h 128: 3.8 ms, of which outlines and keys 0.23, cast 2.4,
// blend 1.2; the tree walk takes 10.0 ms.
constexpr int kCastCap = 512;
constexpr int kCastWarps = 4;
constexpr int kCastBlocks = 4;  // resident blocks an SM
constexpr int kCastSlots = 2;  // record batches: one evaluated, the next in flight

__device__ __forceinline__ void cast_copy16(void* smem, const void* gmem) {
    const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}

union CastSmem {
    WarpSort<kCastCap> s;
    struct {
        uint32_t idx[kCastCap];
        float4 rec[kCastSlots][2][32];    // outlines
        float4 gauss[kCastSlots][3][32];  // rc_prepare_kernel's data
        float4 rx[8], ry[8];              // the rays' pixels about their box centre
        uint4 mask[8];                    // per ray, its candidates in the batch
    } c;
};

// First entry of work ({group, ray begin, ray end, -}, ascending rays) whose
// rays begin at or after ray r.
__device__ __forceinline__ int64_t first_work(const int4* __restrict__ work, int64_t n, int64_t r) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (int64_t(__ldg(&work[mid].y)) < r) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__global__ void __launch_bounds__(kCastWarps * 32, 5) rc_cast_kernel(CastParams P) {
    if (P.skip && *P.skip) return;
    extern __shared__ __align__(16) unsigned char cast_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CastSmem& W = reinterpret_cast<CastSmem*>(cast_smem)[warp];
    const uint32_t* __restrict__ first =
        P.slices.use_alt && *P.slices.use_alt ? P.slices.start_alt : P.slices.start;
    const int64_t n_warps = int64_t(gridDim.x) * kCastWarps;
    const int64_t w_end = first_work(P.work, P.n_work, P.ray0 + P.chunk);
    int64_t item = first_work(P.work, P.n_work, P.ray0) + int64_t(blockIdx.x) * kCastWarps + warp;
    const int64_t claim0 = item - (int64_t(blockIdx.x) * kCastWarps + warp) + n_warps;
    while (item < w_end) {
        uint32_t claim = 0;
        if (lane == 0) claim = atomicAdd(P.claimed, 1u) + 1u;  // from -1 on
        const int4 wi = __ldg(P.work + item);
        const uint32_t start = first[wi.x], end = P.slices.cursor[wi.x];
        const int view = wi.x / P.ntiles;
        const Cam& cam = P.cams[view];
        const int64_t vbase = int64_t(view) * P.n;
        for (int r0 = wi.y; r0 < wi.z; r0 += 32) {
            const int rid = r0 + lane;
            const bool active = rid < wi.z;
            const uint32_t pixel = uint32_t(P.grouped[active ? rid : wi.z - 1].x);
            const Ray ray = make_ray(cam, pixel, P.focal, P.half_w, P.half_h);
            const int col = int(pixel & 0xFFFFu), row = int(pixel >> 16);
            const int c0x = __reduce_min_sync(0xffffffffu, col), c1x = __reduce_max_sync(0xffffffffu, col);
            const int r0y = __reduce_min_sync(0xffffffffu, row), r1y = __reduce_max_sync(0xffffffffu, row);
            const float ox = 0.5f * float(c0x + c1x), oy = 0.5f * float(r0y + r1y);
            // 1 + a margin for the rounding of the test below: with the rays'
            // box of diagonal d, a ray inside an outline is at most sqrt(e) + d
            // pixels (and the box's centre at most that) from the outline's
            // centre, e the largest of E, so the terms are at most that squared
            // over E's floor 0.5 + 2e-5 e, i.e. below 2 d^2 + 5e4.  Six roundings
            // of 2^-24 of that, at least the 0.02 of a 32 x 32 tile (a search of
            // 20 million outlines against 64 bits found 1.25 at most).
            const float dw = float(c1x - c0x), dh = float(r1y - r0y);
            const float inside = 1.f + fmaxf(0.02f, fmaf(dw * dw + dh * dh, 7.2e-7f, 0.018f));
            // lanes past the group's rays add nothing (their rays are not open)
            RayHits<CastList, true> hits;
            hits.list = {P.hits + (rid - P.ray0), P.chunk + kCastSpill};
            hits.cap = P.heap_cap;
            for (uint32_t c0 = start; c0 < end; c0 += kCastCap) {
                const int len = int(min(end - c0, uint32_t(kCastCap)));
                warp_sort<kCastCap>(P.keys, c0, len, W.s);
                for (int base = 0; base < len; base += 32) {  // low words in place of the keys
                    const int i = base + lane;
                    const uint32_t lo = i < len ? uint32_t(W.s.sk[i]) >> 4 : 0u;
                    __syncwarp();
                    if (i < len) W.c.idx[i] = lo;
                    __syncwarp();
                }
                reinterpret_cast<float*>(W.c.rx)[lane] = active ? float(col) - ox : 1e18f;
                reinterpret_cast<float*>(W.c.ry)[lane] = active ? float(row) - oy : 1e18f;
                const int nbatch = (len + 31) / 32;
                auto issue = [&](int b) {
                    const int i = b * 32 + lane, slot = b % kCastSlots;
                    if (i < len) {
                        const int64_t g = W.c.idx[i];
                        const float4* r = P.rec + kRecordFloat4 * (vbase + g);
                        cast_copy16(&W.c.rec[slot][0][lane], r);
                        cast_copy16(&W.c.rec[slot][1][lane], r + 1);
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            cast_copy16(&W.c.gauss[slot][k][lane], P.gauss + 3 * g + k);
                    }
                    asm volatile("cp.async.commit_group;\n" ::: "memory");
                };
                issue(0);
                for (int b = 0; b < nbatch; ++b) {
                    issue(b + 1);  // an empty group past the end
                    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
                    __syncwarp();
                    const int slot = b % kCastSlots, n = min(32, len - b * 32);
                    // the batch's least depth against what the rays still keep
                    const bool open = active && !(hits.bound() < W.c.rec[slot][1][0].y);
                    const unsigned act = __ballot_sync(0xffffffffu, open);
                    if (act == 0u) break;
                    float A = 0.f, B = 0.f, C = 0.f, D = 0.f, E = 0.f, F = -1e30f;
                    if (lane < n) {
                        // 1 + the outline's quadratic, expanded about (ox, oy),
                        // and the margin
                        const float4 q0 = W.c.rec[slot][0][lane];
                        const float du = q0.x - (ox - P.half_w), dv = q0.y - (oy - P.half_h);
                        A = q0.z;
                        B = q0.w;
                        C = W.c.rec[slot][1][lane].x;
                        D = -fmaf(2.f * A, du, B * dv);
                        E = -fmaf(2.f * C, dv, B * du);
                        F = fmaf(du, fmaf(A, du, B * dv), C * dv * dv) + inside;
                    }
                    const float2 A2 = make_float2(A, A), B2 = make_float2(B, B), C2 = make_float2(C, C);
                    const float2 D2 = make_float2(D, D), E2 = make_float2(E, E), F2 = make_float2(F, F);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        if (!((act >> (4 * q)) & 0xFu)) continue;
                        const float4 qx = W.c.rx[q], qy = W.c.ry[q];
                        unsigned m[4];
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const float2 x = k ? make_float2(qx.z, qx.w) : make_float2(qx.x, qx.y);
                            const float2 y = k ? make_float2(qy.z, qy.w) : make_float2(qy.x, qy.y);
                            const float2 t1 = __ffma2_rn(A2, x, __ffma2_rn(B2, y, D2));
                            const float2 v =
                                __ffma2_rn(x, t1, __ffma2_rn(y, __ffma2_rn(C2, y, E2), F2));
                            m[2 * k] = __ballot_sync(0xffffffffu, v.x >= 0.f);
                            m[2 * k + 1] = __ballot_sync(0xffffffffu, v.y >= 0.f);
                        }
                        if (lane == 0) W.c.mask[q] = make_uint4(m[0], m[1], m[2], m[3]);
                    }
                    __syncwarp();
                    unsigned mine = open ? reinterpret_cast<const unsigned*>(W.c.mask)[lane] : 0u;
                    while (mine) {
                        // two candidates evaluated together, taken in order
                        const int s1 = __ffs(mine) - 1;
                        mine &= mine - 1u;
                        const bool two = mine != 0u;
                        const int s2 = two ? __ffs(mine) - 1 : s1;
                        mine &= mine - 1u;
                        float t1, t2;
                        const float a1 = rc_alpha(&W.c.gauss[slot][0][s1], &W.c.gauss[slot][1][s1],
                                                  &W.c.gauss[slot][2][s1], ray.ox, ray.oy, ray.oz,
                                                  ray.dx, ray.dy, ray.dz, t1);
                        const float a2 = rc_alpha(&W.c.gauss[slot][0][s2], &W.c.gauss[slot][1][s2],
                                                  &W.c.gauss[slot][2][s2], ray.ox, ray.oy, ray.oz,
                                                  ray.dx, ray.dy, ray.dz, t2);
                        hits.add(a1, t1, W.c.idx[b * 32 + s1]);
                        if (two) hits.add(a2, t2, W.c.idx[b * 32 + s2]);
                    }
                    __syncwarp();  // the slot and the masks are written again
                }
                asm volatile("cp.async.wait_group 0;\n" ::: "memory");
                __syncwarp();  // the next chunk's keys take the space
            }
            if (active) P.count[rid - P.ray0] = hits.n;
        }
        item = claim0 + int64_t(__shfl_sync(0xffffffffu, claim, 0));
    }
}

constexpr int kBlendThreads = 256;

// Four lanes of a warp blend a ray's list four intersections at a time.  Lane q
// evaluates intersection k + q; the lanes step the transmittance through the
// four together, in order.  Each intersection's SH coefficients are then read
// by all four lanes, 64 contiguous bytes a load (lane q takes the 16-byte
// pieces q, q + 4, ...), and the four lanes' partial sums are reduced so that
// lane q ends with the colour of its own intersection.  Float f of a row
// belongs to channel f mod 3: lane q's sum s holds channel (s + q V) mod 3, V the
// floats of a piece, and the exchanges pick the matching sum of the partner.
template <typename T, int DEG>
__device__ __forceinline__ void blend_quads(const CastList& list, int n, const float4* __restrict__ gauss,
                                            const T* __restrict__ sh, const Ray& r, float* o) {
    constexpr int NC = (DEG + 1) * (DEG + 1), NP = sh_pieces<T, DEG>(), V = 16 / int(sizeof(T));
    constexpr int R = (NP + 3) / 4;  // pieces a lane
    const int lane = threadIdx.x & 31, q = lane & 3, quad = lane & ~3;
    float Y[16];
    sh_basis<DEG>(r.dx, r.dy, r.dz, Y);
    float y[R][V];  // the basis values of the lane's floats
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int e = 0; e < V; ++e) {
            y[i][e] = 0.f;
#pragma unroll
            for (int l = 0; l < 4; ++l)
                if (l + 4 * i < NP && q == l) y[i][e] = Y[((l + 4 * i) * V + e) / 3];
        }
    float tr = 1.f, c[3] = {0.f, 0.f, 0.f};
    bool live = n > 0;
    uint32_t g = q < n ? uint32_t(list.get(q)) : 0u;
    for (int k = 0; __any_sync(0xffffffffu, live); k += 4) {
        const uint32_t next = live && k + 4 + q < n ? uint32_t(list.get(k + 4 + q)) : 0u;
        float a = 0.f, t;
        if (live && k + q < n) a = rc_alpha(gauss, g, r.ox, r.oy, r.oz, r.dx, r.dy, r.dz, t);
        float w = 0.f;
        uint32_t used = 0u;  // the intersections that are blended
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float ah = __shfl_sync(0xffffffffu, a, quad + h);
            const float tn = tr * (1.f - ah);
            live = live && k + h < n && !(tn < 1e-4f);
            if (live) {
                if (q == h) w = ah * tr;
                tr = tn;
                used |= 1u << h;
            }
        }
        float acc[4][3];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const int64_t gh = __shfl_sync(0xffffffffu, g, quad + h);
            acc[h][0] = acc[h][1] = acc[h][2] = 0.f;
            if ((used >> h) & 1u) {
                const uint4* row = reinterpret_cast<const uint4*>(sh + gh * (3 * NC)) + q;
                uint4 raw[R];
#pragma unroll
                for (int i = 0; i < R; ++i)
                    raw[i] = q + 4 * i < NP ? __ldg(row + 4 * i) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    T v[V];
                    memcpy(v, &raw[i], 16);
#pragma unroll
                    for (int e = 0; e < V; ++e)
                        acc[h][(4 * i * V + e) % 3] = fmaf(y[i][e], to_f(v[e]), acc[h][(4 * i * V + e) % 3]);
                }
            }
        }
        // lanes 0 and 1 keep intersections k and k + 1, lanes 2 and 3 the others;
        // then an even lane the first of its two
        constexpr int D2 = 2 * V % 3, D1 = V % 3;
        const bool hi = q & 2, odd = q & 1;
        float two[2][3], col[3];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const float send = hi ? acc[h][(s + 3 - D2) % 3] : acc[h + 2][(s + D2) % 3];
                two[h][s] = (hi ? acc[h + 2][s] : acc[h][s]) + __shfl_xor_sync(0xffffffffu, send, 2);
            }
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const float send = odd ? two[0][(s + 3 - D1) % 3] : two[1][(s + D1) % 3];
            col[s] = (odd ? two[1][s] : two[0][s]) + __shfl_xor_sync(0xffffffffu, send, 1);
            c[s] = fmaf(w, fmaxf(col[s] + 0.5f, 0.f), c[s]);
        }
        g = next;
    }
    // the lanes' colours, by channel, added up; lane q < 3 writes channel q
    const int turn = q * V % 3;  // sum s is channel (s + turn) mod 3
    float out = 0.f;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
        const float mine = turn == 0 ? c[ch] : turn == 1 ? c[(ch + 2) % 3] : c[(ch + 1) % 3];
        float sum = mine + __shfl_xor_sync(0xffffffffu, mine, 2);
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        if (q == ch) out = sum;
    }
    if (n >= 0 && q < 3) o[q] = out;
}

// Blends the lists that rc_cast_kernel found for a chunk's rays (count >= 0: a
// ray of this chunk).  A kernel of its own: what it needs is the first-level
// cache (neighbouring rays, and the views of a tile, blend nearly the same
// Gaussians) and many warps in flight, where the cast needs shared memory; at
// the end of the cast's own loop, with little of that cache left, the blending
// took 3.4 of 5.7 ms at 1080p.  It is bound by the cache lines its gathers look
// up: a thread a ray looks up to 32 lines for each of 15 loads a step, four
// lanes a ray (blend_quads, where the coefficients come in whole 16-byte pieces)
// 32 for three of them and 8 for the twelve others.  1080p, 200k Gaussians, FP32
// SH3, c_h 128: 1.66 -> 1.16 ms.
template <typename T, int DEG>
__global__ void __launch_bounds__(kBlendThreads) rc_blend_kernel(CastParams P, const T* __restrict__ sh) {
    if (P.skip && *P.skip) return;
    constexpr bool kQuads = sh_pieces<T, DEG>() > 0;
    const int64_t tid = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int64_t j = kQuads ? tid >> 2 : tid;
    const bool in = j < P.chunk + kCastSpill;
    const int n = in ? P.count[j] : -1;
    if (kQuads ? __all_sync(0xffffffffu, n < 0) : n < 0) return;
    const int64_t jj = n < 0 ? 0 : j;  // (a lane without a ray blends nothing)
    const int64_t i = P.ray0 + (n < 0 ? 0 : j);
    const int2 order = P.grouped[i];
    const Ray ray = make_ray(P.cams[P.ray_view[order.y]], uint32_t(order.x), P.focal, P.half_w, P.half_h);
    const CastList list{P.hits + jj, P.chunk + kCastSpill};
    if constexpr (kQuads)
        blend_quads<T, DEG>(list, n, P.gauss, sh, ray, P.raycol + 3 * i);
    else
        blend_hits<T, DEG>(list, n, P.gauss, sh, ray, P.raycol + 3 * i);
}
// lanes a ray
template <typename T, int DEG>
constexpr int blend_lanes() { return sh_pieces<T, DEG>() > 0 ? 4 : 1; }

int grid_of(int64_t n, int block) {
    int64_t g = (n + block - 1) / block;
    const int64_t cap = int64_t(num_sms()) * 64;
    if (g > cap) g = cap;
    return int(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t launch_raycast_prepare(int dtype, const void* const* attrs, int64_t n, float4* gauss,
                                   float4* gbox, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int grid = grid_of(n, 256);
    if (dtype == 1) {
        GaussiansView<__nv_bfloat16> G{static_cast<const float*>(attrs[0]),
                                       static_cast<const __nv_bfloat16*>(attrs[1]),
                                       static_cast<const __nv_bfloat16*>(attrs[2]),
                                       static_cast<const __nv_bfloat16*>(attrs[3]),
                                       static_cast<const __nv_bfloat16*>(attrs[4])};
        rc_prepare_kernel<<<grid, 256, 0, s>>>(G, n, gauss, gbox);
    } else if (dtype == 2) {
        GaussiansView<__half> G{static_cast<const float*>(attrs[0]), static_cast<const __half*>(attrs[1]),
                                static_cast<const __half*>(attrs[2]), static_cast<const __half*>(attrs[3]),
                                static_cast<const __half*>(attrs[4])};
        rc_prepare_kernel<<<grid, 256, 0, s>>>(G, n, gauss, gbox);
    } else {
        GaussiansView<float> G{static_cast<const float*>(attrs[0]), static_cast<const float*>(attrs[1]),
                               static_cast<const float*>(attrs[2]), static_cast<const float*>(attrs[3]),
                               static_cast<const float*>(attrs[4])};
        rc_prepare_kernel<<<grid, 256, 0, s>>>(G, n, gauss, gbox);
    }
    return cudaGetLastError();
}

// Build scratch: binary nodes, two task lists, the SAH sweep's areas, the
// counters and two collapse queues.
struct BuildScratch {
    BinNode* bins;
    BuildTask* tasks[2];
    float* sal;
    uint32_t* counters;
    CollapseTask* queue[2];
};
static size_t task_cap(int64_t n) { return size_t(n / (kLeafMax + 1) + 2); }
static BuildScratch carve_build(void* tmp, int64_t n) {
    BuildScratch b;
    char* p = static_cast<char*>(tmp);
    auto take = [&](size_t bytes) {
        char* q = p;
        p += (bytes + 255) & ~size_t(255);
        return q;
    };
    b.bins = reinterpret_cast<BinNode*>(take(sizeof(BinNode) * size_t(n + 1)));
    b.tasks[0] = reinterpret_cast<BuildTask*>(take(sizeof(BuildTask) * task_cap(n)));
    b.tasks[1] = reinterpret_cast<BuildTask*>(take(sizeof(BuildTask) * task_cap(n)));
    b.sal = reinterpret_cast<float*>(take(sizeof(float) * size_t(n + 1)));
    b.counters = reinterpret_cast<uint32_t*>(take(64));
    b.queue[0] = reinterpret_cast<CollapseTask*>(take(sizeof(CollapseTask) * size_t(n + 1)));
    b.queue[1] = reinterpret_cast<CollapseTask*>(take(sizeof(CollapseTask) * size_t(n + 1)));
    return b;
}

size_t raycast_build_tmp_bytes(int64_t n) {
    const size_t r = 255;
    auto up = [&](size_t x) { return (x + r) & ~r; };
    return up(sizeof(BinNode) * size_t(n + 1)) + 2 * up(sizeof(BuildTask) * task_cap(n)) +
           up(sizeof(float) * size_t(n + 1)) + up(64) + 2 * up(sizeof(CollapseTask) * size_t(n + 1));
}

cudaError_t raycast_build_binary(const float4* gbox, int64_t n, void* tmp, int64_t* n_bin,
                                 cudaStream_t s) {
    *n_bin = 0;
    if (n <= kLeafMax) return cudaSuccess;
    BuildScratch b = carve_build(tmp, n);
    uint32_t h[16] = {1u, 0u};  // the root is node 0
    cudaError_t e = cudaMemcpyAsync(b.counters, h, sizeof(h), cudaMemcpyHostToDevice, s);
    const BuildTask root{0u, uint32_t(n), 0u, 0u};
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.tasks[0], &root, sizeof(root), cudaMemcpyHostToDevice, s);
    uint32_t n_tasks = 1;
    int cur = 0;
    while (e == cudaSuccess && n_tasks > 0) {
        sah_split_kernel<<<n_tasks, kBuildThreads, 0, s>>>(b.tasks[cur], gbox, b.sal, b.bins,
                                                           b.tasks[cur ^ 1], b.counters);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, b.counters, 8, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = cudaMemsetAsync(b.counters + 1, 0, 4, s);
        n_tasks = h[1];
        cur ^= 1;
    }
    *n_bin = int64_t(h[0]);
    return e;
}

cudaError_t raycast_collapse(const float4* gbox, int64_t n, void* tmp, int64_t n_bin,
                             RayNode* nodes, int64_t* n_wide, int* depth, cudaStream_t s) {
    *n_wide = 1;
    *depth = 0;
    if (n_bin == 0) {
        leaf_root_kernel<<<1, 32, 0, s>>>(gbox, uint32_t(n > 0 ? n : 0), nodes);
        cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
    }
    BuildScratch b = carve_build(tmp, n);
    uint32_t h[16] = {0u};
    h[2] = 1u;  // the wide root is node 0
    cudaError_t e = cudaMemcpyAsync(b.counters, h, sizeof(h), cudaMemcpyHostToDevice, s);
    const CollapseTask root{0u, 0u, 0u, 0u};
    if (e == cudaSuccess) e = cudaMemcpyAsync(b.queue[0], &root, sizeof(root), cudaMemcpyHostToDevice, s);
    uint32_t nq = 1;
    int cur = 0;
    while (e == cudaSuccess && nq > 0) {
        collapse_kernel<<<grid_of(nq, 128), 128, 0, s>>>(b.queue[cur], nq, b.bins, gbox, nodes,
                                                         b.queue[cur ^ 1], b.counters);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(h, b.counters, 32, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e == cudaSuccess) e = cudaMemsetAsync(b.counters + 3, 0, 4, s);
        nq = h[3];
        cur ^= 1;
    }
    *n_wide = int64_t(h[2]);
    *depth = int(h[4]);
    return e;
}

cudaError_t launch_raycast(int dtype, int sh_degree, const float4* gauss, const RayNode* nodes,
                           int64_t n, const void* sh, const uint32_t* ray_view,
                           const uint32_t* ray_pix, const int2* order, int64_t n_rays,
                           const Cam* cams, float focal, float half_w, float half_h, int heap_cap,
                           float* raycol, const uint32_t* gate, cudaStream_t s) {
    if (n_rays <= 0) return cudaSuccess;
    const unsigned grid = unsigned((n_rays + kTraceThreads - 1) / kTraceThreads);
#define DL_RC(T, D)                                                                          \
    rc_trace_kernel<T, D><<<grid, kTraceThreads, 0, s>>>(gauss, nodes, n, static_cast<const T*>(sh),   \
                                               ray_view, ray_pix, order, n_rays, cams, focal,  \
                                               half_w, half_h, heap_cap, raycol, gate)
#define DL_RC_DEG(T)                  \
    switch (sh_degree) {              \
        case 0: DL_RC(T, 0); break;   \
        case 1: DL_RC(T, 1); break;   \
        case 2: DL_RC(T, 2); break;   \
        default: DL_RC(T, 3); break;  \
    }
    if (dtype == 1) {
        DL_RC_DEG(__nv_bfloat16)
    } else if (dtype == 2) {
        DL_RC_DEG(__half)
    } else {
        DL_RC_DEG(float)
    }
#undef DL_RC
    return cudaGetLastError();
}

size_t cast_tmp_bytes(int64_t chunk, int heap_cap) {
    const size_t rays = size_t(chunk + kCastSpill);
    return 8 * rays * size_t(heap_cap) + 4 * rays + 256;
}

namespace {
template <typename T, int DEG>
cudaError_t launch_cast(CastParams p, int64_t n_rays, void* tmp, const void* sh, cudaStream_t s) {
    const size_t smem = kCastWarps * sizeof(CastSmem);
    cudaError_t e = cudaFuncSetAttribute(rc_cast_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(smem));
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rc_cast_kernel, kCastWarps * 32, smem);
    if (e != cudaSuccess) return e;
    // kCastBlocks an SM (fewer than fit): the rays' lists and the keys need the
    // rest as first-level cache (six blocks 4.43, five 4.42, four 4.30 ms)
    if (per_sm > kCastBlocks) per_sm = kCastBlocks;
    e = cudaFuncSetAttribute(rc_cast_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             int(100 * kCastBlocks * (smem + 1024) / (228 * 1024)) + 1);
    if (e != cudaSuccess) return e;
    const int64_t need = (p.n_work + kCastWarps - 1) / kCastWarps;
    const int64_t fit = int64_t(num_sms()) * (per_sm > 0 ? per_sm : 1);
    const int64_t rays = p.chunk + kCastSpill;
    p.hits = static_cast<unsigned long long*>(tmp);
    p.count = reinterpret_cast<int32_t*>(p.hits + rays * p.heap_cap);
    p.claimed = reinterpret_cast<uint32_t*>(p.count + rays);
    for (p.ray0 = 0; p.ray0 < n_rays; p.ray0 += p.chunk) {
        // counts and the claim counter start at -1
        e = cudaMemsetAsync(p.count, 0xFF, 4 * size_t(rays + 1), s);
        if (e != cudaSuccess) return e;
        rc_cast_kernel<<<unsigned(need < fit ? need : fit), kCastWarps * 32, smem, s>>>(p);
        rc_blend_kernel<T, DEG><<<unsigned((rays * blend_lanes<T, DEG>() + kBlendThreads - 1) / kBlendThreads),
                                  kBlendThreads, 0, s>>>(p, static_cast<const T*>(sh));
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
}  // namespace

cudaError_t launch_raycast_lists(int dtype, int sh_degree, const CastParams& p, int64_t n_rays,
                                 void* tmp, const void* sh, cudaStream_t s) {
    if (p.n_work <= 0 || n_rays <= 0) return cudaSuccess;
#define DL_RC(T, D) return launch_cast<T, D>(p, n_rays, tmp, sh, s)
    if (dtype == 1) {
        DL_RC_DEG(__nv_bfloat16)
    } else if (dtype == 2) {
        DL_RC_DEG(__half)
    } else {
        DL_RC_DEG(float)
    }
#undef DL_RC
#undef DL_RC_DEG
    return cudaErrorInvalidValue;
}

}  // namespace dl
