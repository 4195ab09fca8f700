// kernels_receivers.cu -- the receivers' 4-wide tree built on the device.
//
// Moving receivers upload a new set for every step, so the build is part of each call: the host
// builder (binned surface-area heuristic, host_geometry.cpp) took 0.8 of a street walk's 1.95 ms
// with 4,096 receivers, nearly all of it in the search for splits.  Here every segment of the points
// is split at its median, so segment i of binary level L always holds the places
// [n i / 2^L, n (i + 1) / 2^L) and every node's place in memory follows from n alone.  Only the
// axis is searched: the one whose halves' boxes have the least area.  Receivers along streets make
// that matter: with the widest axis instead, the boxes that a line through the scene meets are 1.5
// times as many (a large city's trace 13.07 -> 13.50 ms); with the least area 1.04 times.
// Two binary levels make one level of 4-wide nodes.
//   - rx_split_kernel, one launch per binary level while segments are longer than kRxSub: a
//     point's place is its rank in its segment on each axis, counted against all of the segment's
//     keys.  That is 6 n^2 comparisons in all, but spread over the chip with no barrier other than
//     the launches.  The three orders are written out; the next launch reads the chosen one.
//   - rx_subtree_kernel: a block takes one segment of at most kRxSub points in shared memory down
//     to the leaves.
// 4,096 receivers: five splits of 17, 14, 11, 7 and 8 us and the subtrees' 29 (launches timed
// alone), bound by the comparisons' issue at first and by the loads' and barriers' latency after;
// the upload 910 -> 111 us.
#include "sbr_device.cuh"
#include "sbr_internal.h"
#include "stream_launch.cuh"

namespace sbr {
namespace {

// 32 points a block and their comparisons over its warps: 4,096 points are 128 blocks.  (256 points
// a block, one per thread, were 16 blocks: the whole upload 268 us.)  8 / 16 / 32 warps: 4,096
// receivers 124 / 111 / 106 us, 65,536 4.41 / 4.49 / 5.03 ms.
constexpr int kSplitWarps = 16;
constexpr int kRxSub = 128;   // 32, 64 and 256 measured the same within 1 us
// Points per leaf at most: with 1 the same times, with 4 (a level of nodes less, four tests for a
// visit) the traces of the office and the canyon ran 1 % longer.
constexpr int kRxLeaf = 2;

struct RxBuild {
    float4 *nodes4;
    int n, level, last;   // this launch's binary level; the leaves' level (even)
};

__host__ __device__ __forceinline__ int rx_bound(int n, int level, int i) { return (int)(((long long)n * i) >> level); }
// id of the node of (even) level's segment i: the levels' nodes follow one another
__host__ __device__ __forceinline__ int rx_node(int level, int i) { return (int)(((1LL << level) - 1) / 3) + i; }

struct RxBox {
    float lo[3], hi[3];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int a = 0; a < 3; ++a) lo[a] = INFINITY, hi[a] = -INFINITY;
    }
    __device__ __forceinline__ void grow(const float4 &p) {
        lo[0] = fminf(lo[0], p.x), lo[1] = fminf(lo[1], p.y), lo[2] = fminf(lo[2], p.z);
        hi[0] = fmaxf(hi[0], p.x), hi[1] = fmaxf(hi[1], p.y), hi[2] = fmaxf(hi[2], p.z);
    }
    __device__ __forceinline__ float widest() const { return max3f(hi[0] - lo[0], hi[1] - lo[1], hi[2] - lo[2]); }
    // half the surface, each side longer by pad: cones meet boxes grown by their radius, and the
    // halves of a line or a point have areas to compare only so
    __device__ __forceinline__ float area(float pad) const {
        const float x = hi[0] - lo[0] + pad, y = hi[1] - lo[1] + pad, z = hi[2] - lo[2] + pad;
        return x * y + y * z + z * x;
    }
};
constexpr float kRxPad = 1.0f / 256.0f;   // of the segment's widest extent

__device__ __forceinline__ int best_axis(float cx, float cy, float cz) {
    return cx <= cy && cx <= cz ? 0 : (cy <= cz ? 1 : 2);
}

// The box of segment i of an even level into its parent's slot.
__device__ void put_child4(const RxBuild &b, int level, int i, int first, int cnt, const RxBox &x) {
    const int parent = rx_node(level - 2, i >> 2), slot = i & 3;
    float *f = reinterpret_cast<float *>(b.nodes4 + 8 * (size_t)parent);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float c = cnt ? (float)(0.5 * ((double)x.lo[a] + (double)x.hi[a])) : 1e30f;
        const double need = cnt ? fmax((double)x.hi[a] - (double)c, (double)c - (double)x.lo[a]) : 0.0;
        f[4 * a + slot] = c;
        reinterpret_cast<unsigned short *>(f + 12)[4 * a + slot] = half_up(need);
    }
    reinterpret_cast<int *>(f + 20)[slot] = cnt <= kRxLeaf || level >= b.last ? leaf_ref(first, cnt) : rx_node(level, i);
}

// The order (0..2: axis of the split one level up) that segment seg's points are read in, and the
// segment's box: a warp takes a half of the parent on an axis.  in: three orders of n points.
template <int kBlock>
__device__ int chosen_order(const RxBuild &b, const float4 *in, int seg, RxBox &box) {
    __shared__ RxBox half[6];
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < 6; w += kBlock / 32) {   // axis w >> 1, half w & 1
        const int sib = (seg & ~1) | (w & 1);
        const int lo = rx_bound(b.n, b.level, sib), hi = rx_bound(b.n, b.level, sib + 1);
        RxBox x;
        x.clear();
#pragma unroll 8
        for (int i = lo + lane; i < hi; i += 32) x.grow(in[(size_t)(w >> 1) * b.n + i]);
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                x.lo[a] = fminf(x.lo[a], __shfl_xor_sync(0xffffffffu, x.lo[a], o));
                x.hi[a] = fmaxf(x.hi[a], __shfl_xor_sync(0xffffffffu, x.hi[a], o));
            }
        if (lane == 0) half[w] = x;
    }
    __syncthreads();
    RxBox all = half[0];
#pragma unroll
    for (int a = 0; a < 3; ++a) all.lo[a] = fminf(all.lo[a], half[1].lo[a]), all.hi[a] = fmaxf(all.hi[a], half[1].hi[a]);
    const float pad = all.widest() * kRxPad;
    const int axis = best_axis(half[0].area(pad) + half[1].area(pad), half[2].area(pad) + half[3].area(pad),
                               half[4].area(pad) + half[5].area(pad));
    box = half[2 * axis + (seg & 1)];
    return axis;
}

// One binary level: blockIdx.y = segment, blockIdx.x = 32 of its points, one per lane; each warp
// counts against every kSplitWarps-th tile of 32 keys.  in: by id at level 0, else the three orders
// of the level above; out: three orders.
__global__ void __launch_bounds__(32 * kSplitWarps) rx_split_kernel(RxBuild b, const float4 *__restrict__ in,
                                                                    float4 *__restrict__ out) {
    __shared__ __align__(16) float keys[kSplitWarps][3][32];
    __shared__ int ranks[kSplitWarps][3][32];
    wait_predecessor();
    const int seg = blockIdx.y, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int first = rx_bound(b.n, b.level, seg), cnt = rx_bound(b.n, b.level, seg + 1) - first;
    if (b.level > 0) {
        RxBox box;
        in += (size_t)chosen_order<32 * kSplitWarps>(b, in, seg, box) * b.n;
        if (threadIdx.x == 0 && blockIdx.x == 0 && !(b.level & 1)) put_child4(b, b.level, seg, first, cnt, box);
    }
    in += first;
    const int own = blockIdx.x, mine = own * 32 + lane;
    float4 p = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (mine < cnt) p = in[mine];
    const float x[3] = {p.x, p.y, p.z};
    int rank[3] = {0, 0, 0};
    const float4 none = make_float4(INFINITY, INFINITY, INFINITY, 0.0f);
    float4 q = w * 32 + lane < cnt ? in[w * 32 + lane] : none;
    for (int tile = w; tile * 32 < cnt; tile += kSplitWarps) {
        __syncwarp();
        keys[w][0][lane] = q.x, keys[w][1][lane] = q.y, keys[w][2][lane] = q.z;
        __syncwarp();
        const int next = (tile + kSplitWarps) * 32 + lane;
        q = next < cnt ? in[next] : none;
        // equal keys keep their order: those of an earlier tile, and of earlier lanes, come before
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float4 *k4 = reinterpret_cast<const float4 *>(keys[w][a]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 k = k4[i];
                if (tile < own) rank[a] += (k.x <= x[a]) + (k.y <= x[a]) + (k.z <= x[a]) + (k.w <= x[a]);
                else rank[a] += (k.x < x[a]) + (k.y < x[a]) + (k.z < x[a]) + (k.w < x[a]);
            }
            if (tile == own)
                for (int i = 0; i < 32; ++i) rank[a] += i < lane && keys[w][a][i] == x[a];
        }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) ranks[w][a][lane] = rank[a];
    __syncthreads();
    if (b.level == 0) p.w = __int_as_float(mine);   // the receiver's id
    if (w < 3 && mine < cnt) {
        int r = 0;
#pragma unroll
        for (int i = 0; i < kSplitWarps; ++i) r += ranks[i][w][lane];
        out[(size_t)w * b.n + first + r] = p;
    }
}

// The levels from b.level to the leaves of one segment of at most kRxSub points.
__global__ void __launch_bounds__(kRxSub) rx_subtree_kernel(RxBuild b, const float4 *__restrict__ in,
                                                            float4 *__restrict__ out) {
    __shared__ float4 pts[kRxSub], order[3][kRxSub];
    __shared__ float areas[3][kRxSub];   // of a half, at its first place
    wait_predecessor();
    int seg = blockIdx.x;   // segment of this thread's place
    const int t = threadIdx.x, base = rx_bound(b.n, b.level, seg);
    const int cnt = rx_bound(b.n, b.level, seg + 1) - base;
    const bool on = t < cnt;
    RxBox box;
    if (b.level > 0) in += (size_t)chosen_order<kRxSub>(b, in, seg, box) * b.n;
    if (on) {
        pts[t] = in[base + t];
        if (b.level == 0) pts[t].w = __int_as_float(t);
    }
    __syncthreads();
    if (b.level == 0) {
        box.clear();
        for (int i = 0; i < cnt; ++i) box.grow(pts[i]);
    }
    for (int level = b.level;; ++level) {
        // places relative to the block's: the segment's first, its halves' border, its end
        int first = 0, mid = 0, end = 0;
        if (on) {
            first = rx_bound(b.n, level, seg) - base;
            mid = rx_bound(b.n, level + 1, 2 * seg + 1) - base;
            end = rx_bound(b.n, level, seg + 1) - base;
            if (t == first && !(level & 1)) {
                if (level >= 2) put_child4(b, level, seg, base + first, end - first, box);
                // the slots that no point will fill
                if (level < b.last)
                    for (int c = 4 * seg; c < 4 * seg + 4; ++c) {
                        const int f = rx_bound(b.n, level + 2, c);
                        if (rx_bound(b.n, level + 2, c + 1) == f) put_child4(b, level + 2, c, f, 0, box);
                    }
            }
        }
        if (level >= b.last) break;
        if (on) {
            const float4 p = pts[t];
            int rx = first, ry = first, rz = first;
            for (int i = first; i < end; ++i) {
                const float4 q = pts[i];
                const bool before = i < t;
                rx += q.x < p.x || (q.x == p.x && before);
                ry += q.y < p.y || (q.y == p.y && before);
                rz += q.z < p.z || (q.z == p.z && before);
            }
            order[0][rx] = p, order[1][ry] = p, order[2][rz] = p;
        }
        __syncthreads();
        const float pad = box.widest() * kRxPad;
        const int lo = t < mid ? first : mid, hi = t < mid ? mid : end;
        RxBox half[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            half[a].clear();
            for (int i = lo; i < hi; ++i) half[a].grow(order[a][i]);
            if (on && t == lo) areas[a][t] = half[a].area(pad);
        }
        __syncthreads();
        if (on) {
            float c[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (first < mid) c[a] += areas[a][first];
                if (mid < end) c[a] += areas[a][mid];
            }
            const int axis = best_axis(c[0], c[1], c[2]);
            box = axis == 0 ? half[0] : (axis == 1 ? half[1] : half[2]);
            pts[t] = order[axis][t];
            seg = 2 * seg + (t >= mid);
        }
        __syncthreads();
    }
    if (on) out[base + t] = pts[t];
}

// The leaves' level: even, at least 2 (the root is always a node), no segment above kRxLeaf points.
int rx_last(int n) {
    int last = 2;
    while (((n - 1) >> last) + 1 > kRxLeaf) last += 2;
    return last;
}

}  // namespace

int rx_tree_nodes(int n) { return rx_node(rx_last(n), 0); }
int64_t rx_tree_scratch(int n) { return n > kRxSub ? 6LL * n : 0; }

cudaError_t launch_rx_tree(const float4 *by_id, int n, float4 *pts, float4 *scratch, float4 *nodes4, cudaStream_t s) {
    RxBuild b{nodes4, n, 0, rx_last(n)};
    const float4 *in = by_id;
    for (int longest = n; longest > kRxSub; longest = ((n - 1) >> ++b.level) + 1) {
        float4 *out = scratch + (b.level & 1 ? 3LL * n : 0);
        const cudaError_t e = launch_chained(rx_split_kernel, dim3((longest - 1) / 32 + 1, 1u << b.level),
                                             32 * kSplitWarps, 0, s, b, in, out);
        if (e != cudaSuccess) return e;
        in = out;
    }
    return launch_chained(rx_subtree_kernel, 1u << b.level, kRxSub, 0, s, b, in, pts);
}

}  // namespace sbr
