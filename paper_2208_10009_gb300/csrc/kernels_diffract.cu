// kernels_diffract.cu -- the rough search for order-1 diffraction paths (§III.A, Fig. 4:
// rays reflect on faces and diffract on wedges; §IV, Figs. 7c-d).
//
// Per (Tx, ray) (five passes, below).  A ray meets a wedge when the edge point X seen at the
// smallest angle to the ray lies inside the ray cone (angle <= cone) and ahead of Tx, Tx
// lies in the wedge's exterior, and X is visible from Tx (segment Tx -> X unblocked, the
// wedge's two faces excluded: a ray grazing one of them just before the edge still has
// the edge in its cone).  The diffracted rays leave X on its Keller cone; a receiver gets
// one when it lies in the exterior, its Eq. 3 error angle in the wedge's unfolded space --
// angle(d, Rx* - Tx), Rx* being Rx rotated about the edge line into the half-plane
// opposite Tx -- is within the cone, and the segment X -> Rx is unblocked (the wedge's two
// faces excluded).  Each such (ray, wedge, Rx) appends a record (order 1, faces[0] =
// -1 - wedge id) to the launch's record buffer, before double-count removal.
//
// Candidate wedges come from a BVH over the wedge segments, each node box grown by
// tan(cone) times the largest foot of its corners on the ray: every point of the box
// inside the ray cone then lies within that margin of the ray (see cone_box).
#include "lattice_order.cuh"
#include "sbr_device.cuh"
#include "stream_launch.cuh"

namespace sbr {

struct WedgeF {
    float3 a, b, w1, w2;
    int f1, f2;
};

__device__ __forceinline__ WedgeF load_wedge(const SceneDev &S, int id) {
    const float4 *p = S.wedges + 4 * (size_t)id;
    float4 A = __ldg(p), B = __ldg(p + 1), W1 = __ldg(p + 2), W2 = __ldg(p + 3);
    return {f3(A), f3(B), f3(W1), f3(W2), __float_as_int(A.w), __float_as_int(B.w)};
}

__device__ __forceinline__ float angle32(float3 d, float3 v) {
    float3 c = cross(d, v);
    return atan2f(sqrtf(dot(c, c)), dot(d, v));
}

// p lies outside the interior sector (the solid) between w1 and w2; e = edge direction
__device__ __forceinline__ bool exterior32(const WedgeF &w, float3 e, float3 p) {
    float3 q = p - w.a;
    q = q - e * dot(q, e);
    float3 n = cross(w.w1, w.w2);
    return !(dot(cross(w.w1, q), n) > 0.0f && dot(cross(q, w.w2), n) > 0.0f);
}

// the edge point seen from o at the smallest angle to d (segment end or the interior
// critical point of the angle along the edge line); returns that angle
__device__ __forceinline__ float nearest_seen(const WedgeF &w, float3 o, float3 d, float3 &X) {
    const float3 a0 = w.a - o, eb = w.b - w.a;
    const float al = dot(d, a0), be = dot(d, eb), c = dot(a0, a0), ep = dot(a0, eb), g = dot(eb, eb);
    float uc = -1.0f;
    const float den = be * ep - al * g;
    if (den != 0.0f) {
        float u = (al * ep - be * c) / den;
        if (u > 0.0f && u < 1.0f) uc = u;
    }
    float best = INFINITY;
    const float cand[3] = {0.0f, 1.0f, uc};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (cand[i] < 0.0f) continue;
        float3 v = a0 + eb * cand[i];
        float ang = angle32(d, v);
        if (ang < best) {
            best = ang;
            X = o + v;
        }
    }
    return best;
}

// Child box of a 2-wide node against the ray cone.  A box point X inside the cone has its
// foot s_X on the ray between 0 and s_max, the largest foot of any box corner, and lies
// within s_X tan(cone) <= s_max tan(cone) of the ray; so the box grown by that radius
// (plus a relative rounding margin) must meet the ray segment t in [0, s_max].  od = o . d.
__device__ __forceinline__ bool cone_box(float lx, float ly, float lz, float hx, float hy, float hz, const RayPre &r,
                                         float od, float tan_cone) {
    const float smax = (r.d.x > 0.0f ? hx : lx) * r.d.x + (r.d.y > 0.0f ? hy : ly) * r.d.y +
                       (r.d.z > 0.0f ? hz : lz) * r.d.z - od;
    if (!(smax > 0.0f)) return false;
    const float g = smax * (tan_cone * 1.001f + 1e-6f);
    const float t0x = (lx - g - r.o.x) * r.inv.x, t1x = (hx + g - r.o.x) * r.inv.x;
    const float t0y = (ly - g - r.o.y) * r.inv.y, t1y = (hy + g - r.o.y) * r.inv.y;
    const float t0z = (lz - g - r.o.z) * r.inv.z, t1z = (hz + g - r.o.z) * r.inv.z;
    const float tn = fmaxf(fmaxf(fminf(t0x, t1x), fminf(t0y, t1y)), fmaxf(fminf(t0z, t1z), 0.0f));
    const float tf = fminf(fminf(fmaxf(t0x, t1x), fmaxf(t0y, t1y)), fminf(fmaxf(t0z, t1z), smax * 1.000001f + g));
    return tn <= tf;
}

// Pass 1: candidate wedges of the rays (edge point X inside the cone, ahead of Tx, Tx in the
// exterior), appended to the candidate list as (X, place) and (tx, wedge).  Rays at consecutive
// places leave Tx almost together, so their walks over the wedge tree are one walk: a warp
// takes kGroup places, bounds their directions by a beam (an axis and the largest angle to it),
// and walks the tree for the beam grown by the cone, its lanes testing 32 child boxes at a time.
// The wedges met are filtered against the beam of each 32 places, a (wedge, beam) pair per lane,
// and only the pairs left run the exact test, a ray per lane.  Where the group does not bundle
// (a beam past kMaxBeam: vertex rays, the ends of the icosahedron's edges, coarse lattices), each
// 32 places make a beam, and where those do not either, each lane walks the tree for its own ray.  Per-ray walks took 3,300 warp instructions for 32 rays of the canyon
// (n = 700, 2,000 faces' wedges, 4.9M rays: 687 us); beams take 670 and the exact tests 170 (179 + 42
// us; groups of 64 / 256 places: 226 / 239 us).
constexpr int kGroup = 128, kSub = 32, kSubs = kGroup / kSub;
constexpr int kBeamStack = 512, kBeamList = 128;   // nodes to visit, wedges to test of a warp
constexpr int kBeamStep = 16;                      // nodes a step visits: both children, a lane each
constexpr float kMaxBeam = 0.7f;                   // rad, cone included

struct BeamShared {
    float4 dir[kGroup];      // directions and ray ids
    float4 axis[kSubs];      // beam of each 32 places: axis, half-angle (rad, > kMaxBeam: none)
    int stack[kBeamStack];
    int list[kBeamList];
};

// Half-angle (rad, rounded up) of the cone about `axis` that holds direction d of every lane in
// `mask` (4 if one is a right angle or more away).
__device__ __forceinline__ float beam_angle(float3 axis, float3 d, unsigned mask, int lane) {
    const bool in = (mask >> lane) & 1u;
    const float3 c = cross(axis, d);
    if (__any_sync(0xffffffffu, in && !(dot(axis, d) > 0.0f))) return 4.0f;
    const unsigned s2 = __reduce_max_sync(0xffffffffu, in ? __float_as_uint(dot(c, c)) : 0u);   // floats >= 0 order like their bits
    return asinf(fminf(sqrtf(__uint_as_float(s2)), 1.0f)) * 1.001f + 1e-6f;
}

// The exact test of wedge `id` for ray d; X is the edge point.
__device__ __forceinline__ bool wedge_candidate(const DiffractArgs &A, int id, float3 o, float3 d, float3 &X) {
    const WedgeF w = load_wedge(A.scene, id);
    return nearest_seen(w, o, d, X) <= A.cone && dot(X - o, d) > 0.0f;
}

// Append candidate (X, place), (tx, wedge) of the lanes of the warp's active mask that have one.
__device__ __forceinline__ void append_candidate(const DiffractArgs &A, bool cand, float3 X, int place, int txi, int id) {
    const unsigned m = __activemask(), want = __ballot_sync(m, cand);
    if (!cand) return;
    const int lane = threadIdx.x & 31, leader = __ffs(want) - 1;
    unsigned long long at = 0;
    if (lane == leader)
        at = atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kDiffCand), (unsigned long long)__popc(want));
    const long long slot = (long long)__shfl_sync(want, at, leader) + __popc(want & ((1u << lane) - 1u));
    if (slot >= A.cand_cap) return;
    if (A.id_order_n > 0) place = schedule_place(place, A.id_order_n);
    A.cand[2 * slot] = make_float4(X.x, X.y, X.z, __int_as_float(place));
    A.cand[2 * slot + 1] = make_float4(__int_as_float(txi), __int_as_float(id), 0.0f, 0.0f);
}

// Can wedge w (the edge point seen at the smallest angle) come within angle g of a beam's axis?  A ray's own test
// finds a point at most its FP32 error beyond the true smallest angle, which the triangle inequality
// carries to the axis; nearest_seen at the axis, though, places its interior point by quotients that lose
// a factor 1 / sin^2 a of their digits, a the angle between the edge and the line of sight to its end:
// found at most 1.3e-7 / sin^2 a rad beyond the smallest angle (4.8e7 random edges against FP64, a from
// 0.4 to 90 degrees), so three times that is allowed.  For edges that point at Tx or pass it closely the
// test then says nothing and the rays are tested.  (Without it 1 in 150 to 1,500 of such edges' candidates
// were lost.)
__device__ __forceinline__ bool beam_sees(const WedgeF &w, float3 o, float3 axis, float g) {
    const float3 a0 = w.a - o, eb = w.b - w.a;
    const float c = dot(a0, a0), ep = dot(a0, eb), cg = c * dot(eb, eb);
    const float s2 = fmaxf((cg - ep * ep) / cg, 1e-7f);
    float3 X;
    return !(nearest_seen(w, o, axis, X) > g + 4e-7f / s2);
}

// The pairs' queue lies in the record array past the trace's n0 records, four to a record; the
// diffraction receptions are parked there only after the exact tests.
__device__ __forceinline__ int4 *pair_list(const DiffractArgs &A, long long n0) {
    return reinterpret_cast<int4 *>(A.recs + n0);
}
__device__ __forceinline__ long long pair_space(const DiffractArgs &A, long long n0) {
    return n0 < A.rec_cap ? 4 * (A.rec_cap - n0) : 0;
}

// Whole warp: wedge `id` against the rays of the 32 places from `base`.
__device__ __forceinline__ void exact_pair(const DiffractArgs &A, int base, int txi, int id, float3 o, int lane,
                                           unsigned &tests) {
    bool cand = base + lane < A.first + A.count;
    float3 X = o;
    if (cand) {
        const float4 dd = __ldg(A.dirs + (A.id_order_n > 0 ? schedule_place(base + lane, A.id_order_n) : base + lane));
        const int ray = __float_as_int(dd.w);
        cand = ray >= A.ray_begin && ray < A.ray_end;
        if (cand) {
            ++tests;
            cand = wedge_candidate(A, id, o, f3(dd), X);
        }
    }
    if (__any_sync(0xffffffffu, cand)) append_candidate(A, cand, X, base + lane, txi, id);
}

// The walk of one lane's ray d by itself.
__device__ __noinline__ void walk_ray(const DiffractArgs &A, int txi, int place, float3 o, float3 d, unsigned &tests) {
    const SceneDev &S = A.scene;
    const RayPre r = make_ray(o, d);
    const float od = dot(o, d);
    int stack[kStackDepth];
    int sp = 0, node = 0;
    for (;;) {
        if (is_leaf(node)) {
            const int first = leaf_first(node), cnt = leaf_count(node);
            for (int i = first; i < first + cnt; ++i) {
                const int id = __ldg(S.wedge_bvh_ids + i);
                const WedgeF w = load_wedge(S, id);
                float3 X = o;
                ++tests;
                bool cand = wedge_candidate(A, id, o, d, X);
                if (cand) {
                    const float3 eb = w.b - w.a;
                    cand = exterior32(w, eb * (1.0f / sqrtf(dot(eb, eb))), o);
                }
                append_candidate(A, cand, X, place, txi, id);
            }
        } else {
            const float4 *nd = S.wnodes + 4 * (size_t)node;
            const float4 p = __ldg(nd), q = __ldg(nd + 1), t = __ldg(nd + 2);
            const int4 refs = __ldg(reinterpret_cast<const int4 *>(nd + 3));
            const bool in0 = cone_box(p.x, p.y, p.z, p.w, q.x, q.y, r, od, A.tan_cone);
            const bool in1 = cone_box(q.z, q.w, t.x, t.y, t.z, t.w, r, od, A.tan_cone);
            if (in0 && in1) {
                if (SBR_CHECKED_ON && sp >= min(S.stack_limit, kStackDepth)) {
                    check_fail(S, SBR_CHECK_BVH2_STACK);
                    return;
                }
                stack[sp++] = refs.y;
            }
            if (in0 || in1) {
                node = in0 ? refs.x : refs.y;
                continue;
            }
        }
        if (sp == 0) return;
        node = stack[--sp];
    }
}

__global__ void __launch_bounds__(128, 6) diffract_candidates(DiffractArgs A) {
    wait_predecessor();
    __shared__ BeamShared s_beam[4];
    BeamShared &sh = s_beam[threadIdx.x >> 5];
    const SceneDev &S = A.scene;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long groups = (A.count + kGroup - 1) / kGroup, total = (long long)A.ntx * groups;
    const long long n0 = A.counters[kRecords], pair_cap = pair_space(A, n0);   // nothing appends records here
    unsigned tests = 0;
    // groups from a queue: one that looks along the streets costs many times one that looks up
    for (;;) {
        long long item = 0;
        if (lane == 0)
            item = (long long)atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kDiffHead), 1ULL);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= total) break;
        const int txi = (int)(item / groups);
        const long long base = (item - (long long)txi * groups) * kGroup;
        const float3 o = f3(__ldg(A.tx + txi));
        // the places' rays, and the beam of every 32 of them
        unsigned valid[kSubs];
        __syncwarp();
#pragma unroll
        for (int q = 0; q < kSubs; ++q) {
            const long long local = base + q * kSub + lane;
            float4 dd = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(-1));
            if (local < A.count) {
                int place = (int)(A.first + local);
                if (A.id_order_n > 0) place = schedule_place(place, A.id_order_n);
                dd = __ldg(A.dirs + place);
            }
            const int ray = __float_as_int(dd.w);
            valid[q] = __ballot_sync(0xffffffffu, local < A.count && ray >= A.ray_begin && ray < A.ray_end);
            sh.dir[q * kSub + lane] = dd;
            const int mid = (valid[q] >> 16) & 1u ? 16 : __ffs(valid[q]) - 1;
            const float3 axis = make_float3(__shfl_sync(0xffffffffu, dd.x, mid & 31), __shfl_sync(0xffffffffu, dd.y, mid & 31),
                                            __shfl_sync(0xffffffffu, dd.z, mid & 31));
            const float g = valid[q] ? beam_angle(axis, f3(dd), valid[q], lane) + A.cone * 1.001f + 1e-5f : 4.0f;
            if (lane == 0) sh.axis[q] = make_float4(axis.x, axis.y, axis.z, g);
        }
        __syncwarp();
        // the beam of the whole group about the axis of its second 32 places
        unsigned any = 0;
#pragma unroll
        for (int q = 0; q < kSubs; ++q) any |= valid[q] ? 1u << q : 0u;
        if (!any) continue;
        const int qm = (any >> 1) & 1u ? 1 : __ffs(any) - 1;
        const float3 gaxis = f3(sh.axis[qm]);
        float gang = 0.0f;
#pragma unroll
        for (int q = 0; q < kSubs; ++q)
            if (valid[q]) gang = fmaxf(gang, beam_angle(gaxis, f3(sh.dir[q * kSub + lane]), valid[q], lane));
        gang += A.cone * 1.001f + 1e-5f;
        // beams in turn: the group, or each 32 places
        while (any) {
            float3 axis = gaxis;
            float ang = gang;
            int q0 = 0, q1 = kSubs;   // places [q0, q1) x 32
            if (gang <= kMaxBeam) {
                any = 0;
            } else {
                q0 = __ffs(any) - 1;
                q1 = q0 + 1;
                any &= any - 1;
                const float4 ax = sh.axis[q0];
                axis = f3(ax);
                ang = ax.w;
                if (ang > kMaxBeam) {
                    const float4 dd = sh.dir[q0 * kSub + lane];
                    if ((valid[q0] >> lane) & 1u)
                        walk_ray(A, txi, (int)(A.first + base) + q0 * kSub + lane, o, f3(dd), tests);
                    __syncwarp();
                    continue;
                }
            }
            const RayPre r = make_ray(o, axis);
            const float od = dot(o, axis), tan_g = tanf(ang) * 1.001f;
            int sp = 1, ln = 0;
            if (lane == 0) sh.stack[0] = 0;
            __syncwarp();
            while (sp > 0 || ln > 0) {
                if (sp > 0 && ln <= kBeamList - 64) {
                    // the last nodes pushed, both children of each (one node once the stack runs full: a
                    // depth-first walk then needs one entry a level)
                    const int m = sp > kBeamStack - kStackDepth - 2 * kBeamStep ? 1 : min(sp, kBeamStep);
                    if (SBR_CHECKED_ON && sp + m > min(S.stack_limit, kBeamStack)) {
                        check_fail(S, SBR_CHECK_BVH2_STACK);
                        sp = 0;
                        continue;
                    }
                    bool hit = false;
                    int ref = 0;
                    if ((lane >> 1) < m) {
                        const int node = sh.stack[sp - 1 - (lane >> 1)];
                        if (is_leaf(node)) {   // a tree of one leaf
                            ref = node;
                            hit = (lane & 1) == 0;
                        } else {
                            const float *nd = reinterpret_cast<const float *>(S.wnodes + 4 * (size_t)node);
                            const float2 *bx = reinterpret_cast<const float2 *>(nd + 6 * (lane & 1));
                            const float2 p = __ldg(bx), q = __ldg(bx + 1), t = __ldg(bx + 2);
                            ref = __float_as_int(__ldg(nd + 12 + (lane & 1)));
                            hit = cone_box(p.x, p.y, q.x, q.y, t.x, t.y, r, od, tan_g);
                        }
                    }
                    sp -= m;
                    __syncwarp();
                    const unsigned inner = __ballot_sync(0xffffffffu, hit && !is_leaf(ref));
                    if (hit && !is_leaf(ref)) sh.stack[sp + __popc(inner & lt)] = ref;
                    sp += __popc(inner);
                    // the leaves' wedges join the list (a leaf holds two as a rule; a long one comes in parts)
                    int cnt = hit && is_leaf(ref) ? leaf_count(ref) : 0, first = leaf_first(ref);
                    while (__any_sync(0xffffffffu, cnt > 0)) {
                        if (ln > kBeamList - 32) break;
                        const unsigned have = __ballot_sync(0xffffffffu, cnt > 0);
                        if (cnt > 0) {
                            sh.list[ln + __popc(have & lt)] = __ldg(S.wedge_bvh_ids + first);
                            ++first;
                            --cnt;
                        }
                        ln += __popc(have);
                    }
                    // parts that did not fit go back as leaves
                    const unsigned rest = __ballot_sync(0xffffffffu, cnt > 0);
                    if (cnt > 0) sh.stack[sp + __popc(rest & lt)] = leaf_ref(first, cnt);
                    sp += __popc(rest);
                    __syncwarp();
                    if (sp > 0 && ln <= kBeamList - 64) continue;
                }
                // filter: a (wedge, 32 places) pair per lane against the pair's beam
                const int subs = q1 - q0, pairs = ln * subs;
                for (int pb = 0; pb < pairs; pb += 32) {
                    const int pr = pb + lane, wi = pr / subs, q = q0 + pr - wi * subs;
                    bool pass = false;
                    int id = 0;
                    if (pr < pairs) {
                        id = sh.list[wi];
                        const float4 ax = sh.axis[q];
                        const WedgeF w = load_wedge(S, id);
                        const float3 eb = w.b - w.a;
                        pass = (ax.w > kMaxBeam || beam_sees(w, o, f3(ax), ax.w)) &&
                               exterior32(w, eb * (1.0f / sqrtf(dot(eb, eb))), o);
                    }
                    unsigned left = __ballot_sync(0xffffffffu, pass);
                    if (!left) continue;
                    // queued for diffract_exact; past the queue's end tested here
                    unsigned long long at = 0;
                    if (lane == 0)
                        at = atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kDiffPairs),
                                       (unsigned long long)__popc(left));
                    const long long slot = (long long)__shfl_sync(0xffffffffu, at, 0) + __popc(left & lt);
                    const int pair_base = (int)(A.first + base) + q * kSub;
                    if (pass && slot < pair_cap) pair_list(A, n0)[slot] = make_int4(pair_base, txi, id, 0);
                    left &= __ballot_sync(0xffffffffu, slot >= pair_cap);
                    while (left) {
                        const int src = __ffs(left) - 1;
                        left &= left - 1;
                        exact_pair(A, __shfl_sync(0xffffffffu, pair_base, src), txi, __shfl_sync(0xffffffffu, id, src), o,
                                   lane, tests);
                    }
                }
                ln = 0;
                __syncwarp();
            }
        }
    }
    tests = __reduce_add_sync(0xffffffffu, tests);
    if (lane == 0 && tests) atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kWedgeTests), tests);
}

// Pass 2: the exact tests of the queued pairs, a warp per pair: a beam along a street leaves hundreds of
// pairs where most leave none, so they are spread over the chip (tested by the warp that found
// them, the last group alone ran for 200 us).
__global__ void __launch_bounds__(128) diffract_exact(DiffractArgs A) {
    wait_predecessor();
    const long long n0 = A.counters[kRecords], cap = pair_space(A, n0);
    long long n = A.counters[kDiffPairs];
    if (n > cap) n = cap;
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    unsigned tests = 0;
    for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += warps) {
        const int4 p = __ldg(pair_list(A, n0) + i);
        exact_pair(A, p.x, p.y, p.z, f3(__ldg(A.tx + p.y)), lane, tests);
    }
    tests = __reduce_add_sync(0xffffffffu, tests);
    if (lane == 0 && tests) atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kWedgeTests), tests);
}

// Pass 3, one candidate per thread: is its edge point visible from Tx (segment Tx -> X unblocked,
// the wedge's faces excluded)?  The answer goes into the candidate.
__global__ void __launch_bounds__(128) diffract_visible(DiffractArgs A) {
    wait_predecessor();
    const SceneDev &S = A.scene;
    long long ncand = A.counters[kDiffCand];
    if (ncand > A.cand_cap) ncand = A.cand_cap;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < ncand; c += (long long)gridDim.x * blockDim.x) {
        const float4 c0 = A.cand[2 * c], c1 = A.cand[2 * c + 1];
        const WedgeF w = load_wedge(S, __float_as_int(c1.y));
        const float3 o = f3(__ldg(A.tx + __float_as_int(c1.x)));
        const bool vis = !any_hit4(S, make_ray(o, f3(c0) - o), 1e-6f, 1.0f - 1e-6f, w.f1, w.f2);
        A.cand[2 * c + 1].z = __int_as_float(vis);
    }
}

// Pass 4, a visible candidate per warp: its lanes test the receivers (exterior, unfolded error
// angle within the cone).  Nearly all receivers are far from the Keller cone, so they are first
// compared with it in the frame of the edge, where the test is two products and needs no sector,
// arc tangent or exact root (60 -> 30 instructions a receiver).  A warp used to take 32
// candidates, whose unlike loops left 21 % of the warp slots in use: with the
// visibility queries inside 186 us, now 42 (diffract_visible) + 71 us (canyon, 240k candidates, 256
// receivers).
// Receptions waiting for their occlusion query (diffract_occlusion) are parked at the top of
// the record array, slot rec_cap - 1 - q for the q-th, while the final records grow from
// the trace's count n0 at the bottom; parking q < (rec_cap - n0) / 2 of them leaves room for
// all of them as final records, so the two ends never meet.  Those past that bound are only
// counted, and the host reports a record overflow (sbr_launch_get_stats): the record count on the
// device stays that of the records written, which is what later kernels read.
__device__ __forceinline__ long long park_limit(const DiffractArgs &A, long long n0) { return (A.rec_cap - n0) / 2; }

__global__ void __launch_bounds__(256) diffract_receive(DiffractArgs A) {
    wait_predecessor();
    const SceneDev &S = A.scene;
    long long ncand = A.counters[kDiffCand];
    if (ncand > A.cand_cap) ncand = A.cand_cap;
    const long long n0 = A.counters[kRecords];   // the trace's records; nothing appends here
    const long long limit = park_limit(A, n0);
    if (blockIdx.x == 0 && threadIdx.x == 0) A.counters[kDiffBase] = n0;
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long c = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < ncand; c += warps) {
        const float4 c1 = __ldg(A.cand + 2 * c + 1);
        if (!__float_as_int(c1.z)) continue;
        const float4 x0 = __ldg(A.cand + 2 * c);
        const int txi = __float_as_int(c1.x), id = __float_as_int(c1.y);
        const WedgeF w = load_wedge(S, id);
        const float3 o = f3(__ldg(A.tx + txi));
        const float4 dd = __ldg(A.dirs + __float_as_int(x0.w));
        const float3 d = f3(dd);
        const int ray = __float_as_int(dd.w);
        const float3 X = f3(x0);
        const float3 eb = w.b - w.a;
        const float3 e = eb * (1.0f / sqrtf(dot(eb, eb)));
        // frame of the plane across the edge: b1 towards Tx, b2 = e x b1.  A point
        // q = p - a has coordinates (x, y, z) = (q.b1, q.b2, q.e); its image rotated
        // into the half-plane opposite Tx is a + z e - sqrt(x^2 + y^2) b1, and it lies in
        // the solid's sector iff it is strictly between w1 and w2 (2-D cross products)
        float3 pt = (o - w.a) - e * dot(o - w.a, e);
        const float rt = sqrtf(dot(pt, pt));
        if (!(rt > 0.0f)) continue;
        const float3 b1 = pt * (1.0f / rt), b2 = cross(e, b1);
        const float w1x = dot(w.w1, b1), w1y = dot(w.w1, b2), w2x = dot(w.w2, b1), w2y = dot(w.w2, b2);
        const float s12 = w1x * w2y - w1y * w2x;
        const float3 a0 = w.a - o;
        const float t2 = A.tan_cone * A.tan_cone * 1.0001f;   // pre-test, the exact test follows
        // the same test in the edge's frame, as a conservative filter: W = A e - B b1 with A = z -
        // z_Tx, B = rho + rho_Tx, so |d x W|^2 = (d_e B + d_b1 A)^2 + d_b2^2 |W|^2.  Beside 1 % of the cone it
        // allows for FP32: b1 is off by up to 2e-7 |Tx - a| / rho_Tx (Tx close to the edge's line), A by
        // 2e-7 (|z| + |z_Tx|), and both enter times |A| + B at most.  (With 2e-6 (|A| + B) alone, receptions
        // within a metre of the line were lost, 1 in 700 at 1 km from the origin and 2 mrad; with twice these
        // bounds none of 1.7e7 is.)
        const float off = 2e-6f + 1e-6f * sqrtf(dot(a0, a0)) / rt, off_z = 1e-6f * fabsf(dot(a0, e));
        const float de = dot(d, e), db = dot(d, b1), dn2 = dot(d, b2) * dot(d, b2), ze = dot(o - w.a, e);
        const float tc = A.tan_cone * 1.01f;
        for (int rx = lane; rx < A.rx.nrx; rx += 32) {
            const float3 R = f3(__ldg(A.rx.by_id + rx));
            const float3 q = R - w.a;
            const float x = dot(q, b1), y = dot(q, b2), z = dot(q, e);
            float rho;
            asm("sqrt.approx.f32 %0, %1;" : "=f"(rho) : "f"(x * x + y * y));
            const float fa = z - ze, fb = rho + rt, u = fmaf(de, fb, db * fa);
            const float lim = fmaf(fabsf(fmaf(de, fa, -db * fb)), tc, fmaf(off, fabsf(fa) + fb, off_z));
            const bool far = fmaf(u, u, dn2 * fmaf(fa, fa, fb * fb)) > lim * lim;
            if (far && !SBR_CHECKED_ON) continue;
            const float c1 = w1x * y - w1y * x, c2 = x * w2y - y * w2x;
            if (c1 * s12 > 0.0f && c2 * s12 > 0.0f) continue;   // Rx inside the solid's sector
            const float3 W = a0 + e * z - b1 * sqrtf(x * x + y * y);
            const float3 cw = cross(d, W);
            const float dw = dot(d, W), cc = dot(cw, cw);
            if (!(dw > 0.0f) || cc > dw * dw * t2) continue;
            const float err = atan2f(sqrtf(cc), dw);
            if (!(err <= A.cone)) continue;
            if (far) {   // SBR_CHECKED builds: the filter let go of a reception
                check_fail(S, SBR_CHECK_RX_FILTER);
                continue;
            }
            // the segment X -> Rx is tested by diffract_occlusion, a query per thread in
            // full warps (here it would run in one lane while the warp waits); the
            // reception is parked with X in its unused face slots 1-3
            const long long pq = (long long)atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kDiffPending), 1ULL);
            if (pq >= limit) continue;
            RecDev rec;
            rec.tx = txi;
            rec.rx = rx;
            rec.ray = ray;
            rec.order = 1;
            rec.faces[0] = -1 - id;
            rec.faces[1] = __float_as_int(X.x);
            rec.faces[2] = __float_as_int(X.y);
            rec.faces[3] = __float_as_int(X.z);
#pragma unroll
            for (int j = 4; j < kMaxOrder; ++j) rec.faces[j] = -1;
            rec.err = err;
            rec.dray = sqrtf(dot(W, W)) * cosf(err);
            rec.slot = -1;
            rec.pad = 0;
            A.recs[A.rec_cap - 1 - pq] = rec;
        }
    }
}

// The occlusion queries of the parked diffraction receptions: a reception whose segment from
// the edge point X to Rx is unblocked (the wedge's two faces excluded) becomes a record,
// appended with one atomic per warp; blocked ones are dropped.  One warp a block, so that a few
// thousand queries spread over the SMs (60 -> 28 us).
__global__ void __launch_bounds__(32) diffract_occlusion(DiffractArgs A) {
    wait_predecessor();
    const SceneDev &S = A.scene;
    long long P = A.counters[kDiffPending];
    const long long limit = park_limit(A, A.counters[kDiffBase]);
    if (P > limit) P = limit;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    unsigned emitted = 0;
    for (long long base = (long long)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < P;
         base += warps * 32) {
        const long long q = base + lane;
        RecDev rec;
        bool keep = false;
        if (q < P) {
            rec = A.recs[A.rec_cap - 1 - q];
            const float3 X = make_float3(__int_as_float(rec.faces[1]), __int_as_float(rec.faces[2]),
                                         __int_as_float(rec.faces[3]));
            const float3 R = f3(__ldg(A.rx.by_id + rec.rx));
            const WedgeF w = load_wedge(S, -1 - rec.faces[0]);
            keep = !any_hit4(S, make_ray(X, R - X), 1e-6f, 1.0f - 1e-6f, w.f1, w.f2);
        }
        const unsigned b = __ballot_sync(0xffffffffu, keep);
        if (!b) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kRecords), (unsigned long long)__popc(b));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & lt);
        if (keep) {
            rec.faces[1] = rec.faces[2] = rec.faces[3] = -1;
            if ((long long)at < A.rec_cap) A.recs[at] = rec;
            ++emitted;
        }
    }
    emitted = __reduce_add_sync(0xffffffffu, emitted);
    if (lane == 0 && emitted) atomicAdd(reinterpret_cast<unsigned long long *>(A.counters + kDiffRecords), emitted);
}

static int candidate_blocks() {
    static int nb = 0;
    if (!nb) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, diffract_candidates, 128, 0);
        if (nb < 1) nb = 1;
    }
    return nb;
}

cudaError_t launch_diffract(const DiffractArgs &a, int num_sms, cudaStream_t s) {
    if (a.scene.nw == 0 || a.rx.nrx == 0) return cudaSuccess;
    cudaError_t e = launch_chained(diffract_candidates, num_sms * candidate_blocks(), 128, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(diffract_exact, num_sms * 8, 128, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(diffract_visible, num_sms * 5, 128, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(diffract_receive, num_sms * 8, 256, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(diffract_occlusion, num_sms * 32, 32, 0, s, a);
    return e;
}

}  // namespace sbr
