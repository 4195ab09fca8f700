// sbr_device.cuh -- device-side geometry: vector helpers, ray/box slab test, watertight
// ray/triangle test, BVH closest-hit and any-hit traversal, receiver candidate query.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <math.h>

#include "sbr_internal.h"

namespace sbr {

__device__ __forceinline__ float3 f3(float4 v) { return make_float3(v.x, v.y, v.z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float3 a, float s) { return make_float3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ float3 cross(float3 a, float3 b) {
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float comp(float3 v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : v.z); }

struct dvec3 {
    double x, y, z;
};
__device__ __forceinline__ dvec3 dv(double x, double y, double z) { return {x, y, z}; }
__device__ __forceinline__ dvec3 operator+(dvec3 a, dvec3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ dvec3 operator-(dvec3 a, dvec3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ dvec3 operator*(dvec3 a, double s) { return {a.x * s, a.y * s, a.z * s}; }
__device__ __forceinline__ double ddot(dvec3 a, dvec3 b) { return fma(a.x, b.x, fma(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ dvec3 dcross(dvec3 a, dvec3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ double dnorm(dvec3 a) { return sqrt(ddot(a, a)); }

// Per-ray precomputation for the slab test and the watertight triangle test.  The
// triangle test's axis permutation and shear are folded into three vectors, so that a
// vertex's sheared coordinates are plain dot products (FMA pipe, no per-component
// selects): with kz the dominant axis of d and (kx, ky) the other two in winding order,
// mx = e_kx - (d_kx / d_kz) e_kz, my = e_ky - (d_ky / d_kz) e_kz, mz = e_kz / d_kz.
struct RayPre {
    float3 o, d, inv;
    float3 mx, my, mz;
};

// The slab tests take a box for met when entry <= exit times this.  It makes up for the rounding of the
// entry and exit distances relative to each other: the approximate reciprocals (an ulp each) and the
// centre's and half extent's product rounded apart, where IEEE reciprocals of lo / hi planes got by with
// 5e-7.  With 1e-6 no more boxes whose edge a ray just meets are passed over than with those: of 4e5 to
// 7e5 such rays 1,756 against 3,275 (coordinates up to 10 m, boxes of 0.5-5 m), 6,530 / 6,995 (boxes of
// 5-50 m; 11,042 with 5e-7), 19,228 / 24,423 (300 m), 39,342 / 44,693 (3.3 km, where the origin's own
// rounding, absolute and the same for both, is most of it).
constexpr float kSlabMargin = 1.000001f;

// 1 / x to one ulp, for the slab tests (their margins cover it); |x| < 1e-30 counts as 1e-30: the
// tests stay correct for axis-parallel rays (huge but finite t), and box * inv - o * inv never
// forms inf - inf.
__device__ __forceinline__ float slab_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fabsf(x) > 1e-30f ? x : copysignf(1e-30f, x)));
    return r;
}

__device__ __forceinline__ RayPre make_ray(float3 o, float3 d) {
    RayPre r;
    r.o = o;
    r.d = d;
    r.inv = make_float3(slab_rcp(d.x), slab_rcp(d.y), slab_rcp(d.z));
    float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    int kz = (ax > ay) ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    int kx = kz == 2 ? 0 : kz + 1;
    int ky = kx == 2 ? 0 : kx + 1;
    if (comp(d, kz) < 0.0f) {
        int t = kx;
        kx = ky;
        ky = t;
    }
    const float sz = 1.0f / comp(d, kz);
    const float sx = comp(d, kx) * sz, sy = comp(d, ky) * sz;
    r.mx = make_float3(kx == 0 ? 1.0f : (kz == 0 ? -sx : 0.0f), kx == 1 ? 1.0f : (kz == 1 ? -sx : 0.0f),
                       kx == 2 ? 1.0f : (kz == 2 ? -sx : 0.0f));
    r.my = make_float3(ky == 0 ? 1.0f : (kz == 0 ? -sy : 0.0f), ky == 1 ? 1.0f : (kz == 1 ? -sy : 0.0f),
                       ky == 2 ? 1.0f : (kz == 2 ? -sy : 0.0f));
    r.mz = make_float3(kz == 0 ? sz : 0.0f, kz == 1 ? sz : 0.0f, kz == 2 ? sz : 0.0f);
    return r;
}

// SBR_CHECKED builds: record a failed bounds check (bit = SBR_CHECK_*) in the launch's
// status word.  The caller then ends the query that failed; nothing traps.
__device__ __forceinline__ void check_fail(const SceneDev &S, unsigned bit) {
    if (S.status) atomicOr(S.status, (unsigned long long)bit);
}
#ifdef SBR_CHECKED
#define SBR_CHECKED_ON 1
#else
#define SBR_CHECKED_ON 0
#endif

// Three-input min / max (one instruction each on sm_100 and later).
__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
// Watertight ray/triangle intersection (Woop, Benthin, Wald, JCGT 2013): edge functions in a
// sheared, permuted frame; an exactly-zero edge function is re-evaluated in double so
// that rays through a shared edge or vertex hit at least one of the triangles.
// Returns t, or a negative value on a miss.
__device__ __forceinline__ float tri_watertight(const RayPre &r, float4 A4, float4 B4, float4 C4) {
    float3 A = f3(A4) - r.o, B = f3(B4) - r.o, C = f3(C4) - r.o;
    float Ax = dot(A, r.mx), Ay = dot(A, r.my), Az = dot(A, r.mz);
    float Bx = dot(B, r.mx), By = dot(B, r.my), Bz = dot(B, r.mz);
    float Cx = dot(C, r.mx), Cy = dot(C, r.my), Cz = dot(C, r.mz);
    float U = Cx * By - Cy * Bx;
    float V = Ax * Cy - Ay * Cx;
    float W = Bx * Ay - By * Ax;
    if (min3f(fabsf(U), fabsf(V), fabsf(W)) == 0.0f) {
        U = (float)((double)Cx * (double)By - (double)Cy * (double)Bx);
        V = (float)((double)Ax * (double)Cy - (double)Ay * (double)Cx);
        W = (float)((double)Bx * (double)Ay - (double)By * (double)Ax);
    }
    // outside if the edge functions have mixed signs
    if (min3f(U, V, W) < 0.0f && max3f(U, V, W) > 0.0f) return -1.0f;
    float det = U + V + W;
    if (det == 0.0f) return -1.0f;
    float T = U * Az + V * Bz + W * Cz;   // mz carries the 1 / d_kz scale
    return T / det;
}

// Two FMAs in one packed f32x2 instruction: (a.x * b + c, a.y * b + c).
__device__ __forceinline__ float2 fma2s(float ax, float ay, float b, float c) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pc, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\t"
        "mov.b64 pb, {%4, %4};\n\t"
        "mov.b64 pc, {%5, %5};\n\t"
        "fma.rn.f32x2 pd, pa, pb, pc;\n\t"
        "mov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(ax), "f"(ay), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ float2 fma2(float2 a, float b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pc, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\t"
        "mov.b64 pb, {%4, %4};\n\t"
        "mov.b64 pc, {%5, %6};\n\t"
        "fma.rn.f32x2 pd, pa, pb, pc;\n\t"
        "mov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float b) {
    float2 r;
    asm("{\n\t.reg .b64 pa, pb, pd;\n\t"
        "mov.b64 pa, {%2, %3};\n\t"
        "mov.b64 pb, {%4, %4};\n\t"
        "mul.rn.f32x2 pd, pa, pb;\n\t"
        "mov.b64 {%0, %1}, pd;\n\t}"
        : "=f"(r.x), "=f"(r.y)
        : "f"(a.x), "f"(a.y), "f"(b));
    return r;
}

// A 4-wide node (layout: sbr_internal.h).
struct NodeAxis {
    float2 c01, c23, h01, h23;
};
struct Node4 {
    NodeAxis x, y, z;
    int4 refs;
};
__device__ __forceinline__ float2 half_pair(unsigned v) { return __half22float2(*reinterpret_cast<__half2 *>(&v)); }
__device__ __forceinline__ void set_axis(NodeAxis &v, float4 c, unsigned h01, unsigned h23) {
    v.c01 = make_float2(c.x, c.y);
    v.c23 = make_float2(c.z, c.w);
    v.h01 = half_pair(h01);
    v.h23 = half_pair(h23);
}
__device__ __forceinline__ Node4 load_node4(const float4 *nd) {
    Node4 v;
    const float4 cx = __ldg(nd), cy = __ldg(nd + 1), cz = __ldg(nd + 2);
    const uint4 hxy = __ldg(reinterpret_cast<const uint4 *>(nd + 3));
    const uint2 hz = __ldg(reinterpret_cast<const uint2 *>(nd + 4));
    v.refs = __ldg(reinterpret_cast<const int4 *>(nd + 5));
    set_axis(v.x, cx, hxy.x, hxy.y);
    set_axis(v.y, cy, hxy.z, hxy.w);
    set_axis(v.z, cz, hz.x, hz.y);
    return v;
}
// The same by three 32-byte loads, for walks whose lanes stand at nodes of their own: the L1 data
// pipe then takes a pass per lane and load (occlusion queries of the office: 92 % busy with 16-byte
// loads).  Coherent lanes share a node's lines and are bound by the bytes returned either way.
__device__ __forceinline__ void load_32(const float4 *p, float4 &a, float4 &b) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}
__device__ __forceinline__ Node4 load_node4_wide(const float4 *nd) {
    Node4 v;
    float4 cx, cy, cz, hxy, hz, rf;
    load_32(nd, cx, cy);
    load_32(nd + 2, cz, hxy);
    load_32(nd + 4, hz, rf);
    v.refs = make_int4(__float_as_int(rf.x), __float_as_int(rf.y), __float_as_int(rf.z), __float_as_int(rf.w));
    set_axis(v.x, cx, __float_as_uint(hxy.x), __float_as_uint(hxy.y));
    set_axis(v.y, cy, __float_as_uint(hxy.z), __float_as_uint(hxy.w));
    set_axis(v.z, cz, __float_as_uint(hz.x), __float_as_uint(hz.y));
    return v;
}

// Where a ray enters and leaves the children's slabs of one axis, t = (c / d - o / d) -+ h / |d|,
// two children per packed FMA.  The walk keeps the SM's issue slots, its ALU pipe and its L1 data
// pipe (a visit's rows come back at 128 bytes a cycle) busy together, so a visit pays for its
// bytes as for its instructions.  Centres and half extents need no near / far row picked by the
// ray's direction signs, so one address serves all rows where lo / hi planes took seven (a visit
// 110 -> 95 instructions, L1 73 -> 81 % busy); FP16 half extents then cut a visit from 112 to 88
// bytes for 12 conversions.  Large city trace 36.19 -> 34.45 ms, canyon 822 -> 802 us.
struct Slab4 {
    float n[4], f[4];
};
__device__ __forceinline__ Slab4 slab4(const NodeAxis &v, float inv, float oi, float ai) {
    const float2 t01 = fma2s(v.c01.x, v.c01.y, inv, -oi), t23 = fma2s(v.c23.x, v.c23.y, inv, -oi);
    const float2 n01 = fma2(v.h01, -ai, t01), n23 = fma2(v.h23, -ai, t23);
    const float2 f01 = fma2(v.h01, ai, t01), f23 = fma2(v.h23, ai, t23);
    return {{n01.x, n01.y, n23.x, n23.y}, {f01.x, f01.y, f23.x, f23.y}};
}

// Pop the next stack entry whose entry distance (sdist, beside the refs in stack) is within
// tcull (the closest-hit range grown by the slab test's tolerance); false once the stack
// holds none.
__device__ __forceinline__ bool pop_near(const int *stack, const float *sdist, int &sp, float tcull, int &node) {
    while (sp > 0) {
        --sp;
        if (sdist[sp] <= tcull) {
            node = stack[sp];
            return true;
        }
    }
    return false;
}

// Closest hit through the 4-wide BVH.  The walk descends inner nodes in an inner loop and
// tests a leaf once it reaches one ("while-while"): a warp then runs the leaf branch only
// when its lanes stand at leaves, not on every step where one lane does.  Per node, slab
// tests of the four child boxes as
// t = (centre - o) / d -+ half extent / |d| (slab4: no per-axis min/max or sign), two children
// per packed FMA and three-input min/max;
// the nearest hit child is visited next and the others are pushed with their entry
// distances; a popped entry whose entry distance already lies beyond the closest hit
// found since its push is dropped unvisited (the box test it would face against the
// shrunk range, so nothing it holds can win).  Closest hit along o + t d over t in (tmin, tmax],
// skipping triangles of face `skip`; ties in t go to the lower face id, then the lower
// triangle index.  Returns the triangle index (BVH order) or -1; t_out, face_out set on a
// hit.  `front`: the entries to start from (FrontArgs) or null.  nodes_visited counts 4-wide nodes (four box tests each).
__device__ __forceinline__ int closest_hit4(const SceneDev &S, const RayPre &r, float tmin, float tmax, int skip,
                                            const int4 *front, float &t_out, int &face_out, unsigned &nodes_visited,
                                            unsigned &tris_tested) {
    int stack[kStack4];    // node or leaf refs
    float sdist[kStack4];  // their entry distances
    int sp = 0;
    int node = 0;
    if (front) {   // start from a frontier (nearest entry first) instead of the root
        t_out = tmax;
        face_out = 0x7fffffff;
        int4 e[kFrontEntries / 2];
#pragma unroll
        for (int j = 0; j < kFrontEntries / 2; ++j) e[j] = __ldg(front + j);
        if (e[0].x == kNoRef) return -1;
#pragma unroll
        for (int j = kFrontEntries / 2 - 1; j >= 0; --j) {
            if (e[j].z != kNoRef) { stack[sp] = e[j].z; sdist[sp++] = __int_as_float(e[j].w); }
            if (j > 0 && e[j].x != kNoRef) { stack[sp] = e[j].x; sdist[sp++] = __int_as_float(e[j].y); }
        }
        node = e[0].x;
    }
    float tbest = tmax;
    float tcull = tmax * kSlabMargin;   // entries entering beyond this are dropped at pop
    int best = -1, bface = 0x7fffffff;
    const float oix = r.o.x * r.inv.x, oiy = r.o.y * r.inv.y, oiz = r.o.z * r.inv.z;
    const float aix = fabsf(r.inv.x), aiy = fabsf(r.inv.y), aiz = fabsf(r.inv.z);
    for (;;) {
        bool done = false;
        while (!is_leaf(node)) {
            ++nodes_visited;
            const float4 *nd = S.nodes4 + 8 * (size_t)node;
            const Node4 v4 = load_node4(nd);
            const int4 refs = v4.refs;
            const Slab4 sx = slab4(v4.x, r.inv.x, oix, aix), sy = slab4(v4.y, r.inv.y, oiy, aiy),
                        sz = slab4(v4.z, r.inv.z, oiz, aiz);
            // hit iff tn <= tf kSlabMargin: tn, or +inf on a miss, as an FMA, a product with +inf
            // (-inf or NaN on a hit) and a max, keeping the compare and select off the busier
            // ALU pipe
            float tn[4], tf[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                tn[c] = max3f(sx.n[c], sy.n[c], fmaxf(sz.n[c], tmin));
                tf[c] = min3f(sx.f[c], sy.f[c], fminf(sz.f[c], tbest));
            }
            const float2 m01 = mul2(fma2(make_float2(tf[0], tf[1]), -kSlabMargin, make_float2(tn[0], tn[1])), INFINITY);
            const float2 m23 = mul2(fma2(make_float2(tf[2], tf[3]), -kSlabMargin, make_float2(tn[2], tn[3])), INFINITY);
            const float d0 = fmaxf(tn[0], m01.x), d1 = fmaxf(tn[1], m01.y), d2 = fmaxf(tn[2], m23.x), d3 = fmaxf(tn[3], m23.y);
            float dmin = fminf(min3f(d0, d1, d2), d3);
            if (dmin < INFINITY) {
                if (SBR_CHECKED_ON && sp + 3 > S.stack_limit) {   // up to three pushes follow
                    check_fail(S, SBR_CHECK_TRACE_STACK);
                    t_out = tbest;
                    face_out = bface;
                    return -1;
                }
                int pick = d0 == dmin ? 0 : (d1 == dmin ? 1 : (d2 == dmin ? 2 : 3));
                if (d3 < INFINITY && pick != 3) { stack[sp] = refs.w; sdist[sp++] = d3; }
                if (d2 < INFINITY && pick != 2) { stack[sp] = refs.z; sdist[sp++] = d2; }
                if (d1 < INFINITY && pick != 1) { stack[sp] = refs.y; sdist[sp++] = d1; }
                if (d0 < INFINITY && pick != 0) { stack[sp] = refs.x; sdist[sp++] = d0; }
                node = pick == 0 ? refs.x : (pick == 1 ? refs.y : (pick == 2 ? refs.z : refs.w));
                continue;
            }
            if (!pop_near(stack, sdist, sp, tcull, node)) {
                done = true;
                break;
            }
        }
        if (done) break;
        {
            int first = leaf_first(node), cnt = leaf_count(node);
            for (int i = first; i < first + cnt; ++i) {
                const float4 *t = S.tris + 3 * (size_t)i;
                float4 a = __ldg(t), b = __ldg(t + 1), c = __ldg(t + 2);
                int f = __float_as_int(a.w);
                if (f == skip) continue;
                ++tris_tested;
                float th = tri_watertight(r, a, b, c);
                if (!(th > tmin) || th > tbest) continue;
                if (th < tbest || f < bface || (f == bface && i < best)) {
                    tbest = th;
                    best = i;
                    bface = f;
                }
            }
            tcull = tbest * kSlabMargin;
        }
        if (!pop_near(stack, sdist, sp, tcull, node)) break;
    }
    t_out = tbest;
    face_out = bface;
    return best;
}

// Any hit of the segment o + t d, t in (tmin, tmax), ignoring faces fa and fb, over the
// 4-wide BVH; inner nodes and leaves in nested loops as in closest_hit4.
__device__ __forceinline__ bool any_hit4(const SceneDev &S, const RayPre &r, float tmin, float tmax, int fa, int fb) {
    int stack[kStack4];
    int sp = 0;
    int node = 0;
    const float oix = r.o.x * r.inv.x, oiy = r.o.y * r.inv.y, oiz = r.o.z * r.inv.z;
    const float aix = fabsf(r.inv.x), aiy = fabsf(r.inv.y), aiz = fabsf(r.inv.z);
    for (;;) {
        bool done = false;
        while (!is_leaf(node)) {
            const float4 *nd = S.nodes4 + 8 * (size_t)node;
            const Node4 v4 = load_node4_wide(nd);
            const int4 refs = v4.refs;
            const Slab4 sx = slab4(v4.x, r.inv.x, oix, aix), sy = slab4(v4.y, r.inv.y, oiy, aiy),
                        sz = slab4(v4.z, r.inv.z, oiz, aiz);
            const int rf[4] = {refs.x, refs.y, refs.z, refs.w};
            int next = 0x7fffffff;
            if (SBR_CHECKED_ON && sp + 3 > S.stack_limit) {   // up to three pushes follow
                check_fail(S, SBR_CHECK_OCCLUSION_STACK);
                return false;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float tn = max3f(sx.n[c], sy.n[c], fmaxf(sz.n[c], tmin));
                float tf = min3f(sx.f[c], sy.f[c], fminf(sz.f[c], tmax)) * kSlabMargin;
                if (tn <= tf) {
                    if (next == 0x7fffffff) next = rf[c];
                    else stack[sp++] = rf[c];
                }
            }
            if (next != 0x7fffffff) {
                node = next;
                continue;
            }
            if (sp == 0) {
                done = true;
                break;
            }
            node = stack[--sp];
        }
        if (done) break;
        {
            int first = leaf_first(node), cnt = leaf_count(node);
            for (int i = first; i < first + cnt; ++i) {
                const float4 *t = S.tris + 3 * (size_t)i;
                float4 a = __ldg(t), b = __ldg(t + 1), c = __ldg(t + 2);
                int f = __float_as_int(a.w);
                if (f == fa || f == fb) continue;
                float th = tri_watertight(r, a, b, c);
                if (th > tmin && th < tmax) return true;
            }
        }
        if (sp == 0) break;
        node = stack[--sp];
    }
    return false;
}

// Largest foot parameter s = (p - o).d of any point p of box [lo, hi].
__device__ __forceinline__ float max_foot(const RxDev &R, float3 o, float3 d) {
    float s = (d.x > 0 ? R.hi[0] : R.lo[0]) * d.x + (d.y > 0 ? R.hi[1] : R.lo[1]) * d.y +
              (d.z > 0 ? R.hi[2] : R.lo[2]) * d.z;
    return s - dot(o, d);
}

}  // namespace sbr
