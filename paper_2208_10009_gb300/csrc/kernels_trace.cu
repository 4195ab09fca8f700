// kernels_trace.cu -- a1 equiangular ray generation (§II.B, Eq. 1-2) and a2-a4 the
// persistent trace kernel: BVH closest hit with a watertight triangle test, specular
// reflection up to max_order (Fig. 4) and the reception judgment with the error angle
// of Eq. 3 on every segment.
#include "lattice_order.cuh"
#include "sbr_device.cuh"
#include "stream_launch.cuh"

namespace sbr {

// ----------------------------------------------------------------------------- a1
// Point j of m equal-angle steps along the great circle u -> v (angle om): Eq. 1 asks the
// points of a layer edge to subtend equal angles.  Normalised afterwards.
__device__ __forceinline__ float3 arc_point(float3 u, float3 v, float om, int j, int m) {
    float a = sinf(om * (float)(m - j) / (float)m);
    float b = sinf(om * (float)j / (float)m);
    float3 p = u * a + v * b;
    float inv = 1.0f / sqrtf(dot(p, p));
    return p * inv;
}


// One thread per ray; 32-bit index arithmetic (N < 2^31 for the supported n).
__global__ void raygen_kernel(LatticeDev L, float4 *__restrict__ dirs, int N) {
    const int n = L.n;
    const int n_edge = 30 * (n - 1);
    const int per_face = (n - 1) * (n - 2) / 2;
    const int layer_pts = layer_prefix(n, L.nl - 1);   // points on layers 1..nl-1
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        float3 d;
        if (id < 12) {
            d = f3(__ldg(L.ico + id));
        } else if (id < 12 + n_edge) {
            int r = id - 12;
            int e = r / (n - 1), j = r - e * (n - 1) + 1;
            int2 ed = __ldg(L.edges + e);
            d = arc_point(f3(__ldg(L.ico + ed.x)), f3(__ldg(L.ico + ed.y)), L.edge_angle, j, n);
        } else {
            int r = id - 12 - n_edge;
            int f = r / per_face;
            int q = r - f * per_face;
            if (q >= layer_pts) {
                d = f3(__ldg(L.centre + f));   // n = 0 mod 3: the face centre ray
            } else {
                // layer a >= 1 with S(a-1) <= q < S(a): estimate from the quadratic, then fix
                float B = 3.0f * n - 4.5f;
                float disc = fmaxf(B * B - 18.0f * (float)q, 0.0f);
                int a = (int)((B - sqrtf(disc)) / 9.0f) + 1;
                if (a < 1) a = 1;
                if (a > L.nl - 1) a = L.nl - 1;
                while (a > 1 && layer_prefix(n, a - 1) > q) --a;
                while (layer_prefix(n, a) <= q) ++a;
                int b = q - layer_prefix(n, a - 1);
                int m = n - 3 * a;
                int e = b / m, j = b - e * m;
                const float4 *W = L.layers + ((size_t)f * L.nl + a) * 3;
                float4 w0 = __ldg(W + e), w1 = __ldg(W + (e == 2 ? 0 : e + 1));
                d = arc_point(f3(w0), f3(w1), w0.w, j, m);
            }
        }
        dirs[id] = make_float4(d.x, d.y, d.z, 0.0f);
    }
}

// Transmitters as float4 and the launch's counters zeroed, by one block of the ray generation.
__device__ __forceinline__ void prepare_launch(const PrepArgs &p) {
    if (p.tx_src)
        for (int i = threadIdx.x; i < p.ntx; i += blockDim.x)
            p.tx[i] = make_float4(p.tx_src[3 * i], p.tx_src[3 * i + 1], p.tx_src[3 * i + 2], 0.0f);
    if (p.counters)
        for (int i = threadIdx.x; i < kNumCounters; i += blockDim.x) p.counters[i] = 0;
}

// The same rays at their places of the schedule, with their ids: the trace then reads a
// refill's rays as they lie, where it used to map each place to an id and a 64-bit work index to
// a transmitter by division (about 150 of the 560 instructions it spent on a segment besides its
// tree walk), once per transmitter.  A block takes one block of rows of a face (or 256 of the
// vertex and edge rays): the layer, side and place of a point follow from its grid coordinates,
// where the id order needs a quadratic search per ray.  Bound by the two sines and the
// divisions of arc_point, not by its 16 bytes a ray: n = 2200 (48.4M rays) 395 -> 297 us
// (2.6 TB/s); with it the large city's trace 37.22 -> 36.19 ms, the canyon's 852 -> 822 us, and a
// quarter range of the city's rays, in id order before, 16.27 -> 14.55 ms.
__global__ void __launch_bounds__(256) raygen_schedule_kernel(LatticeDev L, float4 *__restrict__ dirs, int edge_blocks,
                                                              int row_blocks, PrepArgs prep) {
    wait_predecessor();
    if (blockIdx.x == 0) prepare_launch(prep);
    const int n = L.n, E = 12 + 30 * (n - 1);
    if ((int)blockIdx.x < edge_blocks) {
        const int id = blockIdx.x * 256 + threadIdx.x;
        if (id >= E) return;
        float3 d;
        if (id < 12) {
            d = f3(__ldg(L.ico + id));
        } else {
            int r = id - 12;
            int e = r / (n - 1), j = r - e * (n - 1) + 1;
            int2 ed = __ldg(L.edges + e);
            d = arc_point(f3(__ldg(L.ico + ed.x)), f3(__ldg(L.ico + ed.y)), L.edge_angle, j, n);
        }
        dirs[id] = make_float4(d.x, d.y, d.z, __int_as_float(id));
        return;
    }
    const int item = blockIdx.x - edge_blocks, f = item / row_blocks;
    const RowBlock b = row_block(n, item - f * row_blocks);
    const int base = E + f * ((n - 1) * (n - 2) / 2), points = b.full + b.stair;
    float4 *out = dirs + base + b.first;
    for (int q = threadIdx.x; q < points; q += 256) {
        int p0, p1;
        block_point(n, b, q, p0, p1);
        const GridPoint g = grid_point(n, p0, p1);
        float3 d;
        if (g.m == 0) {
            d = f3(__ldg(L.centre + f));   // n = 0 mod 3: the face centre ray
        } else {
            const float4 *W = L.layers + ((size_t)f * L.nl + g.a) * 3;
            const float4 w0 = __ldg(W + g.e), w1 = __ldg(W + (g.e == 2 ? 0 : g.e + 1));
            d = arc_point(f3(w0), f3(w1), w0.w, g.j, g.m);
        }
        out[q] = make_float4(d.x, d.y, d.z, __int_as_float(grid_ray(n, base, g)));
    }
}

cudaError_t launch_raygen_schedule(const LatticeDev &lat, float4 *dirs, const PrepArgs &prep, cudaStream_t s) {
    const int edge_blocks = (12 + 30 * (lat.n - 1) + 255) / 256;
    const int row_blocks = lat.n > 2 ? (lat.n - 2 + kTileRows - 1) / kTileRows : 0;
    return launch_chained(raygen_schedule_kernel, edge_blocks + 20 * row_blocks, 256, 0, s, lat, dirs, edge_blocks, row_blocks,
                          prep);
}

cudaError_t launch_raygen(const LatticeDev &lat, float4 *dirs, int64_t N, cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long want = (N + 255) / 256;
    int grid = (int)(want < (long long)sms * 16 ? want : (long long)sms * 16);
    if (grid < 1) grid = 1;
    raygen_kernel<<<grid, 256, 0, s>>>(lat, dirs, (int)N);
    return cudaGetLastError();
}

// §II.A equidistant division: flat-face points projected onto the sphere.
// interior rows before row i of a face: sum_{i'=1}^{i-1} (n - 1 - i')
__device__ __forceinline__ long long row_prefix(int n, long long i) { return (i - 1) * (n - 1) - (i - 1) * i / 2; }

__global__ void raygen_equidistant_kernel(PolyDev P, float4 *__restrict__ dirs, long long N, bool tagged,
                                          PrepArgs prep) {
    wait_predecessor();
    if (blockIdx.x == 0) prepare_launch(prep);
    const int n = P.n;
    const long long n_edge = (long long)P.ne * (n - 1);
    const long long per_face = (long long)(n - 1) * (n - 2) / 2;
    for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < N;
         id += (long long)gridDim.x * blockDim.x) {
        float3 p;
        if (id < P.nv) {
            p = f3(__ldg(P.v + id));
        } else if (id < P.nv + n_edge) {
            long long r = id - P.nv;
            int e = (int)(r / (n - 1)), j = (int)(r % (n - 1)) + 1;
            int2 ed = __ldg(P.edges + e);
            float3 lo = f3(__ldg(P.v + ed.x)), hi = f3(__ldg(P.v + ed.y));
            p = lo + (hi - lo) * ((float)j / (float)n);
        } else {
            long long r = id - P.nv - n_edge;
            int f = (int)(r / per_face);
            long long q = r % per_face;
            // row i >= 1 with row_prefix(i) <= q < row_prefix(i + 1): estimate, then fix
            float B = (float)n - 1.5f;
            float disc = fmaxf(B * B - 2.0f * (float)q, 0.0f);
            long long i = (long long)(B - sqrtf(disc)) + 1;
            if (i < 1) i = 1;
            if (i > n - 2) i = n - 2;
            while (i > 1 && row_prefix(n, i) > q) --i;
            while (i < n - 2 && row_prefix(n, i + 1) <= q) ++i;
            int j = (int)(q - row_prefix(n, i)) + 1;
            int4 fc = __ldg(P.faces + f);
            float3 A = f3(__ldg(P.v + fc.x)), Bv = f3(__ldg(P.v + fc.y)), C = f3(__ldg(P.v + fc.z));
            p = A + (Bv - A) * ((float)i / (float)n) + (C - A) * ((float)j / (float)n);
        }
        float inv = 1.0f / sqrtf(dot(p, p));
        dirs[id] = make_float4(p.x * inv, p.y * inv, p.z * inv, tagged ? __int_as_float((int)id) : 0.0f);
    }
}

cudaError_t launch_raygen_equidistant(const PolyDev &P, float4 *dirs, int64_t N, bool tagged, const PrepArgs &prep,
                                      cudaStream_t s) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    long long want = (N + 255) / 256;
    int grid = (int)(want < (long long)sms * 16 ? want : (long long)sms * 16);
    if (grid < 1) grid = 1;
    return launch_chained(raygen_equidistant_kernel, grid, 256, 0, s, P, dirs, (long long)N, tagged, prep);
}

// ----------------------------------------------------------------------------- a2-a4
struct LaneRay {
    float3 o, d;
    float L;
    int k, prev, txi, ray;
    int place;   // of the schedule
};

// Receptions a lane buffers during one segment before its warp flushes them.  Emitting
// each record with its own atomic on the one record counter serialises the records at
// that counter's L2 slice (lanes are divergent inside the receiver leaves, so nothing
// aggregates them); the flush takes one atomic per warp step instead.  The buffer is a
// per-thread array in local memory (L1-cached); a segment can see many receivers when
// the cone has grown wide, so it holds kPend of them, and any further ones take their
// own slot at once.
constexpr int kPend = 16;

constexpr int kTailTake = 16;   // rays that a refill may ask for however few are left (trace_kernel)

// Shared memory of a trace block: the faces of each thread's ray, [kMaxOrder][block].
size_t trace_smem(int block) { return (size_t)kMaxOrder * block * sizeof(int); }

// The lane's pending receptions: receiver id, error angle and ray length of each (arrays
// in the thread's local memory), their count and the order of their segment (registers).
struct Pending {
    int *rx;
    float *err, *dray;
    int n, k;
    __device__ __forceinline__ int &rx_at(int i) { return rx[i]; }
    __device__ __forceinline__ float &err_at(int i) { return err[i]; }
    __device__ __forceinline__ float &dray_at(int i) { return dray[i]; }
};

__device__ __forceinline__ void write_record(const TraceArgs &a, unsigned long long slot, const LaneRay &st, int k,
                                             int rx, float err, float dray, const int *faces_sh, int stride_sh) {
    if ((long long)slot >= a.rec_cap) return;
    RecDev rec;
    rec.tx = st.txi;
    rec.rx = rx;
    rec.ray = st.ray;
    rec.order = k;
#pragma unroll
    for (int j = 0; j < kMaxOrder; ++j) rec.faces[j] = j < k ? faces_sh[j * stride_sh] : -1;
    rec.err = err;
    rec.dray = dray;
    rec.slot = -1;
    rec.pad = 0;
    int4 *dst = reinterpret_cast<int4 *>(a.recs + slot);
    const int4 *src = reinterpret_cast<const int4 *>(&rec);
#pragma unroll
    for (int j = 0; j < 4; ++j) dst[j] = src[j];
}

// A reception past the lane's kPend pending ones (rare): its own slot, written at once.
__device__ __noinline__ void emit_direct(const TraceArgs &a, const LaneRay &st, int rx, float err, float dray,
                                         const int *faces_sh, int stride_sh) {
    const unsigned long long slot = atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kRecords), 1ULL);
    write_record(a, slot, st, st.k, rx, err, dray, faces_sh, stride_sh);
}

// Whole warp: every lane's pending receptions get consecutive slots from one atomic (lane
// order, then reception order) and are written out.
__device__ __forceinline__ void flush_records(const TraceArgs &a, const LaneRay &st, const int *faces_sh,
                                              int stride_sh, Pending &pd, unsigned lane) {
    if (__ballot_sync(0xffffffffu, pd.n > 0) == 0) return;
    int incl = pd.n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (unsigned)o) incl += t;
    }
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kRecords), (unsigned long long)incl);
    base = __shfl_sync(0xffffffffu, base, 31) + (unsigned long long)(incl - pd.n);
    for (int i = 0; i < pd.n; ++i)
        write_record(a, base + i, st, pd.k, pd.rx_at(i), pd.err_at(i), pd.dray_at(i), faces_sh, stride_sh);
    pd.n = 0;
}

// slab4 for boxes grown by the radius: cn and cf are o / d with the growth taken off and added
__device__ __forceinline__ Slab4 slab4_grown(const NodeAxis &v, float inv, float cn, float cf, float ai) {
    const float2 n01 = fma2(v.h01, -ai, fma2s(v.c01.x, v.c01.y, inv, -cn));
    const float2 n23 = fma2(v.h23, -ai, fma2s(v.c23.x, v.c23.y, inv, -cn));
    const float2 f01 = fma2(v.h01, ai, fma2s(v.c01.x, v.c01.y, inv, -cf));
    const float2 f23 = fma2(v.h23, ai, fma2s(v.c23.x, v.c23.y, inv, -cf));
    return {{n01.x, n01.y, n23.x, n23.y}, {f01.x, f01.y, f23.x, f23.y}};
}

// Reception judgment on segment o + s d, s in [0, tseg], of a ray that has travelled L
// metres before it: every Rx whose foot lies on the segment and whose error angle
// (Eq. 3) is within the cone emits a record.  Candidates come from the receivers' 4-wide
// BVH, each box grown by the cone radius at the segment's far end; the growth is folded
// into the per-segment slab offsets (near: o/d + rad/|d|, far: o/d - rad/|d|), so a grown
// box costs what a plain one does.  Receptions go to the lane's pending buffer (past
// kPend in one segment, straight to the record array with their own atomic).
__device__ __forceinline__ void reception(const TraceArgs &a, const RayPre &r, const LaneRay &st, float tseg,
                                          const int *faces_sh, int stride_sh, Pending &pd, unsigned &rx_tests) {
    const RxDev &R = a.rx;
    if (R.nrx == 0) return;
    float tcap = fminf(tseg, max_foot(R, st.o, st.d));
    if (!(tcap >= 0.0f)) return;
    float rad = (st.L + tcap) * a.tan_cone * 1.001f + 1e-5f;
    const float oix = r.o.x * r.inv.x, oiy = r.o.y * r.inv.y, oiz = r.o.z * r.inv.z;
    const float aix = fabsf(r.inv.x), aiy = fabsf(r.inv.y), aiz = fabsf(r.inv.z);
    const float gx = rad * aix, gy = rad * aiy, gz = rad * aiz;
    const float cnx = oix + gx, cny = oiy + gy, cnz = oiz + gz;
    const float cfx = oix - gx, cfy = oiy - gy, cfz = oiz - gz;
    const float tfar = tcap * kSlabMargin + 1e-6f;
    {
        // the receivers' bounding box, grown like the node boxes: one slab test before the
        // walk (most segments, e.g. those rising above every receiver, end here; 2-3 %
        // of the trace measured on the canyon and the large city)
        const bool bx = r.inv.x < 0.0f, by = r.inv.y < 0.0f, bz = r.inv.z < 0.0f;
        const float nx = bx ? R.hi[0] : R.lo[0], fx = bx ? R.lo[0] : R.hi[0];
        const float ny = by ? R.hi[1] : R.lo[1], fy = by ? R.lo[1] : R.hi[1];
        const float nz = bz ? R.hi[2] : R.lo[2], fz = bz ? R.lo[2] : R.hi[2];
        const float tn = max3f(fmaf(nx, r.inv.x, -cnx), fmaf(ny, r.inv.y, -cny), fmaxf(fmaf(nz, r.inv.z, -cnz), 0.0f));
        const float tf = min3f(fmaf(fx, r.inv.x, -cfx), fmaf(fy, r.inv.y, -cfy), fminf(fmaf(fz, r.inv.z, -cfz), tfar));
        if (!(tn <= tf * kSlabMargin)) return;
    }
    int stack[kStack4];
    int sp = 0;
    int node = 0;
    for (;;) {
        if (!is_leaf(node)) {
            const float4 *nd = R.nodes4 + 8 * (size_t)node;
            const Node4 v4 = load_node4(nd);
            const int4 refs = v4.refs;
            const Slab4 sx = slab4_grown(v4.x, r.inv.x, cnx, cfx, aix), sy = slab4_grown(v4.y, r.inv.y, cny, cfy, aiy),
                        sz = slab4_grown(v4.z, r.inv.z, cnz, cfz, aiz);
            const int rf[4] = {refs.x, refs.y, refs.z, refs.w};
            int next = 0x7fffffff;
            if (SBR_CHECKED_ON && sp + 3 > a.scene.stack_limit) {   // up to three pushes follow
                check_fail(a.scene, SBR_CHECK_RX_STACK);
                return;
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                float tn = max3f(sx.n[c], sy.n[c], fmaxf(sz.n[c], 0.0f));
                float tf = min3f(sx.f[c], sy.f[c], fminf(sz.f[c], tfar)) * kSlabMargin;
                if (tn <= tf) {
                    if (next == 0x7fffffff) next = rf[c];
                    else stack[sp++] = rf[c];
                }
            }
            if (next != 0x7fffffff) {
                node = next;
                continue;
            }
        } else {
            int first = leaf_first(node), cnt = leaf_count(node);
            for (int i = first; i < first + cnt; ++i) {
                float4 p = __ldg(R.pts + i);
                ++rx_tests;
                float3 w = f3(p) - st.o;
                float s = dot(w, st.d);
                if (s < 0.0f || s > tseg) continue;
                float3 q = w - st.d * s;
                const float q2 = dot(q, q), dray = st.L + s;
                // far outside the cone (a margin of 1e-4 on tan^2 dwarfs the FP32 rounding):
                // rejected without the square root and arc tangent of the exact test
                if (q2 > a.tan2_pre * dray * dray) continue;
                float err = atan2f(sqrtf(q2), dray);
                if (!(err <= a.cone)) continue;
                if (pd.n < kPend) {
                    pd.rx_at(pd.n) = __float_as_int(p.w);
                    pd.err_at(pd.n) = err;
                    pd.dray_at(pd.n) = dray;
                    ++pd.n;
                } else {
                    emit_direct(a, st, __float_as_int(p.w), err, dray, faces_sh, stride_sh);
                }
            }
        }
        if (sp == 0) break;
        node = stack[--sp];
    }
}

// ----------------------------------------------------------------------------- frontier
// Interval of 1 / |d| over a beam's directions on one axis, the sign of d, and whether d changes
// sign (then s = 0: only |centre - o| - half extent bounds the entry, and nothing the exit).
struct BeamAxis {
    float o, s, lo, hi;
};

__device__ __forceinline__ BeamAxis beam_axis(float o, float dl, float dh) {
    BeamAxis b;
    const float al = fminf(fabsf(dl), fabsf(dh)), ah = fmaxf(fabsf(dl), fabsf(dh));
    const bool cross = !(dl * dh > 0.0f);
    b.o = o;
    b.s = cross ? 0.0f : (dl > 0.0f ? 1.0f : -1.0f);
    b.lo = __fdividef(1.0f, ah) * 0.999999f;
    b.hi = cross || al < 1e-30f ? INFINITY : __fdividef(1.0f, al) * 1.000001f;
    return b;
}

// Bounds over the beam of where its rays enter (not before) and leave (not after) a slab.  The intervals
// of the directions (1e-6 wider on either side) and of their reciprocals (1e-6) cover their own rounding.
// p - h rounds by 6e-8 of |centre - o| and so bounds the entry to that, the size of what a ray's own slab
// test loses when it rounds o / d.  (Tx within 1 mm to 1 m of walls, roofs and the ground, 1.3e9 first
// segments: all segments as from the root.)
__device__ __forceinline__ void beam_slab(const BeamAxis &b, float c, float h, float &tn, float &tf) {
    const float x = c - b.o, p = b.s == 0.0f ? fabsf(x) : x * b.s;
    const float np = p - h, fp = p + h;
    tn = fmaxf(tn, fminf(np * b.lo, np * b.hi));
    tf = fminf(tf, fmaxf(fp * b.lo, fp * b.hi));
}

// The frontier of the first segments: a group's rays leave Tx within a degree or less of each
// other and would each walk the same upper tree; one thread walks it for all of them with the
// interval of their directions, always opening the nearest inner node, until the list is full or
// kFrontOpen nodes were opened.
// A ray then starts among a few nodes and leaves next to what it hits, and a group that looks
// into the sky has an empty list.  (First segments are 43 % of the large city's segments and a
// third of its node visits.)  Groups of 32 / 64 / 128 places cost the trace the same (29.4-29.5 ms on
// the city) and themselves 1,050 / 617 / 548 us there, 67 / 51 / 100 us on the canyon, where one
// thread's chain of openings is what it waits for; 6 / 8 / 12 entries: 29.9 / 29.4 / 29.4 ms.
// Large city trace 34.6 -> 29.5 ms + 0.62, canyon 820 -> 714 us + 51.
__global__ void __launch_bounds__(128) frontier_kernel(FrontArgs A) {
    wait_predecessor();
    const int lane = threadIdx.x & 31;
    const long long g0 = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32;
    if (g0 >= A.groups) return;
    // directions' intervals: the warp reads group by group, lane g keeps group g's.  d + 2 is positive,
    // so its bits order like it; its rounding (2^-22) is given back below.
    float lo[3] = {1.0f, 1.0f, 1.0f}, hi[3] = {-1.0f, -1.0f, -1.0f};
    bool some = false;
#pragma unroll 4
    for (int g = 0; g < 32; ++g) {
        unsigned mn[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, mx[3] = {0, 0, 0}, any = 0;
#pragma unroll
        for (int q = 0; q < kFrontRays; q += 32) {
            const long long place = (A.group0 + g0 + g) * kFrontRays + q + lane;
            if (g0 + g >= A.groups || place < A.first || place >= A.first + A.count) continue;
            const float4 dd = __ldg(A.dirs + place);
            const int ray = __float_as_int(dd.w);
            if (ray < A.ray_begin || ray >= A.ray_end) continue;
            const float v[3] = {dd.x, dd.y, dd.z};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const unsigned u = __float_as_uint(v[k] + 2.0f);
                mn[k] = min(mn[k], u);
                mx[k] = max(mx[k], u);
            }
            any = 1;
        }
        any = __any_sync(0xffffffffu, any);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            mn[k] = __reduce_min_sync(0xffffffffu, mn[k]);
            mx[k] = __reduce_max_sync(0xffffffffu, mx[k]);
            if (lane == g) {
                lo[k] = __uint_as_float(mn[k]) - 2.0f - 1e-6f;
                hi[k] = __uint_as_float(mx[k]) - 2.0f + 1e-6f;
            }
        }
        if (lane == g) some = any;
    }
    if (g0 + lane >= A.groups) return;
    for (int t = 0; t < A.ntx; ++t) {
        // the list stays in registers: every loop over it is unrolled.  Past its n entries dist = +inf.
        int ref[kFrontEntries];
        float dist[kFrontEntries];
#pragma unroll
        for (int j = 0; j < kFrontEntries; ++j) {
            ref[j] = kNoRef;
            dist[j] = INFINITY;
        }
        int n = 0;
        if (some) {
            const float3 o = f3(__ldg(A.tx + t));
            const BeamAxis bx = beam_axis(o.x, lo[0], hi[0]), by = beam_axis(o.y, lo[1], hi[1]), bz = beam_axis(o.z, lo[2], hi[2]);
            ref[0] = 0;
            dist[0] = 0.0f;
            n = 1;
            // the nearest inner node is opened while its four children fit
            for (int opened = 0; n <= kFrontEntries - 3 && opened < kFrontOpen; ++opened) {
                int node = -1;
                bool gone = false;
#pragma unroll
                for (int j = 0; j < kFrontEntries; ++j) {   // found: taken out, the entries after it move up
                    if (!gone && ref[j] != kNoRef && !is_leaf(ref[j])) {
                        node = ref[j];
                        gone = true;
                    }
                    if (gone) {
                        ref[j] = j + 1 < kFrontEntries ? ref[j + 1 < kFrontEntries ? j + 1 : j] : kNoRef;
                        dist[j] = j + 1 < kFrontEntries ? dist[j + 1 < kFrontEntries ? j + 1 : j] : INFINITY;
                    }
                }
                if (node < 0) break;
                --n;
                const Node4 v = load_node4(A.scene.nodes4 + 8 * (size_t)node);
                const float cx[4] = {v.x.c01.x, v.x.c01.y, v.x.c23.x, v.x.c23.y}, hx[4] = {v.x.h01.x, v.x.h01.y, v.x.h23.x, v.x.h23.y};
                const float cy[4] = {v.y.c01.x, v.y.c01.y, v.y.c23.x, v.y.c23.y}, hy[4] = {v.y.h01.x, v.y.h01.y, v.y.h23.x, v.y.h23.y};
                const float cz[4] = {v.z.c01.x, v.z.c01.y, v.z.c23.x, v.z.c23.y}, hz[4] = {v.z.h01.x, v.z.h01.y, v.z.h23.x, v.z.h23.y};
                const int rf[4] = {v.refs.x, v.refs.y, v.refs.z, v.refs.w};
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float tn = 0.0f, tf = INFINITY;
                    beam_slab(bx, cx[c], hx[c], tn, tf);
                    beam_slab(by, cy[c], hy[c], tn, tf);
                    beam_slab(bz, cz[c], hz[c], tn, tf);
                    if (!(tn <= tf * 1.000001f) || rf[c] == leaf_ref(0, 0)) continue;
                    ++n;
                    // behind the entries at most as far
#pragma unroll
                    for (int j = kFrontEntries - 1; j >= 0; --j) {
                        const bool before = j > 0 && dist[j > 0 ? j - 1 : 0] > tn;   // the one before moves here
                        const bool here = !before && dist[j] > tn;
                        if (before) {
                            ref[j] = ref[j > 0 ? j - 1 : 0];
                            dist[j] = dist[j > 0 ? j - 1 : 0];
                        } else if (here) {
                            ref[j] = rf[c];
                            dist[j] = tn;
                        }
                    }
                }
            }
        }
        int4 *out = reinterpret_cast<int4 *>(A.front + ((size_t)t * A.groups + g0 + lane) * kFrontEntries);
#pragma unroll
        for (int j = 0; j < kFrontEntries; j += 2)
            out[j / 2] = make_int4(ref[j], __float_as_int(dist[j]), ref[j + 1], __float_as_int(dist[j + 1]));
    }
}

cudaError_t launch_frontier(const FrontArgs &a, cudaStream_t s) {
    return launch_chained(frontier_kernel, (unsigned)((a.groups + 127) / 128), 128, 0, s, a);
}

// Persistent trace kernel.  Each warp keeps 32 rays in registers; after a segment, once at
// least refill_min lanes hold a finished ray (miss or order cap), those lanes take fresh,
// consecutive places of the schedule from a global counter with
// one warp-aggregated atomic (ballot + popc).  Waiting for several idle lanes keeps a warp's
// rays neighbours on the sphere (coherent traversal) while still keeping warps mostly full
// until the pool drains.  After
// every segment step the warp writes out its lanes' receptions together (flush_records).
// Seven 128-thread blocks per SM (72 registers, no spills) measured faster than eight (64
// registers, spilled).
__global__ void __launch_bounds__(128, 7) trace_kernel(TraceArgs a) {
    wait_predecessor();
    extern __shared__ int faces_sh_all[];   // trace_smem(blockDim.x) bytes
    int *faces_sh = faces_sh_all + threadIdx.x;
    const int stride_sh = blockDim.x;
    int pend_rx[kPend];
    float pend_err[kPend], pend_dray[kPend];
    Pending pd;
    pd.rx = pend_rx;
    pd.err = pend_err;
    pd.dray = pend_dray;
    pd.n = 0;
    const unsigned lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const long long total = (long long)a.ntx * a.count;
    unsigned seg = 0, nodes = 0, tris = 0, rxt = 0;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    int quota = 32;
    bool alive = false, pool_empty = false;
    LaneRay st;
    st.o = st.d = make_float3(0, 0, 0);
    st.L = 0.0f;
    st.k = st.prev = st.txi = st.ray = st.place = 0;
    for (;;) {
        unsigned need = __ballot_sync(0xffffffffu, !alive);
        if (need && !pool_empty && (__popc(need) >= a.refill_min || need == 0xffffffffu)) {
            // near the pool's end no more than a warp's share of what was left: full takes leave
            // the last rays to a few warps.  (One of four shards of the large city 13.15 -> 13.05
            // ms, the whole 31.46 -> 31.34; floors of 4 and 8 measure the same.  Not for a warp's
            // first take: a launch with fewer rays than lanes then runs in more, emptier warps, a
            // room's trace 26 -> 30 us.)
            const int take = min(__popc(need), quota);
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kRayHead),
                                            (unsigned long long)take);
            base = __shfl_sync(0xffffffffu, base, 0);
            if ((long long)base >= total) pool_empty = true;
            quota = min(32, max(kTailTake, (int)min(32LL, (total - (long long)base) / nwarps)));
            if (!alive) {
                const int turn = __popc(need & lt_mask);
                long long gid = (long long)base + turn;
                if (turn < take && gid < total) {
                    // its transmitter, by a product instead of a 64-bit division, then fixed
                    st.txi = a.ntx == 1 ? 0 : (int)((float)gid * a.inv_count);
                    long long local = gid - (long long)st.txi * a.count;
                    while (local < 0) local += a.count, --st.txi;
                    while (local >= a.count) local -= a.count, ++st.txi;
                    int place = (int)(a.first + local);
                    if (a.id_order_n > 0) place = schedule_place(place, a.id_order_n);
                    const float4 dd = __ldg(a.dirs + place);
                    st.o = f3(__ldg(a.tx + st.txi));
                    st.d = f3(dd);
                    st.ray = __float_as_int(dd.w);
                    st.place = place;
                    st.L = 0.0f;
                    st.k = 0;
                    st.prev = -1;
                    alive = st.ray >= a.ray_begin && st.ray < a.ray_end;
                    if (alive && a.dump_stride > 0 && st.ray % a.dump_stride == 0) {
                        int *df = a.dump_faces + ((size_t)st.txi * a.dump_per_tx + st.ray / a.dump_stride) *
                                                     (a.max_order + 1);
                        for (int j = 0; j <= a.max_order; ++j) df[j] = -2;
                    }
                }
            }
        }
        if (__ballot_sync(0xffffffffu, alive) == 0) {
            if (pool_empty) break;
            continue;   // a range passed over every place taken
        }
        if (alive) {
            RayPre r = make_ray(st.o, st.d);
            const int4 *first = nullptr;
            if (a.front && st.k == 0)
                first = reinterpret_cast<const int4 *>(
                    a.front + ((size_t)st.txi * a.groups + (st.place / kFrontRays - a.group0)) * kFrontEntries);
            float th;
            int face;
            const int hit = closest_hit4(a.scene, r, a.scene.tmin, INFINITY, st.prev,
                                         first, th, face, nodes, tris);
            ++seg;
            if (a.dump_stride > 0 && st.ray % a.dump_stride == 0)
                a.dump_faces[((size_t)st.txi * a.dump_per_tx + st.ray / a.dump_stride) * (a.max_order + 1) + st.k] =
                    hit >= 0 ? face : -1;
            float tseg = hit >= 0 ? th : INFINITY;
            pd.k = st.k;
            reception(a, r, st, tseg, faces_sh, stride_sh, pd, rxt);
            if (SBR_CHECKED_ON && hit >= 0 && (unsigned)face >= (unsigned)a.scene.nf) {
                check_fail(a.scene, SBR_CHECK_FACE_ID);
                alive = false;
            } else if (hit < 0 || st.k == a.max_order) {
                alive = false;
            } else {
                // specular reflection on the hit face's plane (faces_sh[j], j < pd.k, stay
                // as the pending receptions need them)
                float4 pl = __ldg(a.scene.planes + face);
                float3 nrm = f3(pl);
                st.o = st.o + st.d * th;
                st.d = st.d - nrm * (2.0f * dot(st.d, nrm));
                st.L += th;
                faces_sh[st.k * stride_sh] = face;
                st.prev = face;
                ++st.k;
            }
        }
        flush_records(a, st, faces_sh, stride_sh, pd, lane);
    }
    // one atomic per warp per counter
    unsigned s0 = __reduce_add_sync(0xffffffffu, seg), s1 = __reduce_add_sync(0xffffffffu, nodes);
    unsigned s2 = __reduce_add_sync(0xffffffffu, tris), s3 = __reduce_add_sync(0xffffffffu, rxt);
    if (lane == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kSegments), (unsigned long long)s0);
        atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kNodeVisits), (unsigned long long)s1);
        atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kTriTests), (unsigned long long)s2);
        atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kRxTests), (unsigned long long)s3);
    }
}

int trace_blocks_per_sm(int block) {
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, trace_kernel, block, trace_smem(block));
    return nb > 0 ? nb : 1;
}

cudaError_t launch_trace(const TraceArgs &a, int grid, int block, cudaStream_t s) {
    return launch_chained(trace_kernel, grid, block, trace_smem(block), s, a);
}

}  // namespace sbr
