// kernels_paths.cu -- a5 double-count removal (§III.A, first path test): among reception
// records with the same (Tx, Rx, face sequence) keep the one with the smallest error
// angle of Eq. 3, ties to the lowest ray id.  Implemented as an open-addressing hash table
// keyed by a 64-bit hash of the face sequence with a 64-bit atomicMin on
// (error-angle bits, ray id); the pass that selects the winners checks every record against
// the record that claimed its slot, so that a hash collision is detected, never silently
// merged.
#include "dedup_keys.cuh"
#include "lattice_order.cuh"
#include "sbr_device.cuh"
#include "stream_launch.cuh"

namespace sbr {

__device__ __forceinline__ long long num_records(const DedupArgs &a) {
    long long n = a.counters[kRecords];
    return n < a.rec_cap ? n : a.rec_cap;
}

// slots in use for this launch (dedup_slots)
__device__ __forceinline__ unsigned long long used_slots(const DedupArgs &a) {
    return dedup_slots(num_records(a), a.slots);
}

// A slot is 16 bytes, its key then its value (one 32-byte sector holds two slots, so an
// insert's compare-and-swap and minimum touch one sector); the owners (the record that claimed
// each slot) follow the slots.  Keys and values to all-ones (empty / +inf) over the used slots.
__global__ void dedup_clear(DedupArgs a) {
    wait_predecessor();
    const unsigned long long m = used_slots(a);
    ulonglong2 *slot = reinterpret_cast<ulonglong2 *>(a.table);
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < m;
         i += (unsigned long long)gridDim.x * blockDim.x)
        slot[i] = make_ulonglong2(~0ULL, ~0ULL);
}

// A record or a path record moves as 32-byte pieces, a sector each: threads take whole records, so
// 16-byte accesses would pass every sector twice.
struct Piece {
    int w[8];
};
__device__ __forceinline__ Piece load_piece(const void *p) {
    Piece v;
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v.w[0]), "=r"(v.w[1]), "=r"(v.w[2]), "=r"(v.w[3]), "=r"(v.w[4]), "=r"(v.w[5]), "=r"(v.w[6]),
                   "=r"(v.w[7])
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ void store_piece(void *p, const Piece &v) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v.w[0]), "r"(v.w[1]),
                 "r"(v.w[2]), "r"(v.w[3]), "r"(v.w[4]), "r"(v.w[5]), "r"(v.w[6]), "r"(v.w[7])
                 : "memory");
}
__device__ __forceinline__ RecDev load_record(const RecDev *p) {
    static_assert(sizeof(RecDev) == 64 && kMaxOrder == 8, "the record is two pieces");
    const Piece a = load_piece(p), b = load_piece(reinterpret_cast<const char *>(p) + 32);
    RecDev r;
    r.tx = a.w[0], r.rx = a.w[1], r.ray = a.w[2], r.order = a.w[3];
#pragma unroll
    for (int j = 0; j < 4; ++j) r.faces[j] = a.w[4 + j], r.faces[4 + j] = b.w[j];
    r.err = __int_as_float(b.w[4]), r.dray = __int_as_float(b.w[5]), r.slot = b.w[6], r.pad = b.w[7];
    return r;
}

// A record's key and value are read before they are written: most records find their path's slot
// claimed (the office: 1.5M records, 236k paths), and many a smaller value in it, and then need no
// atomic.  Keys are written once and values only fall, so an old read costs an atomic, no more.
// Twice the blocks and this: 80 -> 75 us.  A table of 1.25 n instead of 2 n slots gave 4 us more
// but long probe runs once every record is a path of its own.
__global__ void dedup_insert(DedupArgs a) {
    wait_predecessor();
    int *owner = reinterpret_cast<int *>(a.table + 2 * a.slots);
    const long long n = num_records(a);
    unsigned long long *tab = a.table;   // key of slot s at 2 s, its value at 2 s + 1
    const unsigned long long used = used_slots(a), mask = used - 1;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const RecDev r = load_record(a.recs + i);
        unsigned long long h = rec_hash(r), v = rec_value(r);
        unsigned long long s = h & mask;
        for (unsigned long long probe = 0; probe < used; ++probe) {
            unsigned long long key, val;
            asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(key), "=l"(val) : "l"(tab + 2 * s) : "memory");
            if (key == ~0ULL) key = atomicCAS(tab + 2 * s, ~0ULL, h);
            if (key == ~0ULL || key == h) {
                if (v < val) atomicMin(tab + 2 * s + 1, v);
                if (key == ~0ULL) owner[s] = (int)i;
                a.recs[i].slot = (int)s;
                break;
            }
            s = (s + 1) & mask;
        }
    }
}

// Every slot's winner becomes a path, and every record is compared with the record that claimed
// its slot (a differing key is a hash collision): one pass over the records, where a pass of its own
// compared them with the winners (office, 1.5M records: 142 + 32 -> 140 us).  A warp takes places
// for all its winners with one atomic, and the records stay in registers (indexed by the order they
// had been in local memory): 123 -> 85 us for the office, 92 -> 55 for half of its records.  What
// is left are scattered 32-byte reads of the table and the owners' records, 4 TB/s in all; loading
// a record ahead, or more warps with fewer registers, changed nothing.
__global__ void dedup_select(DedupArgs a) {
    wait_predecessor();
    const long long n = num_records(a);
    const unsigned long long *tab = a.table;
    const int *owner = reinterpret_cast<const int *>(a.table + 2 * a.slots);
    const int lane = threadIdx.x & 31;
    unsigned bad = 0;
    for (long long first = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); first < n;
         first += (long long)gridDim.x * blockDim.x) {
        const long long i = first + lane;
        RecDev r;
        bool win = false;
        if (i < n) {
            r = load_record(a.recs + i);
            if (r.slot < 0) {
                ++bad;
            } else {
                const int o = owner[r.slot];
                win = tab[2 * (long long)r.slot + 1] == rec_value(r) &&
                      (a.shard_world <= 1 || (r.tx * a.nrx + r.rx) % a.shard_world == a.shard_rank);
                if (o != (int)i && !same_key(r, load_record(a.recs + o))) ++bad;
            }
        }
        const unsigned winners = __ballot_sync(0xffffffffu, win);
        if (winners == 0) continue;
        unsigned long long p = 0;
        if (lane == 0)
            p = atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kPaths), (unsigned long long)__popc(winners));
        p = __shfl_sync(0xffffffffu, p, 0) + __popc(winners & ((1u << lane) - 1u));
        if (!win || (long long)p >= a.path_cap) continue;
        union {
            sbr_path_record rec;
            Piece piece[4];
        } out;
        static_assert(sizeof(out) == sizeof(sbr_path_record) && sizeof(out) == 128, "the path record is four pieces");
        out.rec.tx = r.tx;
        out.rec.rx = r.rx;
        out.rec.ray = r.ray;
        out.rec.order = r.order;
#pragma unroll
        for (int j = 0; j < kMaxOrder; ++j) out.rec.faces[j] = r.faces[j];
        out.rec.rough_err = r.err;
        out.rec.rough_dray = r.dray;
        out.rec.iters = 0;
        out.rec.valid = 0;
        float4 d = __ldg(a.dirs + (a.sched_n > 0 ? schedule_place(r.ray, a.sched_n) : r.ray));
        out.rec.dir[0] = d.x;
        out.rec.dir[1] = d.y;
        out.rec.dir[2] = d.z;
        out.rec.err = r.err;
        out.rec.delay = 0.0;
        out.rec.aod[0] = out.rec.aod[1] = out.rec.aoa[0] = out.rec.aoa[1] = 0.0f;
        out.rec.power_dbm = 0.0f;
        out.rec.flags = 0;
        char *dst = reinterpret_cast<char *>(a.paths + p);
#pragma unroll
        for (int k = 0; k < 4; ++k) store_piece(dst + 32 * k, out.piece[k]);
    }
    if (bad) atomicAdd(reinterpret_cast<unsigned long long *>(a.counters + kCollisions), (unsigned long long)bad);
}


cudaError_t launch_dedup(const DedupArgs &a, int num_sms, cudaStream_t s) {
    int grid = num_sms * 8;
    cudaError_t e = launch_chained(dedup_clear, grid, 256, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(dedup_insert, grid, 256, 0, s, a);
    if (e == cudaSuccess) e = launch_chained(dedup_select, grid, 256, 0, s, a);
    return e;
}

__global__ void records_reset(long long *counters, long long n) {
    counters[kRecords] = n;
    counters[kPaths] = 0;
    counters[kCollisions] = 0;
    counters[kDiffPending] = 0;
}

cudaError_t launch_records_reset(long long *counters, long long n, cudaStream_t s) {
    records_reset<<<1, 1, 0, s>>>(counters, n);
    return cudaGetLastError();
}

// Valid paths with a non-finite output: an output scan (NaN / Inf in a valid path's
// direction, error angle, delay, angles or power means a numerical fault).
__device__ __forceinline__ bool finite_path(const sbr_path_record &p) {
    bool ok = isfinite(p.dir[0]) && isfinite(p.dir[1]) && isfinite(p.dir[2]) && isfinite(p.err) && isfinite(p.delay);
    ok = ok && isfinite(p.aod[0]) && isfinite(p.aod[1]) && isfinite(p.aoa[0]) && isfinite(p.aoa[1]);
    return ok && isfinite(p.power_dbm);
}

__global__ void nonfinite_scan(const sbr_path_record *paths, long long *counters, long long cap) {
    long long n = counters[kPaths];
    if (n > cap) n = cap;
    unsigned bad = 0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const sbr_path_record &p = paths[i];
        if (p.valid && !finite_path(p)) ++bad;
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && bad)
        atomicAdd(reinterpret_cast<unsigned long long *>(counters + kNonFinite), (unsigned long long)bad);
}

cudaError_t launch_nonfinite_scan(const sbr_path_record *paths, long long *counters, int64_t path_cap, int num_sms,
                                  cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(counters + kNonFinite, 0, sizeof(long long), s);
    if (e != cudaSuccess) return e;
    nonfinite_scan<<<num_sms * 4, 256, 0, s>>>(paths, counters, path_cap);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------- pairs
// Group path indices by (tx, rx) pair: counts, exclusive scan (one block), scatter.
__global__ void pair_count(PairArgs a) {
    long long n = a.counters[kPaths];
    if (n > a.path_cap) n = a.path_cap;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int p = a.paths[i].tx * a.nrx + a.paths[i].rx;
        atomicAdd(a.pair_count + p, 1);
    }
}

__global__ void pair_scan(PairArgs a) {
    // single block: exclusive scan of pair_count[0..npairs) into pair_count, total at [npairs]
    __shared__ int carry;
    __shared__ int buf[1024];
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < a.npairs; base += 1024) {
        int i = base + threadIdx.x;
        int v = i < a.npairs ? a.pair_count[i] : 0;
        buf[threadIdx.x] = v;
        __syncthreads();
        for (int off = 1; off < 1024; off <<= 1) {
            int t = threadIdx.x >= off ? buf[threadIdx.x - off] : 0;
            __syncthreads();
            buf[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < a.npairs) a.pair_count[i] = carry + buf[threadIdx.x] - v;
        __syncthreads();
        if (threadIdx.x == 1023) carry += buf[1023];
        __syncthreads();
    }
    if (threadIdx.x == 0) a.pair_count[a.npairs] = carry;
}

__global__ void pair_scatter(PairArgs a, int *cursor) {
    long long n = a.counters[kPaths];
    if (n > a.path_cap) n = a.path_cap;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        int p = a.paths[i].tx * a.nrx + a.paths[i].rx;
        int at = atomicAdd(cursor + p, 1);
        a.pair_idx[at] = (int)i;
    }
}

cudaError_t launch_pair_bucket(const PairArgs &a, cudaStream_t s) {
    // cursor lives after pair_idx: [npairs] ints (caller sized pair_idx + npairs)
    int *cursor = a.pair_idx + a.path_cap;
    cudaError_t e = cudaMemsetAsync(a.pair_count, 0, sizeof(int) * (size_t)(a.npairs + 1), s);
    if (e != cudaSuccess) return e;
    pair_count<<<256, 256, 0, s>>>(a);
    pair_scan<<<1, 1024, 0, s>>>(a);
    e = cudaMemcpyAsync(cursor, a.pair_count, sizeof(int) * (size_t)a.npairs, cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    pair_scatter<<<256, 256, 0, s>>>(a, cursor);
    return cudaGetLastError();
}

}  // namespace sbr
