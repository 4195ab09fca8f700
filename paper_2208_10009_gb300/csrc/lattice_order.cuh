// lattice_order.cuh -- index arithmetic of the equiangular lattice (§II.B) shared by ray
// generation, the trace and the diffraction search: the layer prefix and the schedule in
// which a launch keeps and takes its rays.
#pragma once

#include <cuda_runtime.h>

namespace sbr {

// interior points of layers 1..a of a face: S(a) = sum_{a'=1..a} 3(n - 3a') (fits 32 bits
// for n <= 14000)
__host__ __device__ __forceinline__ int layer_prefix(int n, int a) { return (6 * n * a - 9 * a * a - 9 * a) / 2; }

// ------------------------------------------------------------------ trace schedule
// The order in which a launch of the equiangular lattice generates its rays and the trace and
// the diffraction search take them (rays are independent, §III.A, so no result depends on it).
// Lattice id order runs along the rings of a face's layers (§II.B): the 24-32 consecutive ids
// of a warp's refill form a thin strip of directions.  The schedule puts the rays at places w in
// [0, N) so that consecutive ones form a compact patch instead.  The vertex and edge rays keep their ids.  A face's interior points
// are the triangular grid p0 + p1 + p2 = n, every p_k >= 1: layer a is the ring min(p) = a,
// and its side e runs from the layer's vertex e (nearest the face's corner e) towards vertex
// e + 1, so the ring index of (p0, p1, p2) is e (n - 3a) + j with (e, j) = (0, p1 - a) where
// p2 = a < p0, (1, p2 - a) where p0 = a < p1, and (2, p0 - a) where p1 = a < p2.  The points
// are taken in tiles of kTileRows values of p0 by kTileCols of p1, a block of rows at a time:
// its full tiles, then the rest of its rows (the staircase under the grid's diagonal); every
// other block runs the other way, so consecutive tiles stay neighbours.
constexpr int kTileRows = 6, kTileCols = 4;

// interior points in rows p0 = 1..x of a face (row p0 holds n - 1 - p0 of them)
__host__ __device__ __forceinline__ int rows_before(int n, int x) { return x * (n - 1) - x * (x + 1) / 2; }

// Grid point (p0, p1, n - p0 - p1) of a face: its layer a, the layer's edge length m (0: the face
// centre, n = 0 mod 3), its side e and the place j on it.
struct GridPoint {
    int a, m, e, j;
};

__host__ __device__ __forceinline__ GridPoint grid_point(int n, int p0, int p1) {
    const int p2 = n - p0 - p1;
    GridPoint g;
    g.a = min(p0, min(p1, p2));
    g.m = n - 3 * g.a;
    if (p2 == g.a && p0 > g.a) g.e = 0, g.j = p1 - g.a;
    else if (p0 == g.a && p1 > g.a) g.e = 1, g.j = p2 - g.a;
    else g.e = 2, g.j = p0 - g.a;
    return g;
}

// its ray id; face_base: the id of the face's first interior ray
__host__ __device__ __forceinline__ int grid_ray(int n, int face_base, const GridPoint &g) {
    return face_base + layer_prefix(n, g.a - 1) + (g.m == 0 ? 0 : g.e * g.m + g.j);
}

// The block of rows s..e (h of them) that holds row p0: its first place in the face's schedule,
// the columns fw of its full tiles (fw h points) and the points of its staircase.
struct RowBlock {
    int s, h, first, fw, full, stair;
    bool back;   // every other block runs backwards: its staircase first, then its tiles from the right
};

__host__ __device__ __forceinline__ RowBlock row_block(int n, int blk) {
    RowBlock b;
    b.s = blk * kTileRows + 1;
    const int e = min(b.s + kTileRows - 1, n - 2);
    b.h = e - b.s + 1;
    b.fw = (n - 1 - e) / kTileCols * kTileCols;
    b.full = b.fw * b.h;
    b.first = rows_before(n, b.s - 1);
    b.stair = rows_before(n, e) - b.first - b.full;
    b.back = blk & 1;
    return b;
}

// (p0, p1) of place q of block b
__host__ __device__ __forceinline__ void block_point(int n, const RowBlock &b, int q, int &p0, int &p1) {
    const int qt = b.back ? q - b.stair : q;
    if (qt >= 0 && qt < b.full) {
        const int size = kTileCols * b.h;
        // (the divisor of all but a face's last block is a constant)
        const int t = b.h == kTileRows ? qt / (kTileCols * kTileRows) : qt / size, rem = qt - t * size;
        p0 = b.s + rem / kTileCols;
        p1 = 1 + (b.back ? b.fw / kTileCols - 1 - t : t) * kTileCols + rem % kTileCols;
        return;
    }
    int qs = b.back ? q : q - b.full;
    for (p0 = b.s; p0 < b.s + b.h - 1; ++p0) {
        const int len = n - 1 - p0 - b.fw;
        if (qs < len) break;
        qs -= len;
    }
    p1 = b.fw + 1 + qs;
}

// The place of ray id `ray` in the schedule: the inverse of the order above.
__host__ __device__ __forceinline__ int schedule_place(int ray, int n) {
    const int E = 12 + 30 * (n - 1);
    if (ray < E) return ray;
    const int per_face = (n - 1) * (n - 2) / 2;
    const int r = ray - E, f = r / per_face, q = r - f * per_face;
    // layer a with S(a - 1) <= q < S(a): estimate from the quadratic, then fix
    const int nl = (n - 1) / 3;   // last layer
    const float B = 3.0f * n - 4.5f;
    int a = (int)((B - sqrtf(fmaxf(B * B - 18.0f * (float)q, 0.0f))) / 9.0f) + 1;
    a = max(1, min(a, nl));
    while (a > 1 && layer_prefix(n, a - 1) > q) --a;
    while (a < nl && layer_prefix(n, a) <= q) ++a;
    int p0, p1;
    const int m = n - 3 * a, b = q - layer_prefix(n, a - 1);
    if (3 * (a + 1) == n && q >= layer_prefix(n, a)) {   // the face centre (n = 0 mod 3)
        p0 = p1 = n / 3;
    } else if (m == 0) {
        p0 = p1 = a;
    } else {
        const int e = b / m, j = b - e * m;
        if (e == 0) p1 = a + j, p0 = n - a - p1;
        else if (e == 1) p0 = a, p1 = n - a - (a + j);
        else p1 = a, p0 = a + j;
    }
    const RowBlock k = row_block(n, (p0 - 1) / kTileRows);
    const int c = p1 - 1;
    int pos;
    if (c < k.fw) {
        const int t = c / kTileCols;
        pos = (k.back ? k.stair + (k.fw / kTileCols - 1 - t) * kTileCols * k.h : t * kTileCols * k.h) +
              (p0 - k.s) * kTileCols + c % kTileCols;
    } else {
        pos = (k.back ? 0 : k.full) + (c - k.fw);
        for (int x = k.s; x < p0; ++x) pos += n - 1 - x - k.fw;
    }
    return E + f * per_face + k.first + pos;
}

}  // namespace sbr
