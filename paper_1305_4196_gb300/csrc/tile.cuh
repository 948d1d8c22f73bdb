// tile.cuh - the on-chip neighbourhood of one 2x2x2-cell block.
//
// A cell task of the paper (Sec. II.A) reads the particles of its cell and
// of the 26 surrounding cells.  Blocking 2x2x2 cells into one task
// (Sec. II.D.2) widens that neighbourhood to the 4x4x4 cells around the
// block: the "tile".  One CTA stages its tile in shared memory once and
// serves every list build / force evaluation of its block from there, so the
// neighbour lists can hold 16-bit tile-local indices.
//
// Tile order: the block's own 8 cells first (in the block's cell order, so
// the block's atoms keep their cell-sorted order and own atom k has tile
// index k), then the other 56 cells of the 4x4x4 neighbourhood, x fastest.
// Coordinates in the tile are FP32, relative to the block centre: each
// atom's FP32 offset from its own cell centre plus the (t - 3/2) cell-width
// offset of its tile cell, which is the same for every periodic image.
#pragma once

#include "mdgb_internal.cuh"

namespace mdgb {

struct TileTables {
    int8_t coord_of_idx[64];  // tile slot -> tile coordinate
};

// Tile cell (x, y, z) (0..3 each; the block's own cells are 1..2) is a Newton-3 half-shell
// target of some own cell: the cell itself, or a forward neighbour (dz > 0; dz = 0 and
// dy > 0; dz = dy = 0 and dx > 0; Sec. II.D.3).  Half-list reactions only reach these.
__host__ __device__ constexpr bool tile_receives(int x, int y, int z) {
    for (int oz = 1; oz <= 2; ++oz)
        for (int oy = 1; oy <= 2; ++oy)
            for (int ox = 1; ox <= 2; ++ox) {
                const int dx = x - ox, dy = y - oy, dz = z - oz;
                if (dx < -1 || dx > 1 || dy < -1 || dy > 1 || dz < -1 || dz > 1) continue;
                if (dz > 0 || (dz == 0 && (dy > 0 || (dy == 0 && dx >= 0)))) return true;
            }
    return false;
}

// Slots: the 8 own cells first, then the other cells a half list reaches, then the rest.
// So the own atoms are tile entries 0 .. prefix[8] - 1 and every half-list target lies in
// entries 0 .. prefix[TILE_RECV_CELLS] - 1.
constexpr int TILE_RECV_CELLS = 43;

__host__ __device__ constexpr TileTables make_tile_tables() {
    TileTables t{};
    int k = 8, r = TILE_RECV_CELLS;
    for (int c = 0; c < 64; ++c) {
        int x = c & 3, y = (c >> 2) & 3, z = c >> 4;
        bool own = x >= 1 && x <= 2 && y >= 1 && y <= 2 && z >= 1 && z <= 2;
        int i = own ? (x - 1) + 2 * (y - 1) + 4 * (z - 1) : (tile_receives(x, y, z) ? k++ : r++);
        t.coord_of_idx[i] = (int8_t)c;
    }
    return t;
}

__host__ __device__ constexpr int count_tile_receivers() {
    int k = 0;
    for (int c = 0; c < 64; ++c) k += tile_receives(c & 3, (c >> 2) & 3, c >> 4) ? 1 : 0;
    return k;
}
static_assert(count_tile_receivers() == TILE_RECV_CELLS, "half-shell targets of a 2x2x2 block");

// Entries of the reaction sums a mixed half-list CTA keeps for a tile capacity: 11/16 of
// it (the 43 of 64 cells a half list reaches hold about 2/3 of a tile's atoms), and the
// smallest tile capacity whose share holds `recv` entries.
__host__ __device__ inline int half_recv_cap(int tile_cap) { return ((tile_cap * 11 + 15) / 16 + 31) & ~31; }
__host__ __device__ inline int tile_cap_for_recv(int recv) { return (recv * 16 + 10) / 11; }

// Tile coordinate of slot t, from the table as 2-bit digits in immediate operands: an indexed read
// of constant memory takes some 600 cycles here, which every CTA would wait for before its
// first load (and once per cell while staging; those read TileMeta instead).
__host__ __device__ constexpr unsigned long long tile_digits(int axis, int half) {
    constexpr TileTables t = make_tile_tables();
    unsigned long long v = 0;
    for (int k = 0; k < 32; ++k)
        v |= (unsigned long long)((t.coord_of_idx[32 * half + k] >> (2 * axis)) & 3) << (2 * k);
    return v;
}

__device__ __forceinline__ int tile_coord_of(int t) {
    constexpr unsigned long long x0 = tile_digits(0, 0), x1 = tile_digits(0, 1), y0 = tile_digits(1, 0),
                                 y1 = tile_digits(1, 1), z0 = tile_digits(2, 0), z1 = tile_digits(2, 1);
    const int sh = 2 * (t & 31);
    const bool lo = t < 32;
    const int x = (int)((lo ? x0 : x1) >> sh) & 3, y = (int)((lo ? y0 : y1) >> sh) & 3,
              z = (int)((lo ? z0 : z1) >> sh) & 3;
    return x + 4 * y + 16 * z;
}

// Cell id at tile coordinate c of the block with coordinates (bx, by, bz).
__device__ __forceinline__ int tile_cell_id(const Geometry& g, int bx, int by, int bz, int c) {
    const int tx = c & 3, ty = (c >> 2) & 3, tz = c >> 4;
    int cx = 2 * bx - 1 + tx, cy = 2 * by - 1 + ty, cz = 2 * bz - 1 + tz;
    cx += cx < 0 ? g.nc[0] : (cx >= g.nc[0] ? -g.nc[0] : 0);
    cy += cy < 0 ? g.nc[1] : (cy >= g.nc[1] ? -g.nc[1] : 0);
    cz += cz < 0 ? g.nc[2] : (cz >= g.nc[2] ? -g.nc[2] : 0);
    return cell_id_of(g, cx, cy, cz);
}

// Fill meta for block b (threads 0..63 of the CTA take part; ends with __syncthreads).
__device__ __forceinline__ void tile_meta(const Geometry& g, const int32_t* __restrict__ cell_start, int b,
                                          TileMeta& m) {
    const int t = threadIdx.x;
    if (t < 64) {
        int bx, by, bz;
        block_coords(g, b, bx, by, bz);
        const int c = tile_coord_of(t);
        int id = tile_cell_id(g, bx, by, bz, c);
        int st = cell_start[id];
        int cnt = cell_start[id + 1] - st;
        m.start[t] = st;
        m.coord[t] = (int8_t)c;
        m.slot[c] = (int8_t)t;
        // inclusive scan of the 64 counts over two warps
        int lane = t & 31;
        int v = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        m.prefix[t + 1] = v;  // warp-local inclusive prefix for now
    }
    __syncthreads();
    if (t >= 32 && t < 64) m.prefix[t + 1] += m.prefix[32];
    if (t == 0) m.prefix[0] = 0;
    __syncthreads();
}

// Tile slot holding tile index u (binary search in the 65-entry prefix).
__device__ __forceinline__ int tile_slot_of(const TileMeta& m, int u) {
    int lo = 0, hi = 64;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (m.prefix[mid] <= u) lo = mid; else hi = mid;
    }
    return lo;
}

// The FP64 pair test of the definition, in the oracle's operation order: minimum image
// d - L*rint(d/L) per dimension, r^2 = ((dx*dx) + dy*dy) + dz*dz, strict r^2 < cut2.
// Used wherever an FP32 distance lies too close to a threshold (list radius or cutoff)
// to decide the comparison.
__device__ __forceinline__ double mic_rn(double d, double L) {
    return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

__device__ __forceinline__ bool fp64_pair_test(const double* __restrict__ x, const double* __restrict__ y,
                                            const double* __restrict__ z, double Lx, double Ly, double Lz, int i,
                                            int j, double rl2) {
    double dx = mic_rn(__dsub_rn(x[i], x[j]), Lx);
    double dy = mic_rn(__dsub_rn(y[i], y[j]), Ly);
    double dz = mic_rn(__dsub_rn(z[i], z[j]), Lz);
    double r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return r2 < rl2;
}

// Cell-ordered global index of tile index u.
__device__ __forceinline__ int tile_global_index(const TileMeta& m, int u) {
    const int slot = tile_slot_of(m, u);
    return m.start[slot] + (u - m.prefix[slot]);
}

// o[t] for t in 0..3, where o = (-3/2, -1/2, 1/2, 3/2) w: by two selects (dynamic indexing would
// copy the table to local memory, and nested conditions compile to branches: 600 cycles for
// the six offsets of two tile cells)
__device__ __forceinline__ float pick4(const float (&o)[4], int t) {
    const float a = ((t + 1) & 2) ? o[2] : o[3];  // t = 1, 2: the inner cells
    return __int_as_float(__float_as_int(a) ^ (t < 2 ? (int)0x80000000 : 0));
}

// Stage the block-frame FP32 coordinates of the tile, one warp per tile cell (lanes
// over the cell's atoms, two cells per step so that two loads are in flight).  W: the .w
// entries from w (one value per atom, read from L2) in place of the species bits.
template <bool W = false>
__device__ __forceinline__ void tile_stage_f32_cells(const TileMeta& m, const float4* __restrict__ xr,
                                                     const TileOffsets& to, float4* __restrict__ tile,
                                                     const float* __restrict__ w = nullptr) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int slot = warp; slot < 64; slot += 2 * nw) {
        const int slot2 = slot + nw;
        const int c = m.coord[slot];
        const int u0 = m.prefix[slot], cnt = m.prefix[slot + 1] - u0, j0 = m.start[slot];
        const int c2 = slot2 < 64 ? m.coord[slot2] : 0;
        const int v0 = slot2 < 64 ? m.prefix[slot2] : 0;
        const int cnt2 = slot2 < 64 ? m.prefix[slot2 + 1] - v0 : 0;
        const int k0 = slot2 < 64 ? m.start[slot2] : 0;
        const float ox = pick4(to.off[0], c & 3), oy = pick4(to.off[1], (c >> 2) & 3), oz = pick4(to.off[2], c >> 4);
        const float ox2 = pick4(to.off[0], c2 & 3), oy2 = pick4(to.off[1], (c2 >> 2) & 3),
                    oz2 = pick4(to.off[2], c2 >> 4);
        const int most = cnt > cnt2 ? cnt : cnt2;
        for (int e = lane; e < most; e += 32) {
            float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p;
            if (e < cnt) p = xr[j0 + e];
            if (e < cnt2) q = xr[k0 + e];
            if (W) {
                if (e < cnt) p.w = __ldcg(w + j0 + e);
                if (e < cnt2) q.w = __ldcg(w + k0 + e);
            }
            if (e < cnt) tile[u0 + e] = make_float4(p.x + ox, p.y + oy, p.z + oz, p.w);
            if (e < cnt2) tile[v0 + e] = make_float4(q.x + ox2, q.y + oy2, q.z + oz2, q.w);
        }
    }
}

constexpr int STAGE64_AHEAD = 4;

// The tile cells (bit per slot) that the lists of a CTA's own atoms can reach, when CTAs share a block
// and this one takes `per` own atoms from part * per on (and every split * per): the cells around
// those own cells.  Every lane of a warp gets the mask.
__device__ __forceinline__ unsigned long long tile_needed(const TileMeta& m, int part, int split, int per) {
    const int lane = threadIdx.x & 31;
    const int lo = part * per, hi = split * per >= m.prefix[8] ? lo + per : m.prefix[8];
    const bool own = lane < 8 && m.prefix[lane & 7] < hi && m.prefix[(lane & 7) + 1] > lo;
    const unsigned touched = __ballot_sync(0xffffffffu, own);  // own cell 1 + (o & 1), 1 + (o >> 1 & 1), 1 + (o >> 2)
    unsigned half[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = m.coord[lane + 32 * h], x = c & 3, y = (c >> 2) & 3, z = c >> 4;
        const unsigned near = (x == 0 ? 0x55u : (x == 3 ? 0xaau : 0xffu)) & (y == 0 ? 0x33u : (y == 3 ? 0xccu : 0xffu)) &
                              (z == 0 ? 0x0fu : (z == 3 ? 0xf0u : 0xffu));
        half[h] = __ballot_sync(0xffffffffu, (near & touched) != 0u);
    }
    return half[0] | ((unsigned long long)half[1] << 32);
}

// The cells of `need` as a prefix over the tile slots, like TileMeta::prefix: pre[64] is the number of their
// atoms.  By the CTA's first warp; ends with __syncthreads.
__device__ __forceinline__ void tile_needed_prefix(const TileMeta& m, unsigned long long need, int (&pre)[65]) {
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x, a = 2 * lane;
        const int c0 = need >> a & 1 ? m.prefix[a + 1] - m.prefix[a] : 0;
        const int c1 = need >> (a + 1) & 1 ? m.prefix[a + 2] - m.prefix[a + 1] : 0;
        int v = c0 + c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane == 0) pre[0] = 0;
        pre[a + 1] = v - c1;
        pre[a + 2] = v;
    }
    __syncthreads();
}

// Stage the FP64 tile of block b: coordinates relative to the block centre (periodic
// images shifted by one box length where the tile wraps), species, and a dummy slot T
// far outside every cutoff.  pre: the atoms to stage, by slot (m.prefix: all; tile_needed_prefix).
// A lane per atom over the cells' borders, as a warp's FP64 addition takes 16 cycles of the SM however few
// of its lanes take part; STAGE64_AHEAD atoms of a lane on their way together (a CTA with an SM to
// itself waits for nothing else).  Full-list forces with a warp per cell and so: 62,500 atoms with 2 in a cell
// 172 -> 49 us (half lists 286 -> 122), 55,296 with 32 176 -> 167, 4,000 with 63 32.9 -> 28.6.
__device__ __forceinline__ void tile_stage_f64(const DevState& s, const Geometry& g, const TileMeta& m, int b,
                                               double* __restrict__ tx_, double* __restrict__ ty_,
                                               double* __restrict__ tz_, int* __restrict__ tsp,
                                               const int (&pre)[65]) {
    int bx, by, bz;
    block_coords(g, b, bx, by, bz);
    const int T = m.prefix[64], count = pre[64];
    const double cx = (2.0 * bx + 1.0) * g.w[0], cy = (2.0 * by + 1.0) * g.w[1], cz = (2.0 * bz + 1.0) * g.w[2];
    for (int i0 = threadIdx.x; i0 < count; i0 += STAGE64_AHEAD * (int)blockDim.x) {
        double x[STAGE64_AHEAD], y[STAGE64_AHEAD], z[STAGE64_AHEAD];
        int sp[STAGE64_AHEAD], at[STAGE64_AHEAD], coord[STAGE64_AHEAD];
#pragma unroll
        for (int k = 0; k < STAGE64_AHEAD; ++k) {
            const int i = i0 + k * (int)blockDim.x;
            at[k] = -1;
            if (i < count) {
                int slot = 0;
#pragma unroll
                for (int h = 32; h > 0; h >>= 1) slot += pre[slot + h] <= i ? h : 0;
                const int e = i - pre[slot], j = m.start[slot] + e;
                at[k] = m.prefix[slot] + e;
                coord[k] = m.coord[slot];
                x[k] = s.x[j], y[k] = s.y[j], z[k] = s.z[j];
                sp[k] = s.species[j];
            }
        }
#pragma unroll
        for (int k = 0; k < STAGE64_AHEAD; ++k) {
            if (at[k] < 0) continue;
            const int c = coord[k];
            const int rx = 2 * bx - 1 + (c & 3), ry = 2 * by - 1 + ((c >> 2) & 3), rz = 2 * bz - 1 + (c >> 4);
            if (rx < 0) x[k] -= g.L[0];
            else if (rx >= g.nc[0]) x[k] += g.L[0];
            if (ry < 0) y[k] -= g.L[1];
            else if (ry >= g.nc[1]) y[k] += g.L[1];
            if (rz < 0) z[k] -= g.L[2];
            else if (rz >= g.nc[2]) z[k] += g.L[2];
            tx_[at[k]] = x[k] - cx;
            ty_[at[k]] = y[k] - cy;
            tz_[at[k]] = z[k] - cz;
            tsp[at[k]] = sp[k];
        }
    }
    if (threadIdx.x == 0) {
        tx_[T] = ty_[T] = tz_[T] = 1.0e4;
        tsp[T] = 0;
    }
}

}  // namespace mdgb
