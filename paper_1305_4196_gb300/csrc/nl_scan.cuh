// nl_scan.cuh - the candidate scan of the neighbour-list builders (k_nlist.cu, and the
// block systems of the ensemble kernel in k_batch.cu).
//
// A CTA stages its block's tile as three FP32 arrays; then one warp builds the lists of up to
// 32 own atoms of one cell against the cell itself and its neighbour cells, in stages that need
// no barrier beyond the warp:
//  1. Cull: the neighbour cells' atoms, a lane each, against the bounding box of the own
//     atoms.  Of the ~740 atoms of 27 cells of a liquid (3.2 sigma wide, list radius 2.8) about
//     375 can have a neighbour among the own atoms; their tile indices go to a buffer in scan
//     order.
//  2. Test: 64 candidates at a time, each lane holding two neighbouring ones in packed
//     registers, while the own atoms pass by as broadcast loads: seven packed operations and
//     two compares for 64 pairs.
//  3. Append: two ballots give every hit its place behind the own atom's entries (two bit counts
//     per lane, as a lane's two candidates follow each other), and the lanes write their
//     candidates' tile indices there, into a row of shared memory per own atom.  After the 64
//     candidates a lane per own atom writes the row's complete chunks of 8 entries to global
//     memory (16 bytes each; the lanes' chunks are consecutive).
// The scan order is that of the cells, and inside a cell that of its atoms.
#pragma once

#include "fixpt.cuh"
#include "tile.cuh"

namespace mdgb {

constexpr int NL_WARPS = 8;
constexpr int NL_BATCH = 64;    // candidates tested at a time (two per lane)
constexpr int NL_CAND = 288;    // candidate buffer
constexpr int NL_ROW = 56;      // entries of an own atom's row
constexpr float NL_FAR = 1.0e6f;  // coordinate of an empty candidate slot

// One warp's shared memory.  A batch can add 64 entries to the up to 7 left in a row: one that
// runs over its row (into the next, or the slack behind the last) is found by its length and
// done again in two halves.
struct __align__(16) NlWarp {
    float4 own_xy[32];          // own atoms' coordinates, each twice (packed operands)
    float4 own_z[32];           // z twice, then the shared address behind the atom's last entry
    uint16_t row[32 * NL_ROW + 16];
    uint16_t cand[NL_CAND];     // tile indices
};

__device__ __forceinline__ float warp_min(float v) {
    int i = __float_as_int(v);
    i ^= (i >> 31) & 0x7fffffff;  // integers in the order of the floats
    i = __reduce_min_sync(0xffffffffu, i);
    return __int_as_float(i ^ ((i >> 31) & 0x7fffffff));
}

__device__ __forceinline__ void lds_f2x2(unsigned addr, f2_t& a, f2_t& b) {
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

// This thread's lane, read once (a plain threadIdx.x is read again in every loop).
__device__ __forceinline__ int nl_lane() {
    int l;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(l));
    return l;
}

// A lane's two candidates of a batch.
struct NlPair {
    f2_t x, y, z;
    unsigned u0, u1;  // their tile indices
    int index;        // scan index of the first one (the own cell's atoms are 0, 1, ...)
};

// Append a warp's hits (ra, rb < hi, and for OWN the index rule) to an own atom's row; az: shared
// address of its own_z, tail: the address behind the row's last entry.  In assembly so that
// the comparisons, votes and stores share their predicates.
template <int HALF, bool OWN>
__device__ __forceinline__ void nl_append(unsigned az, unsigned tail, int lane, unsigned below, float ra, float rb,
                                          float hi, int self, const NlPair& c) {
#define NL_APPEND(RULE)                                                                                       \
    asm volatile(                                                                                             \
        "{\n\t.reg .pred p, q, l;\n\t.reg .b32 a, b;\n\t.reg .b16 u, v;\n\t"                                  \
        "setp.lt.f32 p, %0, %2;\n\tsetp.lt.f32 q, %1, %2;\n\t" RULE "setp.eq.s32 l, %3, 31;\n\t"              \
        "vote.sync.ballot.b32 a, p, 0xffffffff;\n\tvote.sync.ballot.b32 b, q, 0xffffffff;\n\t"                \
        "and.b32 a, a, %4;\n\tand.b32 b, b, %4;\n\tpopc.b32 a, a;\n\tpopc.b32 b, b;\n\tadd.u32 a, a, b;\n\t"  \
        "mad.lo.u32 a, a, 2, %5;\n\tcvt.u16.u32 u, %6;\n\tcvt.u16.u32 v, %7;\n\t"                             \
        "@p st.shared.u16 [a], u;\n\t@p add.u32 a, a, 2;\n\t"                                                 \
        "@q st.shared.u16 [a], v;\n\t@q add.u32 a, a, 2;\n\t"                                                 \
        "@l st.shared.u32 [%8+8], a;\n\t}" ::"f"(ra),                                                         \
        "f"(rb), "f"(hi), "r"(lane), "r"(below), "r"(tail), "r"(c.u0), "r"(c.u1), "r"(az), "r"(c.index),      \
        "r"(self), "r"(self - 1)                                                                              \
        : "memory")
    if (!OWN) NL_APPEND("");
    else if (HALF) NL_APPEND("setp.gt.and.s32 p, %9, %10, p;\n\tsetp.gt.and.s32 q, %9, %11, q;\n\t");
    else NL_APPEND("setp.ne.and.s32 p, %9, %10, p;\n\tsetp.ne.and.s32 q, %9, %11, q;\n\t");
#undef NL_APPEND
}

// One batch against every own atom.  OWN: the batch holds atoms of the own cell, of which an own
// atom takes no pair with itself (half lists: only with later ones); self0: own atom 0's index
// in its cell.  EXACT decides the pairs with r^2 in [lo, hi) by retest(own, u); without it they
// count as hits, and the smallest bit pattern of r^2 - lo is returned: below that of hi - lo if
// there was one, as negative numbers have the highest bit set.
template <int HALF, bool OWN, bool EXACT, typename Retest>
__device__ __forceinline__ unsigned nl_test(unsigned axy, int lane, int self0, int own_n, const NlPair& c, float hi,
                                            float lo, Retest&& retest) {
    const f2_t lo2 = f2_pack(lo, lo);
    const unsigned below = (1u << lane) - 1u;
    unsigned near_lo = 0xffffffffu;
    const unsigned end = axy + 16u * (unsigned)own_n;
    constexpr unsigned DZ = 32u * sizeof(float4);  // own_z lies behind own_xy
    int a = 0;
#pragma unroll(EXACT ? 1 : 2)
    for (; axy != end; axy += 16u, ++a) {
        f2_t ox, oy, oz, tail;
        lds_f2x2(axy, ox, oy);
        lds_f2x2(axy + DZ, oz, tail);
        const f2_t dx = f2_sub(ox, c.x), dy = f2_sub(oy, c.y), dz = f2_sub(oz, c.z);
        const f2_t r2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
        float ra, rb;
        f2_unpack(r2, ra, rb);
        if (EXACT) {  // a pair of the band that the definition excludes: out of reach
            if (ra < hi && !(ra < lo) && !retest(a, (int)c.u0)) ra = hi;
            if (rb < hi && !(rb < lo) && !retest(a, (int)c.u1)) rb = hi;
        } else {
            float ta, tb;
            f2_unpack(f2_sub(r2, lo2), ta, tb);
            near_lo = min(near_lo, min(__float_as_uint(ta), __float_as_uint(tb)));
        }
        nl_append<HALF, OWN>(axy + DZ, (unsigned)tail, lane, below, ra, rb, hi, self0 + a, c);
    }
    return near_lo;
}

// Shared memory of the tile's arrays (T <= tile_cap atoms and the padding of a 16-byte start).
__host__ __device__ inline size_t nl_tile_bytes(int tile_cap) {
    return (size_t)((tile_cap + 3) & ~3) * 3 * sizeof(float);
}

// Stage the tile's FP32 coordinates in the frame of the block, by tile index, one warp per cell
// (two cells at a time); load(j): the cell-relative coordinates of cell-ordered atom j.
template <typename Load>
__device__ __forceinline__ void nl_stage(const TileMeta& m, const TileOffsets& to, float* __restrict__ tx,
                                         float* __restrict__ ty, float* __restrict__ tz, Load&& load) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
#pragma unroll 2
    for (int slot = warp; slot < 64; slot += nw) {
        const int c = m.coord[slot];
        const float ox = pick4(to.off[0], c & 3), oy = pick4(to.off[1], (c >> 2) & 3), oz = pick4(to.off[2], c >> 4);
        const int u0 = m.prefix[slot], cnt = m.prefix[slot + 1] - u0, j0 = m.start[slot];
        for (int e = lane; e < cnt; e += 32) {
            const float4 p = load(j0 + e);
            tx[u0 + e] = p.x + ox;
            ty[u0 + e] = p.y + oy;
            tz[u0 + e] = p.z + oz;
        }
    }
}

// The lists of own atoms lo_own .. lo_own + own_n - 1 (own_n <= 32) of the cell in tile slot
// `own` (< 8), whose tile coordinate is own_coord.  out: chunk 0 of lane 0's list, the other lanes' behind
// it, chunk c at out[c * np]; cap: entries a list holds (a multiple of 8; more are counted only).
// Returns this lane's list length.
template <int HALF, typename Retest>
__device__ __forceinline__ int nl_scan_cell(NlWarp& w, const TileMeta& m, const float* __restrict__ tx,
                                            const float* __restrict__ ty, const float* __restrict__ tz, int own,
                                            int own_coord, int lo_own, int own_n, float hi, float lo, uint4* out,
                                            size_t np, int cap, Retest&& retest) {
    const int lane = nl_lane();
    constexpr int NK = HALF ? 14 : 27;
    // the own cell, then the others in the order of key = dx + 3 dy + 9 dz (half lists: key > 0);
    // lane k holds the k-th one's tile range
    int my_first = 0, my_end = 0;
    if (lane < NK) {
        const int k13 = lane == 0 ? 13 : (HALF ? lane : (lane <= 13 ? lane - 14 : lane - 13)) + 13;
        const int slot = m.slot[own_coord + (k13 % 3 - 1) + 4 * ((k13 / 3) % 3 - 1) + 16 * (k13 / 9 - 1)];
        my_first = m.prefix[slot];
        my_end = m.prefix[slot + 1];
    }
    const int own_count = __shfl_sync(0xffffffffu, my_end - my_first, 0);
    const int T = m.prefix[64];
    float xl, yl, zl, xh, yh, zh;  // the box of the own atoms
    {
        const int u = m.prefix[own] + lo_own + min(lane, own_n - 1);
        const float x = tx[u], y = ty[u], z = tz[u];
        w.own_xy[lane] = make_float4(x, x, y, y);
        w.own_z[lane] = make_float4(z, z, 0.f, 0.f);
        xl = warp_min(x), yl = warp_min(y), zl = warp_min(z);
        xh = -warp_min(-x), yh = -warp_min(-y), zh = -warp_min(-z);
    }
    uint4* const row = reinterpret_cast<uint4*>(w.row + lane * NL_ROW);
    const unsigned first = (unsigned)__cvta_generic_to_shared(row);
    unsigned* const tail = reinterpret_cast<unsigned*>(&w.own_z[lane].z);
    const unsigned axy = (unsigned)__cvta_generic_to_shared(w.own_xy);
    const unsigned below = (1u << lane) - 1u;
    out += lane;
    uint4 part = make_uint4(0u, 0u, 0u, 0u);  // the list's open chunk: cnt % 8 entries
    int cnt = 0;
    int nc = 0, base = 0;  // candidates in the buffer; scan index of its first one
    // (the loops below run on values the compiler knows to be the same in every lane: ballots,
    // reductions and loop counters)
    const int n_own = (int)__reduce_max_sync(0xffffffffu, (unsigned)own_n);
    const int n_cell = (int)__reduce_max_sync(0xffffffffu, (unsigned)own_count);
#pragma unroll 1
    for (int k = 0; k <= NK; ++k) {  // k = NK: no cell, what is left in the buffer
        int u = __shfl_sync(0xffffffffu, my_first, k);
        const int end = __shfl_sync(0xffffffffu, my_end, k);
        bool more;
        do {
            // ---- 1. cull up to 32 atoms of the cell
            const int ui = u + lane, ur = max(min(ui, end - 1), 0);
            const float x = tx[ur], y = ty[ur], z = tz[ur];
            // distance to the box of the own atoms: each rounded difference is at most that to
            // any own atom, so no pair with r^2 < hi is lost
            const float dx = fmaxf(fmaxf(xl - x, x - xh), 0.f), dy = fmaxf(fmaxf(yl - y, y - yh), 0.f),
                        dz = fmaxf(fmaxf(zl - z, z - zh), 0.f);
            const float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
            const bool keep = (ui < end) & ((d2 < hi) | (k == 0));
            const unsigned kept = __ballot_sync(0xffffffffu, keep);
            if (keep) w.cand[nc + __popc(kept & below)] = (uint16_t)ui;
            nc += __popc(kept);
            u += 32;
            more = __any_sync(0xffffffffu, u < end);
            if (nc <= NL_CAND - 32 && k < NK) continue;
            // ---- 2. and 3. whole batches, and at the end what is left
            __syncwarp();
            int s = 0, width = NL_BATCH;
            while (k == NK ? s < nc : s + NL_BATCH <= nc) {
                const int nb = min(nc - s, width);
                if (cnt & 7) row[0] = part;
                *tail = first + 2u * (unsigned)(cnt & 7);
                __syncwarp();
                NlPair c;
                {
                    const int i = 2 * lane;
                    const bool p = i < nb, q = i + 1 < nb;
                    c.u0 = p ? w.cand[s + i] : 0u;
                    c.u1 = q ? w.cand[s + i + 1] : 0u;
                    c.x = f2_pack(p ? tx[c.u0] : NL_FAR, q ? tx[c.u1] : NL_FAR);
                    c.y = f2_pack(p ? ty[c.u0] : NL_FAR, q ? ty[c.u1] : NL_FAR);
                    c.z = f2_pack(p ? tz[c.u0] : NL_FAR, q ? tz[c.u1] : NL_FAR);
                    c.index = base + s + i;
                }
                const unsigned near_lo = base + s < n_cell
                                             ? nl_test<HALF, true, false>(axy, lane, lo_own, n_own, c, hi, lo, retest)
                                             : nl_test<HALF, false, false>(axy, lane, lo_own, n_own, c, hi, lo, retest);
                __syncwarp();
                int open = (int)(*tail - first) >> 1;
                if (__any_sync(0xffffffffu, open > NL_ROW)) {  // a row ran over: again, half as many
                    width = NL_BATCH / 2;
                    continue;
                }
                if (__any_sync(0xffffffffu, near_lo < __float_as_uint(hi - lo))) {  // rare: the definition decides in [lo, hi)
                    *tail = first + 2u * (unsigned)(cnt & 7);
                    __syncwarp();
                    nl_test<HALF, true, true>(axy, lane, lo_own, n_own, c, hi, lo, retest);
                    __syncwarp();
                    open = (int)(*tail - first) >> 1;
                }
                // complete chunks to global memory, the open one to the lane's registers
                const int c0 = cnt >> 3, nch = open >> 3;
                const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)nch);
                uint4* to = out + (size_t)c0 * np;
                for (int j = 0; j < most; ++j) {
                    if (j < nch && 8 * (c0 + j) < cap) *to = row[j];
                    to += np;
                }
                part = row[nch];
                cnt = 8 * c0 + open;
                s += nb;
                __syncwarp();
            }
            // what is left (less than a batch) to the front of the buffer
            const int left = nc - s;
            const uint16_t v0 = lane < left ? w.cand[s + lane] : (uint16_t)0;
            const uint16_t v1 = lane + 32 < left ? w.cand[s + lane + 32] : (uint16_t)0;
            __syncwarp();
            if (lane < left) w.cand[lane] = v0;
            if (lane + 32 < left) w.cand[lane + 32] = v1;
            base += s;
            nc = left;
            __syncwarp();
        } while (more);
    }
    if ((cnt & 7) && lane < own_n && cnt < cap) {  // the last chunk, padded with the tile's dummy slot
        row[0] = part;
        for (int e = cnt & 7; e < 8; ++e) w.row[lane * NL_ROW + e] = (uint16_t)T;
        out[(size_t)(cnt >> 3) * np] = row[0];
    }
    __syncwarp();  // the next own atoms reuse the buffers
    return cnt;
}

}  // namespace mdgb
