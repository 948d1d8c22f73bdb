// k_force.cu - Lennard-Jones forces by cell tasks (Sec. II.A, step 2).
//
// One CTA is the task of one 2x2x2-cell block (Sec. II.D.2 blocking): it
// stages the block's 4x4x4-cell tile in shared memory and evaluates the
// neighbour lists of the block's own atoms against it.
//
//  * Full lists: one thread per atom i, accumulating only F_i.  No thread
//    ever writes an atom it does not own, so the paper's requirement that no
//    particle is updated by two workers at once (Sec. II.A) holds with no
//    synchronisation at all.
//  * Half lists (Newton's third law, Sec. II.D.3): each pair once; the
//    reaction -f_ij goes to the tile copy of j in shared memory, and the tile
//    is added back to global memory at the end.  Blocks of one colour class
//    have disjoint tiles, so one launch per colour runs only non-overlapping
//    tasks - the barrier-separated waves of Sec. II.B, 8 of them.  No global
//    atomics are used; within a CTA the tile accumulators take shared-memory
//    integer adds.
//
// Mixed precision: pair arithmetic in FP32 on block-frame coordinates; every
// pair force component q = rint(f * 2^32) is added in Q31.32 fixed point,
// split exactly into a high part (multiples of 2^21) and a low part, each
// summed in a 32-bit integer.  Integer sums do not depend on order, so the
// result is bit-reproducible for any list order, thread mapping or list kind,
// and f_ji = -f_ij bit for bit makes the total force exactly zero.
//
// FP64: the same structure with FP64 tile coordinates and FP64 sums (k_force_fp64.cu).
#include "full_task.cuh"
#include "launch.cuh"

#include <type_traits>

namespace mdgb {

constexpr int F_THREADS = 256;
constexpr int FULL_THREADS = 256;  // CTA size of the full-list mixed kernel
// Register cap of the full-list mixed kernel: 48 keeps 5 CTAs (40 warps) resident per SM.
// The kernel is latency bound, and more resident warps beat longer per-thread schedules.
#define MDGB_FULL_MAX_REGS 48
// With several species the pair constants come from shared memory, and 48 registers spill; so do the
// seven sums of an energy and virial launch (1,048,576 atoms: 221 us at 48 registers, 182 at 56
// and 64, 190 at 80).
#define MDGB_FULL_MAX_REGS_WIDE 64
// per-pair LJ in FP32: returns fs2 = (|f|/r) * 2^11 (not masked) and whether the FP32
// r^2 is inside the cutoff
template <bool SINGLE>
__device__ __forceinline__ float lj_fs_unmasked(const PairTable& pt, int t, float r2, float& s6_out, bool& inside) {
    const float sig2 = SINGLE ? pt.sig2_f[0] : pt.sig2_f[t];
    const float c48 = SINGLE ? pt.c48_f[0] : pt.c48_f[t];
    const float c24 = SINGLE ? pt.c24_f[0] : pt.c24_f[t];
    const float rc2 = SINGLE ? pt.rc2_f[0] : pt.rc2_f[t];
    const float inv = rcp_approx(r2);
    const float s2 = sig2 * inv;
    const float s6 = s2 * s2 * s2;
    inside = r2 < rc2;
    s6_out = s6;
    return (c48 * s6 - c24) * s6 * inv;  // constants carry the 2^11 scale
}

// ---------------------------------------------------------------- mixed, full list
// One thread per atom, two neighbours per iteration in packed FP32x2 arithmetic; each
// neighbour is one 128-bit shared-memory load.
//
// MODE selects what follows each atom's force (fused velocity Verlet, the same
// operations as k_integrate's mixed path, so fused and separate steps agree bit for
// bit):
//   FM_FORCE  store the fixed-point force;
//   FM_KICK   store it and apply the closing half kick v += (dt/2m) F;
//   FM_KKD    closing and next opening kick in one, v += 2 (dt/2m) F, then the drift
//             x += dt v into out (the other position buffers: other CTAs may still be
//             staging this atom's current FP32 coordinates or testing a pair near r_cut
//             with its current FP64 position), the new FP32 coordinates beside it, and
//             the skin/2 displacement test.  The force itself is not stored.
//
// full_block is the task of block b for the CTA that calls it; k_force_mixed_full runs one
// block per CTA in spatial order, k_force_mixed_occ loops over the occupied blocks of a
// compact system.
template <bool SINGLE, bool EV, int MODE>
__device__ __forceinline__ void full_block(const DevState& s, const Geometry& g, const PairTable& pt,
                                           const TileOffsets& to, int tile_cap, float fs2_max, const StepOut& out,
                                           double dt, float lim2_f, int b) {
    static_assert(!EV || MODE == FM_FORCE, "energy/virial launches only evaluate forces");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    __shared__ SpeciesTable stab;
    __shared__ WarpWide wwide[FULL_THREADS / 32];
    float4* tile = reinterpret_cast<float4*>(smem);
    // own atoms left to finish_atom_warp: bit ui % 32 of word ui / 32.  Own atom ui runs on
    // thread ui % blockDim.x, so word w is written and read by warp w % (warps) alone
    unsigned* qmask = reinterpret_cast<unsigned*>(tile + tile_cap);
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (!SINGLE) load_species_table(pt, stab);
    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    if (T + 1 > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        return;
    }
    const int nown = m.prefix[8];
    if (nown == 0) return;
    tile_stage_f32_cells(m, s.xr, to, tile);
    stage_dummy_f32(tile, T);
    __syncthreads();
    const unsigned tile_s = (unsigned)__cvta_generic_to_shared(tile);
    const int blk0 = m.start[0];
    const int64_t n = s.n;
    const size_t np = s.np;
    const int nsp = pt.nsp;
    const f2_t magic2 = f2_pack(MAGIC, MAGIC);
    const f2_t two21 = f2_pack(TWO21, TWO21);
    for (int w = warp; w < (nown + 31) >> 5; w += nwarps)
        if ((threadIdx.x & 31) == 0) qmask[w] = 0u;
    __syncwarp();
    for (int ui = threadIdx.x; ui < nown; ui += blockDim.x) {
        const int gi = blk0 + ui;
        const float4 pi = tile[ui];
        const int si = __float_as_int(pi.w);
        const int nch = (s.nl_cnt[gi] + 7) >> 3;
        const uint4* lp = reinterpret_cast<const uint4*>(s.nl) + gi;
        if (MODE == FM_KKD) {
            // the velocity Verlet update's state into L2 while the pairs run (an L2 prefetch
            // holds no register: 0.3012 -> 0.2991 ms per fused step at 2,048,000 atoms)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.vx + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.vy + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.vz + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.x + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.y + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.z + gi));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(s.xr_ref + gi));
        }
        FixAcc ax{0u, 0u}, ay{0u, 0u}, az{0u, 0u};
        float pe = 0.f, w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
        // the 32-bit split sums are exact up to FIX_SPLIT_MAX_TERMS terms; a longer list
        // (only at densities several times a liquid's) goes to the exact finish
        bool bad = nch * 8 > FIX_SPLIT_MAX_TERMS;
        // one species: the band and large-force tests as two running minima, checked once
        float mdist = 3.0e38f, mr2 = 3.0e38f;
        for_each_neighbour_pair(lp, np, nch, [&](int u0, int u1) {
            full_pair<SINGLE, EV>(pt, stab, tile_s, pi, si, nsp, fs2_max, magic2, two21, u0, u1, ax, ay, az, pe,
                                  w0, w1, w2, w3, w4, w5, bad, mdist, mr2);
        });
        // a pair in the band (|r^2 - r_cut^2| up to its half width) or close enough for a
        // term beyond the split sends the atom to the exact finish; NaN distances give no
        // force on either path
        if (SINGLE) bad |= (mdist <= pt.band_half_f) | (mr2 < pt.r2_wide_f);
        if (bad) {  // finished after the loop by finish_atom_warp, epilogue included
            atomicOr(&qmask[ui >> 5], 1u << (ui & 31));
            continue;
        }
        const int nterms = nch * 8;
        const long long qx = fix_final(ax, nterms), qy = fix_final(ay, nterms), qz = fix_final(az, nterms);
        full_epilogue<SINGLE, MODE>(s, pt, gi, si, qx, qy, qz, out, dt, lim2_f);
        if (EV) {
            // full lists see every pair twice: each atom keeps half of each pair energy / virial
            s.pe_atom_f[gi] = 0.5f * pe;
            s.vir_atom_f[gi] = 0.5f * w0;
            s.vir_atom_f[n + gi] = 0.5f * w1;
            s.vir_atom_f[2 * n + gi] = 0.5f * w2;
            s.vir_atom_f[3 * n + gi] = 0.5f * w3;
            s.vir_atom_f[4 * n + gi] = 0.5f * w4;
            s.vir_atom_f[5 * n + gi] = 0.5f * w5;
        }
    }
    // the warp's queued atoms, as soon as its own loop is done (the tile stays unchanged
    // until the CTA ends)
    __syncwarp();
    for (int w = warp; w < (nown + 31) >> 5; w += nwarps) {
        unsigned bits = qmask[w];
        while (bits) {
            const int ui = (w << 5) + __ffs(bits) - 1;
            bits &= bits - 1u;
            finish_atom_warp<SINGLE, EV, MODE>(s, g, pt, tile, stab, m, ui, fs2_max, out, dt, lim2_f, wwide[warp]);
        }
    }
}

template <bool SINGLE, bool EV, int MODE>
__global__ void __maxnreg__(SINGLE && !EV ? MDGB_FULL_MAX_REGS : MDGB_FULL_MAX_REGS_WIDE) k_force_mixed_full(DevState s, Geometry g, PairTable pt,
                                                                TileOffsets to, int tile_cap, float fs2_max,
                                                                StepOut out, double dt,
                                                                float lim2_f) {
    full_block<SINGLE, EV, MODE>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, spatial_block(g, blockIdx.x));
}

// The same over the occupied blocks of a compact system: a grid of s.compact CTAs, each
// taking every gridDim-th entry of the list.  (A separate kernel: the loop in the
// one-block kernel cost the dense case 10 % through its register allocation.)
template <bool SINGLE, bool EV, int MODE>
__global__ void __maxnreg__(SINGLE && !EV ? MDGB_FULL_MAX_REGS : MDGB_FULL_MAX_REGS_WIDE) k_force_mixed_occ(DevState s, Geometry g, PairTable pt,
                                                                TileOffsets to, int tile_cap, float fs2_max,
                                                                StepOut out, double dt,
                                                                float lim2_f) {
    const int count = s.stats[4];
    for (int k = blockIdx.x; k < count; k += gridDim.x) {
        full_block<SINGLE, EV, MODE>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, s.blk_list[k]);
        __syncthreads();  // the next block reuses the shared memory
    }
}

// Programmatic dependent launch: let the next launch of the stream begin; wait until the launch
// before this one has ended and its writes are visible.
__device__ __forceinline__ void colour_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void colour_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---------------------------------------------------------------- mixed, half list, one colour
// Shared memory: tile coordinates, then the tile's fixed-point accumulators
// (hi and lo parts per component, 32-bit) and their term counts.  Pair energies
// and virials are booked in full on the listing atom (only totals are reported).
//
// The colours' launches overlap up to the point where they write: a launch may start once every
// CTA of the one before it runs (programmatic dependent launch), stages its tiles and evaluates
// its pairs beside it, and waits for its end before the first global write.  So the writes of
// the colours stay separated as by barriers, and a colour of few blocks does not leave SMs idle:
// with its 20 evaluations a pass of 20 steps takes 1.79 instead of 3.13 ms at 108,000 atoms,
// 5.28 instead of 6.80 at 500,000 and 18.3 instead of 19.6 at 2,048,000.
//
// LPA lanes per own atom (CTAs of 256 LPA threads): lane q takes its part of every 16-byte list
// chunk, and the lanes' exact integer sums are added by shuffles.  Shared memory allows two or
// three CTAs per SM whatever their size, so that more lanes are more warps in flight, and in
// a small system, whose colours have fewer blocks than there are SMs, a shorter CTA: 27.9 -> 16.4 us
// a launch with four lanes at 108,000 atoms (64 blocks a colour).
template <bool SINGLE, bool EV, int LPA>
__global__ void __launch_bounds__(F_THREADS * LPA, LPA == 1 ? 3 : 1) k_force_mixed_half(DevState s, Geometry g, PairTable pt,
                                                                      TileOffsets to, int tile_cap, float fs2_max,
                                                                      int block0) {
    static_assert(!EV || LPA == 1, "energy sums are FP32: one lane adds them in list order");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    // terms beyond the two-part split (atoms closer than about 0.75 sigma) do not go
    // through the 32-bit tile sums: they wait here as exact 64-bit values
    constexpr int WQ = 64;
    __shared__ long long wq[WQ][3];
    __shared__ uint16_t wq_u[WQ];  // (tile indices; with 32 bits a tile of 6,784 atoms would not fit an SM)
    __shared__ int nwq;
    // Reaction sums only for the tile entries a half list reaches (the own cells and their
    // forward neighbours come first in the tile, Sec. II.D.3): 6 x rcap, hx, lx, hy, ly, hz,
    // lz, with the split's offset taken off each term; then, where a block needs them,
    // each entry's term count in 16 bits, two to a word (fewer than the tile's atoms, < 2^15).
    const int rcap = half_recv_cap(tile_cap);
    float4* tile = reinterpret_cast<float4*>(smem);
    unsigned* acc = reinterpret_cast<unsigned*>(tile + tile_cap);
    unsigned* cnt2 = acc + 6 * rcap;
    __shared__ int max_nch;  // the longest own list, in chunks
    const int b = block0 + blockIdx.x;
    colour_begin();
    if (threadIdx.x == 0) {
        nwq = 0;
        max_nch = 0;
    }
    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    const int recv = m.prefix[TILE_RECV_CELLS];
    if (T + 1 > tile_cap || recv > rcap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        colour_wait();
        return;
    }
    // (the own lists' lengths are on their way while the tile is staged)
    const int nown0 = m.prefix[8];
    const int my_cnt = (int)threadIdx.x < nown0 ? s.nl_cnt[m.start[0] + threadIdx.x] : 0;
    tile_stage_f32_cells(m, s.xr, to, tile);
    stage_dummy_f32(tile, T);
    for (int u = threadIdx.x; u < recv; u += blockDim.x) {
#pragma unroll
        for (int c = 0; c < 6; ++c) acc[c * rcap + u] = 0u;
        if ((u & 1) == 0) cnt2[u >> 1] = 0u;
    }
    if ((int)threadIdx.x < nown0) atomicMax(&max_nch, (my_cnt + 7) >> 3);
    for (int ui = threadIdx.x + blockDim.x; ui < nown0; ui += blockDim.x)
        atomicMax(&max_nch, (s.nl_cnt[m.start[0] + ui] + 7) >> 3);
    __syncthreads();
    const unsigned magic_bits = __float_as_uint(MAGIC);
    const int blk0 = m.start[0];
    const int nown = m.prefix[8];
    const int64_t n = s.n;
    const int np = s.np;
    // Each term's high part is below 2^22 in magnitude, so a 32-bit sum stays exact up to
    // FIX_SPLIT_MAX_TERMS terms.  An entry takes at most its own list's terms (own atoms)
    // and one reaction per own atom, so the counts are only kept for blocks where that
    // bound exceeds the limit (small boxes with whole-box tiles, high densities)
    const bool count = nown + 8 * max_nch > FIX_SPLIT_MAX_TERMS;
    const int lq = threadIdx.x % LPA;
    const int rounds = (nown * LPA + (int)blockDim.x - 1) / (int)blockDim.x;  // the same in every thread
    for (int r = 0; r < rounds; ++r) {
        const int ua = (r * (int)blockDim.x + (int)threadIdx.x) / LPA;
        const bool active = ua < nown;
        if (LPA == 1 && !active) break;
        const int ui = active ? ua : 0;
        const int gi = blk0 + ui;
        const float4 pi = tile[ui];
        const int si = __float_as_int(pi.w);
        const int nch = active ? (s.nl_cnt[gi] + 7) >> 3 : 0;
        FixAcc ax{0u, 0u}, ay{0u, 0u}, az{0u, 0u};
        float pe = 0.f, w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
        auto pair = [&](const int u) {
            const float4 pj = tile[u];
            const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
            const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
            const int t = SINGLE ? 0 : si * pt.nsp + __float_as_int(pj.w);
            float s6;
            bool inside;
            const float fs = lj_fs_unmasked<SINGLE>(pt, t, r2, s6, inside);
            if (r2 < pt.rc2hi_f[t] && !(r2 < pt.rc2lo_f[t]))  // rare: decide the cutoff in FP64
                inside = fp64_pair_test(s.x, s.y, s.z, g.L[0], g.L[1], g.L[2], gi, tile_global_index(m, u),
                                        SINGLE ? pt.rc2_d[0] : pt.rc2_d[t]);
            const float fs2 = inside ? fs : 0.0f;
            FixAcc bx{0u, 0u}, by{0u, 0u}, bz{0u, 0u};
            if (fabsf(fs2) < fs2_max) {
                fix_add(ax, fs2, dx);
                fix_add(ay, fs2, dy);
                fix_add(az, fs2, dz);
                fix_sub(bx, fs2, dx);
                fix_sub(by, fs2, dy);
                fix_sub(bz, fs2, dz);
            } else {  // rare: both atoms' terms into the queue (its count bounds the 64-bit sums)
                const long long qx = fix_term_wide(fs2, dx, s.err), qy = fix_term_wide(fs2, dy, s.err),
                                qz = fix_term_wide(fs2, dz, s.err);
                // the split sums count this pair as a zero term (offset bits only)
                fix_add(ax, 0.0f, 0.0f);
                fix_add(ay, 0.0f, 0.0f);
                fix_add(az, 0.0f, 0.0f);
                fix_add(bx, 0.0f, 0.0f);
                fix_add(by, 0.0f, 0.0f);
                fix_add(bz, 0.0f, 0.0f);
                const int k = atomicAdd(&nwq, 2);
                if (k + 1 < WQ && k + 2 <= FIX_WIDE_MAX_TERMS) {
                    wq_u[k] = (uint16_t)ui;
                    wq[k][0] = qx;
                    wq[k][1] = qy;
                    wq[k][2] = qz;
                    wq_u[k + 1] = (uint16_t)u;
                    wq[k + 1][0] = -qx;
                    wq[k + 1][1] = -qy;
                    wq[k + 1][2] = -qz;
                } else {
                    atomicOr(s.err, ERR_NONFINITE);
                }
            }
            if (u < recv) {  // else the padding's dummy slot: a zero term
                atomicAdd(&acc[0 * rcap + u], bx.hi - magic_bits);
                atomicAdd(&acc[1 * rcap + u], bx.lo - magic_bits);
                atomicAdd(&acc[2 * rcap + u], by.hi - magic_bits);
                atomicAdd(&acc[3 * rcap + u], by.lo - magic_bits);
                atomicAdd(&acc[4 * rcap + u], bz.hi - magic_bits);
                atomicAdd(&acc[5 * rcap + u], bz.lo - magic_bits);
                if (count) atomicAdd(&cnt2[u >> 1], 1u << ((u & 1) << 4));
            }
            if (EV) {
                const float c4 = SINGLE ? pt.c4_f[0] : pt.c4_f[t];
                const float fs = fs2 * (1.0f / FS_SCALE);
                pe += inside ? c4 * s6 * (s6 - 1.0f) : 0.0f;
                w0 = fmaf(dx, fs * dx, w0);
                w1 = fmaf(dy, fs * dy, w1);
                w2 = fmaf(dz, fs * dz, w2);
                w3 = fmaf(dx, fs * dy, w3);
                w4 = fmaf(dx, fs * dz, w4);
                w5 = fmaf(dy, fs * dz, w5);
            }
        };
        // this lane's part of a chunk: eight, four or two entries in one load
        using Part = std::conditional_t<LPA == 1, uint4, std::conditional_t<LPA == 2, uint2, unsigned>>;
        const Part* parts = reinterpret_cast<const Part*>(reinterpret_cast<const uint4*>(s.nl) + gi) + lq;
        Part nxt{};
        if (nch > 0) nxt = __ldcs(parts);
        for (int c = 0; c < nch; ++c) {
            const Part cur = nxt;
            if (c + 1 < nch) nxt = __ldcs(parts + (size_t)(c + 1) * np * LPA);
            unsigned w[4 / LPA];
            if constexpr (LPA == 1) w[0] = cur.x, w[1] = cur.y, w[2] = cur.z, w[3] = cur.w;
            else if constexpr (LPA == 2) w[0] = cur.x, w[1] = cur.y;
            else w[0] = cur;
#pragma unroll
            for (int h = 0; h < 4 / LPA; ++h) {
                pair((int)(w[h] & 0xffffu));
                pair((int)(w[h] >> 16));
            }
        }
#pragma unroll
        for (int o = LPA / 2; o > 0; o >>= 1) {
            ax.hi += __shfl_xor_sync(0xffffffffu, ax.hi, o);
            ax.lo += __shfl_xor_sync(0xffffffffu, ax.lo, o);
            ay.hi += __shfl_xor_sync(0xffffffffu, ay.hi, o);
            ay.lo += __shfl_xor_sync(0xffffffffu, ay.lo, o);
            az.hi += __shfl_xor_sync(0xffffffffu, az.hi, o);
            az.lo += __shfl_xor_sync(0xffffffffu, az.lo, o);
        }
        if (!active || lq != 0) continue;
        // own atom's part goes through the same tile accumulator, its nch * 8 offsets removed
        const unsigned bias = (unsigned)(nch * 8) * magic_bits;
        atomicAdd(&acc[0 * rcap + ui], ax.hi - bias);
        atomicAdd(&acc[1 * rcap + ui], ax.lo - bias);
        atomicAdd(&acc[2 * rcap + ui], ay.hi - bias);
        atomicAdd(&acc[3 * rcap + ui], ay.lo - bias);
        atomicAdd(&acc[4 * rcap + ui], az.hi - bias);
        atomicAdd(&acc[5 * rcap + ui], az.lo - bias);
        if (count) atomicAdd(&cnt2[ui >> 1], (unsigned)(nch * 8) << ((ui & 1) << 4));
        if (EV) {
            s.pe_atom_f[gi] = pe;
            s.vir_atom_f[gi] = w0;
            s.vir_atom_f[n + gi] = w1;
            s.vir_atom_f[2 * n + gi] = w2;
            s.vir_atom_f[3 * n + gi] = w3;
            s.vir_atom_f[4 * n + gi] = w4;
            s.vir_atom_f[5 * n + gi] = w5;
        }
    }
    // With 1,024 threads, where this thread's first two atoms are (mostly all that it has), before the wait.
    const int bs = (int)blockDim.x, u0 = threadIdx.x, u1 = u0 + bs;
    int g0 = 0, g1 = 0;
    if constexpr (LPA > 1) {
        if (u0 < recv) g0 = tile_global_index(m, u0);
        if (u1 < recv) g1 = tile_global_index(m, u1);
    }
    __syncthreads();
    colour_wait();
    // add the tile back, an atom per thread: this CTA is the only one of its colour touching these atoms.
    // (A warp per cell instead: 82 us an evaluation instead of 57 at 70,304 atoms, 41 in a cell, whose second rows
    // are mostly empty, 383 instead of 263 at 202,612 atoms with 2, as long, 66, at 108,000 with 26.  The
    // search before the wait takes 2 to 5 us off an evaluation; with 256 threads it cost 16 of 209.)
    const auto add_back = [&](int u, int gj) {
        if (count) {
            const unsigned nt = (cnt2[u >> 1] >> ((u & 1) << 4)) & 0xffffu;
            if (nt == 0) return;
            // more than FIX_SPLIT_MAX_TERMS terms on one atom could wrap its 32-bit sums
            if (nt > FIX_SPLIT_MAX_TERMS) atomicOr(s.err, ERR_NONFINITE);
        }
        FixAcc fx{acc[0 * rcap + u], acc[1 * rcap + u]};
        FixAcc fy{acc[2 * rcap + u], acc[3 * rcap + u]};
        FixAcc fz{acc[4 * rcap + u], acc[5 * rcap + u]};
        s.fq[gj] += fix_final(fx, 0);
        s.fq[n + gj] += fix_final(fy, 0);
        s.fq[2 * n + gj] += fix_final(fz, 0);
    };
    if (LPA > 1 && u0 < recv) add_back(u0, g0);
    if (LPA > 1 && u1 < recv) add_back(u1, g1);
    for (int u = LPA > 1 ? u1 + bs : u0; u < recv; u += bs) add_back(u, tile_global_index(m, u));
    __syncthreads();
    if (threadIdx.x == 0) {  // the queued large terms, exact in 64 bits
        const int nq = nwq < WQ ? nwq : WQ;
        for (int k = 0; k < nq; ++k) {
            const int u = wq_u[k];
            const int slot = tile_slot_of(m, u);
            const int gj = m.start[slot] + (u - m.prefix[slot]);
            s.fq[gj] += wq[k][0];
            s.fq[n + gj] += wq[k][1];
            s.fq[2 * n + gj] += wq[k][2];
        }
    }
}

size_t force_smem_bytes(int mixed, int half, int with_energy, int tile_cap) {
    (void)with_energy;
    if (mixed) {
        size_t b = (size_t)tile_cap * sizeof(float4);
        if (half) {  // reaction sums and 16-bit term counts of the entries a half list reaches
            const size_t r = (size_t)half_recv_cap(tile_cap);
            b += r * 6 * sizeof(unsigned) + (((r + 1) / 2 * sizeof(unsigned) + 15) & ~(size_t)15);
        }
        else b += ((size_t)(tile_cap + 31) / 32 * sizeof(unsigned) + 15) & ~(size_t)15;  // own atoms to finish
        return b;
    }
    size_t b = (size_t)tile_cap * (3 * sizeof(double) + sizeof(int));
    if (half) b += (size_t)tile_cap * 3 * sizeof(double);
    return b;
}

// Raise every force kernel's dynamic shared-memory limit to what the SM allows
// (once per device, before any launch or stream capture).
template <bool SINGLE>
static void init_force_kernels_of(int half) {
    if (half) {
        allow_max_smem(k_force_mixed_half<SINGLE, false, 1>);
        allow_max_smem(k_force_mixed_half<SINGLE, false, 4>);
        allow_max_smem(k_force_mixed_half<SINGLE, true, 1>);
        return;
    }
    allow_max_smem(k_force_mixed_full<SINGLE, false, FM_FORCE>);
    allow_max_smem(k_force_mixed_full<SINGLE, true, FM_FORCE>);
    allow_max_smem(k_force_mixed_full<SINGLE, false, FM_KICK>);
    allow_max_smem(k_force_mixed_full<SINGLE, false, FM_KKD>);
    allow_max_smem(k_force_mixed_occ<SINGLE, false, FM_FORCE>);
    allow_max_smem(k_force_mixed_occ<SINGLE, true, FM_FORCE>);
    allow_max_smem(k_force_mixed_occ<SINGLE, false, FM_KICK>);
    allow_max_smem(k_force_mixed_occ<SINGLE, false, FM_KKD>);
    init_force_split_kernels(SINGLE);
}

// The kernels that a system of this kind launches (each costs its creation some microseconds).
void init_force_kernels(int mixed, int half, int single) {
    if (!mixed) init_force_fp64_kernels(half, single);
    else if (single) init_force_kernels_of<true>(half);
    else init_force_kernels_of<false>(half);
}

// |fs2 * d| < 2^22 (the exact range of the two-part split) is guaranteed when |fs2| < 2^22 / r_cut
float fs2_max_of(const PairTable& pt) {
    float rcmax2 = 0.f;
    for (int t = 0; t < pt.nsp * pt.nsp; ++t) rcmax2 = pt.rc2_f[t] > rcmax2 ? pt.rc2_f[t] : rcmax2;
    return 4194304.0f / sqrtf(rcmax2) * 0.999f;
}

// One full-list launch: a CTA per block, or with a compact system a grid of s.compact CTAs
// over the occupied blocks.
template <bool SINGLE, bool EV, int MODE>
static void launch_full(const DevState& s, const Geometry& g, const PairTable& pt, const TileOffsets& to,
                        int tile_cap, float fs2_max, StepOut out, double dt, float lim2_f, size_t smem,
                        cudaStream_t st) {
    if (s.compact)
        k_force_mixed_occ<SINGLE, EV, MODE><<<s.compact, FULL_THREADS, smem, st>>>(s, g, pt, to, tile_cap, fs2_max,
                                                                                 out, dt, lim2_f);
    else
        k_force_mixed_full<SINGLE, EV, MODE><<<g.nblock, FULL_THREADS, smem, st>>>(s, g, pt, to, tile_cap, fs2_max,
                                                                                 out, dt, lim2_f);
}

void launch_forces_mixed(const DevState& s, const LaunchGeometry& g, const PairTable& pt, const TileOffsets& to,
                         int tile_cap, int half, int with_energy, cudaStream_t st) {
    if (s.n == 0) return;
    const size_t smem = force_smem_bytes(1, half, with_energy, tile_cap);
    const float fs2_max = fs2_max_of(pt);
    const bool single = pt.nsp == 1;
    if (!half) {
        if (launch_forces_mixed_split(s, g, pt, to, tile_cap, fs2_max, with_energy != 0, FM_FORCE, StepOut{}, 0.0, 0.f,
                                      smem, st))
            return;
        if (single && !with_energy)
            launch_full<true, false, FM_FORCE>(s, g, pt, to, tile_cap, fs2_max, StepOut{}, 0.0, 0.f, smem, st);
        else if (single)
            launch_full<true, true, FM_FORCE>(s, g, pt, to, tile_cap, fs2_max, StepOut{}, 0.0, 0.f, smem, st);
        else if (!with_energy)
            launch_full<false, false, FM_FORCE>(s, g, pt, to, tile_cap, fs2_max, StepOut{}, 0.0, 0.f, smem, st);
        else
            launch_full<false, true, FM_FORCE>(s, g, pt, to, tile_cap, fs2_max, StepOut{}, 0.0, 0.f, smem, st);
        return;
    }
    cudaMemsetAsync(s.fq, 0, sizeof(long long) * 3 * (size_t)s.n, st);
    const int per = g.nblock / 8;
    // Four lanes per atom while a colour has fewer than two blocks per SM.  An evaluation with four lanes and
    // with one: 219,488 atoms (125 blocks) 109 and 126 us, 389,344 (216) 183 and 195, 500,000 (343) 245 and
    // 209; 296,352 (216 as well, 1,372 atoms each) 155 and 136.
    const int lpa = with_energy || per >= 2 * g.sms ? 1 : 4;
    using K = void (*)(DevState, Geometry, PairTable, TileOffsets, int, float, int);
    K k;
    if (with_energy) k = single ? (K)k_force_mixed_half<true, true, 1> : (K)k_force_mixed_half<false, true, 1>;
    else if (lpa == 1) k = single ? (K)k_force_mixed_half<true, false, 1> : (K)k_force_mixed_half<false, false, 1>;
    else k = single ? (K)k_force_mixed_half<true, false, 4> : (K)k_force_mixed_half<false, false, 4>;
    cudaLaunchAttribute overlap{};
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = per;
    cfg.blockDim = F_THREADS * lpa;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &overlap;
    for (int col = 0; col < 8; ++col) {
        cfg.numAttrs = col > 0 ? 1 : 0;  // the first follows the reset of the forces
        cudaLaunchKernelEx(&cfg, k, s, g, pt, to, tile_cap, fs2_max, col * per);
    }
}

// Full-list mixed forces fused with velocity Verlet (mode FM_KICK: closing half kick;
// FM_KKD: closing + opening kick and drift, the new positions into out).
void launch_forces_mixed_fused(const DevState& s, const LaunchGeometry& g, const PairTable& pt, const TileOffsets& to,
                               int tile_cap, int mode, StepOut out, double dt, double lim2, cudaStream_t st) {
    if (s.n == 0) return;
    const size_t smem = force_smem_bytes(1, 0, 0, tile_cap);
    const float fs2_max = fs2_max_of(pt);
    // the FP32 displacement test is slightly stricter than skin/2 (as in k_integrate)
    const float lim2_f = (float)(lim2 * (1.0 - 1e-4));
    const bool single = pt.nsp == 1;
    if (launch_forces_mixed_split(s, g, pt, to, tile_cap, fs2_max, false, mode == FUSE_KICK ? FM_KICK : FM_KKD, out, dt,
                                  lim2_f, smem, st))
        return;
    if (mode == FM_KICK) {
        if (single)
            launch_full<true, false, FM_KICK>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, smem, st);
        else
            launch_full<false, false, FM_KICK>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, smem, st);
    } else {
        if (single)
            launch_full<true, false, FM_KKD>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, smem, st);
        else
            launch_full<false, false, FM_KKD>(s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, smem, st);
    }
}

}  // namespace mdgb
