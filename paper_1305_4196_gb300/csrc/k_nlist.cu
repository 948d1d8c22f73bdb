// k_nlist.cu - neighbour-list construction by cell tasks (Sec. II.A).
//
// The paper builds the neighbour lists of all particles of one cell per task
// (Sec. II.A) and gives each task its own list storage so that no two tasks
// update the same structure (Sec. II.A, Sec. II.C).  Here one CTA is the task
// of one 2x2x2-cell block: it stages the block's 4x4x4-cell tile in shared
// memory and each of its 8 warps scans the 27 cells around one cell of the
// block (nl_scan.cuh).  Each list is written by one warp alone, so the lists
// need no synchronisation at all.
//
// The set is exactly the FP64 definition: pairs with minimum-image
// |x_i - x_j|^2 < r_list^2 evaluated as ((dx*dx)+dy*dy)+dz*dz.  The FP32
// tile test decides every candidate whose r^2 is further from r_list^2 than
// twice the bound on its FP32 error (tile_frame_cut_band, a relative 3e-6 for a
// liquid); candidates inside that band are re-tested with the FP64 positions in
// exactly the definition's operation order (minimum image d - L*rint(d/L)).
//
// Full lists hold every neighbour of every atom.  Half lists (Newton's third
// law, Sec. II.D.3) hold each pair once: a neighbour in the same cell only if
// it comes later in cell order, plus all neighbours of the 13 "forward" cells.
//
// Bound by instruction issue (68 % of cycles at 24 warps per SM; 80 registers, and
// 42 KB of scan buffers beside the tile).  At 1,048,576 atoms: 590 us and 567 M warp
// instructions with a lane per own atom that tested every atom of the 27 cells and
// appended its own hits, 391 us and 322 M with the scan of nl_scan.cuh, 384 and 309 M with cheaper tile
// offsets and the copy of the atoms' state (other forms of the scan:
// 439 us with hit masks turned into entries by a loop over their bits; 551 us with the self
// pair and the band sieved out of the rows by a lane each).
#include "launch.cuh"
#include "nl_scan.cuh"

#include <algorithm>

namespace mdgb {

// Atom i of the new order from the gather's copy to the state.
__device__ __forceinline__ void copy_atom(const DevState& s, const DevState& d, int i) {
    const double x = d.x[i], y = d.y[i], z = d.z[i], vx = d.vx[i], vy = d.vy[i], vz = d.vz[i];
    const int ix = d.ix[i], iy = d.iy[i], iz = d.iz[i], sp = d.species[i], orig = d.orig[i];
    s.x[i] = x, s.y[i] = y, s.z[i] = z;
    s.vx[i] = vx, s.vy[i] = vy, s.vz[i] = vz;
    s.ix[i] = ix, s.iy[i] = iy, s.iz[i] = iz;
    s.species[i] = sp, s.orig[i] = orig;
}

// The lists of the own atoms of block b (the CTA's task): warp w takes own cell w, or of each
// cell the share `part` of `split` (small systems, whose blocks are too few to fill the SMs).
// d: the state in the new order as the gather left it; a warp copies its atoms to s behind their
// lists, and the re-tests read d.
template <int HALF>
__device__ __forceinline__ void build_block(const DevState& s, const DevState& d, const Geometry& g,
                                            const TileOffsets& to, double rl2,
                                            float band_lo, float band_hi, int list_cap, int tile_cap, int b, int part,
                                            int split) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;

    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    // the tile capacity this block needs: its atoms and the dummy slot, and for half lists
    // also room for the mixed kernel's reaction sums over the cells a half list reaches
    const int need = HALF ? max(T + 1, tile_cap_for_recv(m.prefix[TILE_RECV_CELLS])) : T + 1;
    if (threadIdx.x == 0) atomicMax(&s.stats[1], need);
    if (need > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        if (part == 0)
            for (int u = threadIdx.x; u < m.prefix[8]; u += blockDim.x) copy_atom(s, d, m.start[0] + u);
        return;
    }
    if (m.prefix[8] == 0) return;  // empty block (vacuum): no lists to build
    const int stride = (tile_cap + 3) & ~3;
    const int nw = blockDim.x >> 5;
    float* const tx = reinterpret_cast<float*>(smem + nw * sizeof(NlWarp));
    float* const ty = tx + stride;
    float* const tz = ty + stride;
    nl_stage(m, to, tx, ty, tz, [&](int j) { return s.xr[j]; });
    __syncthreads();

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    NlWarp& w = reinterpret_cast<NlWarp*>(smem)[warp];
    int max_cnt = 0;
    unsigned long long sum_cnt = 0;
    for (int oc = warp; oc < 8; oc += nw) {
        const int own_coord = (1 + (oc & 1)) + 4 * (1 + ((oc >> 1) & 1)) + 16 * (1 + (oc >> 2));
        const int count = m.prefix[oc + 1] - m.prefix[oc];
        const int per = (count + split - 1) / split;
        const int hi_own = min(count, (part + 1) * per);
        for (int lo_own = part * per; lo_own < hi_own; lo_own += 32) {
            const int own_n = min(32, hi_own - lo_own);
            const int g0 = m.start[oc] + lo_own;
            const int cnt = nl_scan_cell<HALF>(
                w, m, tx, ty, tz, oc, own_coord, lo_own, own_n, band_hi, band_lo, reinterpret_cast<uint4*>(s.nl) + g0,
                (size_t)s.np, list_cap, [&](int own, int u) {
                    return fp64_pair_test(d.x, d.y, d.z, g.L[0], g.L[1], g.L[2], g0 + own, tile_global_index(m, u),
                                          rl2);
                });
            if (lane < own_n) {
                if (cnt > list_cap) atomicOr(s.err, ERR_LIST_OVERFLOW);
                s.nl_cnt[g0 + lane] = (uint16_t)(cnt < list_cap ? cnt : list_cap);
                max_cnt = cnt > max_cnt ? cnt : max_cnt;
                sum_cnt += (unsigned long long)cnt;
                copy_atom(s, d, g0 + lane);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        max_cnt = max(max_cnt, __shfl_xor_sync(0xffffffffu, max_cnt, o));
        sum_cnt += __shfl_xor_sync(0xffffffffu, sum_cnt, o);
    }
    if (lane == 0 && max_cnt > 0) {
        atomicMax(&s.stats[0], max_cnt);
        atomicAdd(reinterpret_cast<unsigned long long*>(&s.stats[2]), sum_cnt);
    }
}

// `split` CTAs per block, blocks in spatial order.
template <int HALF>
__global__ void __launch_bounds__(NL_WARPS * 32, 3) k_build_lists(DevState s, DevState d, Geometry g,
                                                                  TileOffsets to, double rl2, float band_lo,
                                                                  float band_hi, int list_cap, int tile_cap,
                                                                  int split) {
    build_block<HALF>(s, d, g, to, rl2, band_lo, band_hi, list_cap, tile_cap, spatial_block(g, blockIdx.x / split),
                      blockIdx.x % split, split);
}

// A compact system: a grid of s.compact CTAs over the occupied blocks.
template <int HALF>
__global__ void __launch_bounds__(NL_WARPS * 32, 3) k_build_lists_occ(DevState s, DevState d, Geometry g,
                                                                      TileOffsets to, double rl2, float band_lo,
                                                                      float band_hi, int list_cap, int tile_cap) {
    const int count = s.stats[4];
    for (int k = blockIdx.x; k < count; k += gridDim.x) {
        build_block<HALF>(s, d, g, to, rl2, band_lo, band_hi, list_cap, tile_cap, s.blk_list[k], 0, 1);
        __syncthreads();  // the next block reuses the shared memory
    }
}

// Shared memory of a CTA of `warps` warps.
static size_t nl_smem_bytes(int tile_cap, int warps) { return nl_tile_bytes(tile_cap) + warps * sizeof(NlWarp); }

// The size the callers hold against the limit of an SM's shared memory: 12 B per tile atom and
// about 35 KB (with a tile close to the limit a CTA runs four warps).
size_t build_lists_smem(int tile_cap) {
    return (size_t)((tile_cap + 227) & ~3) * 3 * sizeof(float) + 32768;
}

void launch_build_lists(const DevState& s, const DevState& d, const LaunchGeometry& g, const TileOffsets& to, double rl2, int list_cap,
                        int tile_cap, int half, cudaStream_t st) {
    if (s.n == 0) return;
    const int warps = nl_smem_bytes(tile_cap, NL_WARPS) <= 226 * 1024 ? NL_WARPS : NL_WARPS / 2;
    const size_t smem = nl_smem_bytes(tile_cap, warps);
    // candidates whose FP32 r^2 the error bound of the tile's coordinates leaves undecided
    const double band = tile_frame_cut_band(std::max({g.w[0], g.w[1], g.w[2]}), 0.0, std::sqrt(rl2));
    const float lo = (float)(rl2 * (1.0 - band)), hi = (float)(rl2 * (1.0 + band));
    const int threads = warps * 32;
    if (s.compact) {
        if (half) k_build_lists_occ<1><<<s.compact, threads, smem, st>>>(s, d, g, to, rl2, lo, hi, list_cap, tile_cap);
        else k_build_lists_occ<0><<<s.compact, threads, smem, st>>>(s, d, g, to, rl2, lo, hi, list_cap, tile_cap);
        return;
    }
    // CTAs per block, each a share of every cell's atoms: as many as run at once, down to shares of two
    // atoms (32,000 atoms, 64 blocks, two CTAs per SM: 95 us with one CTA per block, 39 with four, 55
    // with five, whose last 16 start when the others end; 2,048 atoms, 8 blocks: 43 with one, 16 with
    // sixteen).
    const int64_t per_sm = std::min<int64_t>(3, (int64_t)g.sm_smem / (int64_t)(smem + 1024));
    const int64_t per_cell = (s.n + g.ncell - 1) / g.ncell;
    const int split = (int)std::max<int64_t>(1, std::min<int64_t>({per_cell / 2, per_sm * g.sms / g.nblock, 16}));
    const unsigned grid = (unsigned)g.nblock * (unsigned)split;
    if (half) k_build_lists<1><<<grid, threads, smem, st>>>(s, d, g, to, rl2, lo, hi, list_cap, tile_cap, split);
    else k_build_lists<0><<<grid, threads, smem, st>>>(s, d, g, to, rl2, lo, hi, list_cap, tile_cap, split);
}

void init_list_kernels(int half) {
    if (half) {
        allow_max_smem(k_build_lists<1>);
        allow_max_smem(k_build_lists_occ<1>);
    } else {
        allow_max_smem(k_build_lists<0>);
        allow_max_smem(k_build_lists_occ<0>);
    }
}

// ---------------------------------------------------------------- export
// The list as unordered pairs of original ids (i < j).  A full list holds
// each pair twice and reports it from the side with the smaller id.
__global__ void k_pairs_out(DevState s, Geometry g, int half, unsigned long long* __restrict__ counter,
                            int32_t* __restrict__ pairs, long long cap) {
    __shared__ TileMeta m;
    const int b = blockIdx.x;
    tile_meta(g, s.cell_start, b, m);
    const int blk0 = m.start[0];
    const int nown = m.prefix[8];
    for (int ui = threadIdx.x; ui < nown; ui += blockDim.x) {
        const int gi = blk0 + ui;
        const int oi = s.orig[gi];
        const int cnt = s.nl_cnt[gi];
        const uint16_t* rows = s.nl;
        for (int k = 0; k < cnt; ++k) {
            const int u = rows[((size_t)(k >> 3) * s.np + gi) * 8 + (k & 7)];
            if (u >= m.prefix[64]) continue;  // an idle step of an atom-free schedule
            const int slot = tile_slot_of(m, u);
            const int gj = m.start[slot] + (u - m.prefix[slot]);
            const int oj = s.orig[gj];
            if (!half && oi > oj) continue;
            const unsigned long long at = atomicAdd(counter, 1ull);
            if ((long long)at < cap) {
                pairs[2 * at] = oi < oj ? oi : oj;
                pairs[2 * at + 1] = oi < oj ? oj : oi;
            }
        }
    }
}

void launch_pairs_out(const DevState& s, const Geometry& g, int half, unsigned long long* counter,
                      int32_t* pairs, long long cap, cudaStream_t st) {
    if (s.n == 0) return;
    k_pairs_out<<<g.nblock, 128, 0, st>>>(s, g, half, counter, pairs, cap);
}

}  // namespace mdgb
