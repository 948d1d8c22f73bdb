// k_force_split.cu - the full-list mixed force task (Sec. II.A, step 2) for systems with too few
// blocks to fill the SMs with one CTA each.
//
// Several CTAs share a block: each stages the block's tile and takes every split-th group of its
// own atoms, LPA lanes per atom.  The lanes of an atom take the entries of each 16-byte list
// chunk side by side (LPA 2: four each, 4: two each, 8: two each of every other chunk), and
// their exact integer sums are added by shuffles, so the forces are bit for bit those of one
// thread per atom (k_force.cu), which stays the faster form where blocks suffice: a lane reads
// 4 or 8 bytes of a chunk instead of 16, and every CTA stages the whole tile.
//
// Bound by latency: a CTA alone on its SM waits for the cells' starts, the tile, the list and the
// update's state in turn.  So the first list words and the state are on their way while the tile
// is staged, and the update's components are spread over the atom's lanes (FP64 instructions
// are issued per warp).  Fused step, one CTA per block against this form: 28.4 -> 19.2 us at
// 32,000 atoms (64 blocks), 21.5 -> 14.8 us at 16,384; forces alone 15.3 -> 7.0 us at 2,048.
#include "full_task.cuh"
#include "launch.cuh"

#include <algorithm>

namespace mdgb {

constexpr int SPLIT_THREADS = 256;

template <bool SINGLE, bool EV, int MODE, int LPA>
__global__ void __launch_bounds__(SPLIT_THREADS) k_force_mixed_split(DevState s, Geometry g, PairTable pt,
                                                                     TileOffsets to, int tile_cap, float fs2_max,
                                                                     StepOut out, double dt, float lim2_f, int split) {
    static_assert(!EV || (MODE == FM_FORCE && LPA == 1), "energy sums are FP32: one lane adds them in list order");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    __shared__ SpeciesTable stab;
    __shared__ WarpWide wwide[SPLIT_THREADS / 32];
    float4* tile = reinterpret_cast<float4*>(smem);
    const int b = spatial_block(g, blockIdx.x / split), part = blockIdx.x % split;
    if (!SINGLE) load_species_table(pt, stab);
    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    if (T + 1 > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        return;
    }
    const int nown = m.prefix[8];
    constexpr int PER = SPLIT_THREADS / LPA;  // own atoms at a time
    if (part * PER >= nown) return;
    const int64_t n = s.n;
    const size_t np = s.np;
    const int nsp = pt.nsp;
    const f2_t magic2 = f2_pack(MAGIC, MAGIC);
    const f2_t two21 = f2_pack(TWO21, TWO21);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lq = threadIdx.x % LPA;
    const unsigned tile_s = (unsigned)__cvta_generic_to_shared(tile);
    const int blk0 = m.start[0];
    const unsigned pad = (unsigned)T | ((unsigned)T << 16);
    // A lane's list words: `at` of chunk 0, one 16-byte chunk every np * 4 words; lanes 0..3 take
    // one word each of every STEP-th chunk (LPA >= 4), lanes 0, 1 two words each (LPA 2)
    constexpr int STEP = LPA == 8 ? 2 : 1;
    constexpr int WORDS = LPA == 2 ? 2 : 1;
    constexpr int AHEAD = LPA == 1 ? 1 : 4;  // chunks on their way together
    auto list_words = [&](int gi) {
        return reinterpret_cast<const unsigned*>(s.nl) + (size_t)gi * 4 + (LPA == 2 ? 2 * lq : (lq & 3));
    };
    auto load_word = [&](const unsigned* at, int c, int k) {
        return __ldcs(at + (size_t)c * np * 4 + k);
    };
    bool staged = false;
    for (int u0 = part * PER; u0 < nown; u0 += split * PER) {
        const int ui = u0 + (int)threadIdx.x / LPA;
        const bool active = ui < nown;
        const int uc = active ? ui : 0, gi = blk0 + uc;
        // the list's first words before its length is known, and the state of the update: on their
        // way while the tile is staged
        const int cnt = s.nl_cnt[gi];
        const unsigned* const words = list_words(gi);
        const int cq = LPA == 8 ? lq >> 2 : 0;
        unsigned e[AHEAD][WORDS];
        if (LPA > 1) {
#pragma unroll
            for (int k = 0; k < AHEAD; ++k)
#pragma unroll
                for (int h = 0; h < WORDS; ++h) e[k][h] = cq + k * STEP < s.nl_chunks ? load_word(words, cq + k * STEP, h) : pad;
        }
        LaneState<MODE, LPA> st;
        st.load(s, gi, lq);
        if (!staged) {
            tile_stage_f32_cells(m, s.xr, to, tile);
            stage_dummy_f32(tile, T);
            __syncthreads();
            staged = true;
        }
        const float4 pi = tile[uc];
        const int si = __float_as_int(pi.w);
        const int nch = active ? (cnt + 7) >> 3 : 0;
        FixAcc ax{0u, 0u}, ay{0u, 0u}, az{0u, 0u};
        float pe = 0.f, w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
        bool bad = nch * 8 > FIX_SPLIT_MAX_TERMS;
        float mdist = 3.0e38f, mr2 = 3.0e38f;
        auto pair = [&](unsigned w) {
            full_pair<SINGLE, EV>(pt, stab, tile_s, pi, si, nsp, fs2_max, magic2, two21, (int)(w & 0xffffu),
                                  (int)(w >> 16), ax, ay, az, pe, w0, w1, w2, w3, w4, w5, bad, mdist, mr2);
        };
        if (LPA == 1) {
            for_each_neighbour_pair(reinterpret_cast<const uint4*>(s.nl) + gi, np, nch,
                                    [&](int v0, int v1) { pair((unsigned)v0 | ((unsigned)v1 << 16)); });
        } else {
            for (int c0 = cq; c0 < nch; c0 += AHEAD * STEP) {
                unsigned cur[AHEAD][WORDS];
#pragma unroll
                for (int k = 0; k < AHEAD; ++k)
#pragma unroll
                    for (int h = 0; h < WORDS; ++h) {
                        cur[k][h] = c0 + k * STEP < nch ? e[k][h] : pad;
                        const int c = c0 + (AHEAD + k) * STEP;
                        if (c < nch) e[k][h] = load_word(words, c, h);
                    }
#pragma unroll
                for (int k = 0; k < AHEAD; ++k)
                    if (c0 + k * STEP < nch) {
#pragma unroll
                        for (int h = 0; h < WORDS; ++h) pair(cur[k][h]);
                    }
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
        if (SINGLE) bad |= (mdist <= pt.band_half_f) | (mr2 < pt.r2_wide_f);
        // an atom whose lanes found a pair for the exact finish: once per atom, by the whole warp
        unsigned left = __ballot_sync(0xffffffffu, bad && active);
        constexpr unsigned GROUP = LPA == 32 ? 0xffffffffu : (1u << LPA) - 1u;
        const bool mine_bad = (left >> (lane & ~(LPA - 1)) & GROUP) != 0u;
        const int nterms = nch * 8;
        const long long q[3] = {fix_final(ax, nterms), fix_final(ay, nterms), fix_final(az, nterms)};
        const bool write = active && !mine_bad;
        if (LPA > 1) full_epilogue_lanes<SINGLE, MODE, LPA>(s, pt, gi, si, q, st, lq, write, out, dt, lim2_f);
        if (LPA == 1 && write) {
            full_epilogue<SINGLE, MODE>(s, pt, gi, si, q[0], q[1], q[2], out, dt, lim2_f);
            if (EV) {  // full lists see every pair twice: each atom keeps half of each pair energy / virial
                s.pe_atom_f[gi] = 0.5f * pe;
                s.vir_atom_f[gi] = 0.5f * w0;
                s.vir_atom_f[n + gi] = 0.5f * w1;
                s.vir_atom_f[2 * n + gi] = 0.5f * w2;
                s.vir_atom_f[3 * n + gi] = 0.5f * w3;
                s.vir_atom_f[4 * n + gi] = 0.5f * w4;
                s.vir_atom_f[5 * n + gi] = 0.5f * w5;
            }
        }
        while (left) {
            const int grp = (__ffs(left) - 1) / LPA;
            left &= ~(GROUP << (grp * LPA));
            finish_atom_warp<SINGLE, EV, MODE>(s, g, pt, tile, stab, m, u0 + warp * (32 / LPA) + grp, fs2_max, out, dt,
                                               lim2_f, wwide[warp]);
        }
    }
}

namespace {

using SplitKernel = void (*)(DevState, Geometry, PairTable, TileOffsets, int, float, StepOut, double, float, int);

template <bool SINGLE, int MODE>
SplitKernel split_of(int lpa) {
    switch (lpa) {
        case 2: return k_force_mixed_split<SINGLE, false, MODE, 2>;
        case 4: return k_force_mixed_split<SINGLE, false, MODE, 4>;
        default: return k_force_mixed_split<SINGLE, false, MODE, 8>;
    }
}

SplitKernel split_kernel(bool single, bool ev, int mode, int lpa) {
    if (ev) return single ? k_force_mixed_split<true, true, FM_FORCE, 1> : k_force_mixed_split<false, true, FM_FORCE, 1>;
    if (single) {
        if (mode == FM_FORCE) return split_of<true, FM_FORCE>(lpa);
        return mode == FM_KICK ? split_of<true, FM_KICK>(lpa) : split_of<true, FM_KKD>(lpa);
    }
    if (mode == FM_FORCE) return split_of<false, FM_FORCE>(lpa);
    return mode == FM_KICK ? split_of<false, FM_KICK>(lpa) : split_of<false, FM_KKD>(lpa);
}

}  // namespace

void init_force_split_kernels(int single) {
    allow_max_smem(split_kernel(single, true, FM_FORCE, 1));
    for (int mode = FM_FORCE; mode <= FM_KKD; ++mode)
        for (int lpa = 2; lpa <= 8; lpa *= 2) allow_max_smem(split_kernel(single, false, mode, lpa));
}

bool launch_forces_mixed_split(const DevState& s, const LaunchGeometry& g, const PairTable& pt, const TileOffsets& to,
                               int tile_cap, float fs2_max, bool with_energy, int mode, StepOut out, double dt,
                               float lim2_f, size_t smem, cudaStream_t st) {
    // Below two blocks per SM (70,304 atoms, 216 blocks: 26.8 us here, 28.3 with a CTA per block;
    // 108,000 atoms, 512 blocks: 30.6 against 27.0).  The fewest lanes per atom that give every SM
    // a CTA: at 32,000 atoms two lanes (256 CTAs) take 19.2 us, four (512 CTAs) 22.6.
    const int sms = g.sms;
    if (s.compact || g.nblock >= 2 * sms) return false;
    const int64_t per_block = (s.n + g.nblock - 1) / g.nblock;
    int lpa = with_energy ? 1 : 2;
    int64_t split = 1;
    for (;; lpa *= 2) {
        split = std::max<int64_t>(1, (per_block * lpa + SPLIT_THREADS - 1) / SPLIT_THREADS);
        if (with_energy || lpa == 8 || g.nblock * split >= sms) break;
    }
    split_kernel(pt.nsp == 1, with_energy, mode, lpa)<<<(unsigned)(g.nblock * split), SPLIT_THREADS, smem, st>>>(
        s, g, pt, to, tile_cap, fs2_max, out, dt, lim2_f, (int)split);
    return true;
}

}  // namespace mdgb
