// k_force_fp64.cu - Lennard-Jones forces in FP64 throughout, by cell tasks (Sec. II.A).
//
// The same task structure as the mixed-precision kernels (k_force.cu): one CTA per
// 2x2x2-cell block with the block's 4x4x4-cell tile staged in shared memory, here as FP64
// coordinates relative to the block.
//  * Full lists: one thread per atom i, accumulating only F_i (no particle is written by
//    two workers, Sec. II.A).
//  * Half lists (Newton's third law, Sec. II.D.3): the reaction -f_ij goes to the tile copy
//    of j in shared memory; one launch per colour class of blocks, whose tiles are disjoint
//    (the barrier-separated waves of Sec. II.B).
//
// On GB300 the FP64 pipe bounds these kernels: an SM takes 16 cycles for a warp's FP64
// operation, while it issues 64 others (the list and coordinates stream through with DRAM
// nearly idle).  So the full-list kernel spends other instructions to save FP64 ones:
//  * the list entries are tested in FP32 first, on the upper halves of the tile's coordinates,
//    and only those that may lie inside the cutoff go to an atom's queue in shared memory; the
//    lanes of a warp then take them in step, an atom's lanes side by side (a 76-entry list
//    holds 55 inside, where a masked loop runs all 80 padded entries);
//  * 17 FP64 operations per pair: three differences, three for r^2, one reciprocal by a cubic
//    step from an FP32 seed (three), five for f / r = inv^4 (a inv^3 - b), three sums; the
//    exact cutoff test compares bit patterns.
// Every result is that of FP64 arithmetic throughout.  At 360,703 atoms a force evaluation took
// 1.38 ms and one with energy and virial 2.11 ms with 22 operations for each of the 80 padded
// entries, and takes 0.76 and 1.23 ms; the FP64 pipe is 88 % busy.
#include "fp64_math.cuh"
#include "launch.cuh"
#include "tile.cuh"

#include <algorithm>

namespace mdgb {

constexpr int F_THREADS = 256;

// ---------------------------------------------------------------- full list
constexpr int FQ = 16;  // queue slots per lane; the lanes of an atom share theirs

__host__ __device__ constexpr size_t fp64_queue_bytes(int threads) { return (size_t)threads * FQ * sizeof(uint16_t); }

template <bool EV>
struct Fp64Sums {
    double f[3] = {0, 0, 0};
    double pe = 0, w[6] = {0, 0, 0, 0, 0, 0};
};

// One pair: r^2 and the cutoff decision in FP64, and the force of an inside pair.
template <bool SINGLE, bool EV>
__device__ __forceinline__ void fp64_pair(const PairTable& pt, const double* __restrict__ tx,
                                          const double* __restrict__ ty, const double* __restrict__ tz,
                                          const int* __restrict__ tsp, int u, double xi, double yi, double zi, int si,
                                          Fp64Sums<EV>& a) {
    const double dx = xi - tx[u], dy = yi - ty[u], dz = zi - tz[u];
    const double r2 = dx * dx + dy * dy + dz * dz;
    const int t = SINGLE ? 0 : si * pt.nsp + tsp[u];
    const double inv = rcp_cubic(r2);
    const double inv2 = inv * inv, inv3 = inv2 * inv;
    double fr = fma(SINGLE ? pt.lj_a_d[0] : pt.lj_a_d[t], inv3, -(SINGLE ? pt.lj_b_d[0] : pt.lj_b_d[t])) * (inv2 * inv2);
    // r^2 >= 0 compares like its bits
    const bool in = __double_as_longlong(r2) < __double_as_longlong(SINGLE ? pt.rc2_d[0] : pt.rc2_d[t]);
    if (!in) fr = 0.0;
    if (EV) {
        const double px = fr * dx, py = fr * dy, pz = fr * dz;
        a.f[0] += px;
        a.f[1] += py;
        a.f[2] += pz;
        // 4 eps (s6^2 - s6) = inv^3 (a inv^3 / 12 - b / 6)
        const double e = fma(SINGLE ? pt.lj_a12_d[0] : pt.lj_a12_d[t], inv3, -(SINGLE ? pt.lj_b6_d[0] : pt.lj_b6_d[t]));
        a.pe = fma(in ? inv3 : 0.0, e, a.pe);
        a.w[0] = fma(dx, px, a.w[0]);
        a.w[1] = fma(dy, py, a.w[1]);
        a.w[2] = fma(dz, pz, a.w[2]);
        a.w[3] = fma(dx, py, a.w[3]);
        a.w[4] = fma(dx, pz, a.w[4]);
        a.w[5] = fma(dy, pz, a.w[5]);
    } else {
        a.f[0] = fma(fr, dx, a.f[0]);
        a.f[1] = fma(fr, dy, a.f[1]);
        a.f[2] = fma(fr, dz, a.f[2]);
    }
}

// LPA lanes per atom, which share its list and the queue of pairs to evaluate; `split` CTAs share
// one block, each staging the tile and taking every split-th group of own atoms.  rc2_test: r_cut^2
// plus the bound on the FP32 test's error, largest over the species pairs.  QUEUE = false evaluates
// every entry (a tile that leaves no room for the queues).
template <bool SINGLE, bool EV, int LPA, bool QUEUE>
__global__ void __launch_bounds__(F_THREADS) k_force_fp64_full(DevState s, Geometry g, PairTable pt, int tile_cap,
                                                               int split, float rc2_test) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    __shared__ int needed[65];
    double* tx = reinterpret_cast<double*>(smem);
    double* ty = tx + tile_cap;
    double* tz = ty + tile_cap;
    int* tsp = reinterpret_cast<int*>(tz + tile_cap);
    uint16_t* const queues = reinterpret_cast<uint16_t*>(tsp + tile_cap);
    const int b = spatial_block(g, blockIdx.x / split), part = blockIdx.x % split;
    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    if (T + 1 > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        return;
    }
    const int nown = m.prefix[8];
    const int per = blockDim.x / LPA;  // own atoms at a time
    if (part * per >= nown) return;
    if (split > 1) tile_needed_prefix(m, tile_needed(m, part, split, per), needed);
    tile_stage_f64(s, g, m, b, tx, ty, tz, tsp, split > 1 ? needed : m.prefix);
    __syncthreads();
    const int blk0 = m.start[0];
    const int64_t n = s.n;
    const size_t np = s.np;
    const int lq = threadIdx.x % LPA;
    for (int u0 = part * per; u0 < nown; u0 += split * per) {
        const int ui = u0 + (int)threadIdx.x / LPA;
        const bool active = ui < nown;
        const int gi = blk0 + (active ? ui : 0);
        const double xi = tx[active ? ui : 0], yi = ty[active ? ui : 0], zi = tz[active ? ui : 0];
        const int si = SINGLE ? 0 : tsp[active ? ui : 0];
        const int nch = active ? (s.nl_cnt[gi] + 7) >> 3 : 0;
        const uint4* lp = reinterpret_cast<const uint4*>(s.nl) + gi;
        Fp64Sums<EV> a;
        if (QUEUE) {
            // The lanes of an atom share its queue, so that they evaluate the same number of pairs: lane q
            // tests the list's words (two entries) q, q + LPA, ..., and takes every LPA-th pair.
            constexpr int CAP = FQ * LPA;
            constexpr unsigned GROUP = (1u << LPA) - 1u;
            const int l0 = (int)(threadIdx.x & 31) & ~(LPA - 1);
            const unsigned below = (1u << lq) - 1u;
            uint16_t* const mine = queues + ((int)threadIdx.x - lq) * FQ;
            const unsigned* const words = reinterpret_cast<const unsigned*>(s.nl) + (size_t)gi * 4;
            const auto word = [&](int w) { return __ldcs(words + (size_t)(w >> 2) * np * 4 + (w & 3)); };
            const int nw = nch * 4;
            const float xf = upper_f32(xi), yf = upper_f32(yi), zf = upper_f32(zi);
            int head = 0, tail = 0;
            const auto take = [&]() {
                if (head + lq < tail)
                    fp64_pair<SINGLE, EV>(pt, tx, ty, tz, tsp, mine[(head + lq) & (CAP - 1)], xi, yi, zi, si, a);
                head = min(head + LPA, tail);
            };
            unsigned nxt = lq < nw ? word(lq) : 0u;
            for (int w0 = 0; __any_sync(0xffffffffu, w0 < nw); w0 += LPA) {
                const unsigned cur = nxt;
                const int w = w0 + lq;
                if (w + LPA < nw) nxt = word(w + LPA);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int u = (int)((cur >> (16 * h)) & 0xffffu);
                    bool near = false;
                    if (w < nw) {
                        const float dx = xf - upper_f32(tx[u]), dy = yf - upper_f32(ty[u]), dz = zf - upper_f32(tz[u]);
                        near = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) < rc2_test;
                    }
                    const unsigned group = __ballot_sync(0xffffffffu, near) >> l0 & GROUP;
                    if (near) mine[(tail + __popc(group & below)) & (CAP - 1)] = (uint16_t)u;
                    tail += __popc(group);
                }
                __syncwarp();
                // in step while every atom has pairs for all its lanes, or some atom too many for the next words
                while (__any_sync(0xffffffffu, tail - head > CAP - 2 * LPA) ||
                       __all_sync(0xffffffffu, tail - head >= LPA))
                    take();
                __syncwarp();  // (before the next entries overwrite those just taken)
            }
            while (__any_sync(0xffffffffu, tail > head)) take();
            __syncwarp();
        } else {
            for (int c = lq; c < nch; c += LPA) {
                const uint4 cur = __ldcs(lp + (size_t)c * np);
                const unsigned wd[4] = {cur.x, cur.y, cur.z, cur.w};
#pragma unroll 1
                for (int e = 0; e < 8; ++e)
                    fp64_pair<SINGLE, EV>(pt, tx, ty, tz, tsp, (int)((wd[e >> 1] >> ((e & 1) * 16)) & 0xffffu), xi, yi,
                                          zi, si, a);
            }
        }
#pragma unroll
        for (int o = LPA / 2; o > 0; o >>= 1) {
#pragma unroll
            for (int d = 0; d < 3; ++d) a.f[d] += __shfl_xor_sync(0xffffffffu, a.f[d], o);
            if (EV) {
                a.pe += __shfl_xor_sync(0xffffffffu, a.pe, o);
#pragma unroll
                for (int d = 0; d < 6; ++d) a.w[d] += __shfl_xor_sync(0xffffffffu, a.w[d], o);
            }
        }
        if (!active) continue;
        if (!(isfinite(a.f[0]) && isfinite(a.f[1]) && isfinite(a.f[2]))) atomicOr(s.err, ERR_NONFINITE);
        if (lq) continue;
        s.f[gi] = a.f[0];
        s.f[n + gi] = a.f[1];
        s.f[2 * n + gi] = a.f[2];
        if (EV) {
            s.pe_atom_d[gi] = 0.5 * a.pe;
#pragma unroll
            for (int d = 0; d < 6; ++d) s.vir_atom_d[d * n + gi] = 0.5 * a.w[d];
        }
    }
}

// FP64 half list, one colour: reactions through FP64 shared-memory accumulators.
template <bool EV>
__global__ void __launch_bounds__(F_THREADS) k_force_fp64_half(DevState s, Geometry g, PairTable pt, int tile_cap,
                                                               int block0) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    double* tx = reinterpret_cast<double*>(smem);
    double* ty = tx + tile_cap;
    double* tz = ty + tile_cap;
    double* acc = tz + tile_cap;  // 3 x tile_cap
    int* tsp = reinterpret_cast<int*>(acc + 3 * tile_cap);
    const int b = block0 + blockIdx.x;
    tile_meta(g, s.cell_start, b, m);
    const int T = m.prefix[64];
    if (T + 1 > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        return;
    }
    tile_stage_f64(s, g, m, b, tx, ty, tz, tsp, m.prefix);
    for (int u = threadIdx.x; u <= T; u += blockDim.x) {
        acc[u] = 0;
        acc[tile_cap + u] = 0;
        acc[2 * tile_cap + u] = 0;
    }
    __syncthreads();
    const int blk0 = m.start[0];
    const int nown = m.prefix[8];
    const int64_t n = s.n;
    const int np = s.np;
    for (int ui = threadIdx.x; ui < nown; ui += blockDim.x) {
        const int gi = blk0 + ui;
        const double xi = tx[ui], yi = ty[ui], zi = tz[ui];
        const int si = tsp[ui];
        const int nch = (s.nl_cnt[gi] + 7) >> 3;
        double fx = 0, fy = 0, fz = 0, pe = 0, w0 = 0, w1 = 0, w2 = 0, w3 = 0, w4 = 0, w5 = 0;
        MDGB_FOR_EACH_NEIGHBOUR(reinterpret_cast<const uint4*>(s.nl) + gi, np, nch, {
            const double dx = xi - tx[u], dy = yi - ty[u], dz = zi - tz[u];
            const double r2 = dx * dx + dy * dy + dz * dz;
            const int t = si * pt.nsp + tsp[u];
            if (r2 < pt.rc2_d[t]) {
                const double inv = rcp_nr(r2);
                const double sr2 = pt.sig2_d[t] * inv;
                const double s6 = sr2 * sr2 * sr2;
                const double e = pt.eps_d[t];
                const double fr = 24.0 * e * (2.0 * s6 * s6 - s6) * inv;
                fx += fr * dx;
                fy += fr * dy;
                fz += fr * dz;
                atomicAdd(&acc[u], -fr * dx);
                atomicAdd(&acc[tile_cap + u], -fr * dy);
                atomicAdd(&acc[2 * tile_cap + u], -fr * dz);
                if (EV) {
                    pe += 4.0 * e * (s6 * s6 - s6);
                    w0 += dx * (fr * dx);
                    w1 += dy * (fr * dy);
                    w2 += dz * (fr * dz);
                    w3 += dx * (fr * dy);
                    w4 += dx * (fr * dz);
                    w5 += dy * (fr * dz);
                }
            }
        })
        // a non-finite pair force leaves its mark on the i-side sum (a pair at r = 0 gives inf * 0)
        if (!(isfinite(fx) && isfinite(fy) && isfinite(fz))) atomicOr(s.err, ERR_NONFINITE);
        atomicAdd(&acc[ui], fx);
        atomicAdd(&acc[tile_cap + ui], fy);
        atomicAdd(&acc[2 * tile_cap + ui], fz);
        if (EV) {
            s.pe_atom_d[gi] = pe;
            s.vir_atom_d[gi] = w0;
            s.vir_atom_d[n + gi] = w1;
            s.vir_atom_d[2 * n + gi] = w2;
            s.vir_atom_d[3 * n + gi] = w3;
            s.vir_atom_d[4 * n + gi] = w4;
            s.vir_atom_d[5 * n + gi] = w5;
        }
    }
    __syncthreads();
    for (int u = threadIdx.x; u < T; u += blockDim.x) {
        const int slot = tile_slot_of(m, u);
        const int gj = m.start[slot] + (u - m.prefix[slot]);
        s.f[gj] += acc[u];
        s.f[n + gj] += acc[tile_cap + u];
        s.f[2 * n + gj] += acc[2 * tile_cap + u];
    }
}

// ---------------------------------------------------------------- launchers
using Fp64Full = void (*)(DevState, Geometry, PairTable, int, int, float);

template <bool SINGLE, bool EV, bool QUEUE>
static Fp64Full full_of(int lpa) {
    switch (lpa) {
        case 2: return k_force_fp64_full<SINGLE, EV, 2, QUEUE>;
        case 4: return k_force_fp64_full<SINGLE, EV, 4, QUEUE>;
        default: return k_force_fp64_full<SINGLE, EV, 8, QUEUE>;
    }
}

static Fp64Full full_kernel(bool single, bool ev, bool queue, int lpa) {
    if (single) {
        if (ev) return queue ? full_of<true, true, true>(lpa) : full_of<true, true, false>(lpa);
        return queue ? full_of<true, false, true>(lpa) : full_of<true, false, false>(lpa);
    }
    if (ev) return queue ? full_of<false, true, true>(lpa) : full_of<false, true, false>(lpa);
    return queue ? full_of<false, false, true>(lpa) : full_of<false, false, false>(lpa);
}

static void launch_full(const DevState& s, const Geometry& g, const PairTable& pt, int tile_cap, int split, int lpa,
                        int with_energy, float rc2_test, size_t smem, cudaStream_t st) {
    // (the FP32 test needs r_cut^2 well inside FP32's range)
    const bool queue = smem + fp64_queue_bytes(F_THREADS) <= 226 * 1024 && rc2_test > 1e-24f && rc2_test < 1e30f;
    if (queue) smem += fp64_queue_bytes(F_THREADS);
    const unsigned grid = (unsigned)g.nblock * (unsigned)split;
    full_kernel(pt.nsp == 1, with_energy != 0, queue, lpa)<<<grid, F_THREADS, smem, st>>>(s, g, pt, tile_cap, split,
                                                                                        rc2_test);
}

void launch_forces_fp64(const DevState& s, const LaunchGeometry& g, const PairTable& pt, int tile_cap, int half,
                        int with_energy, cudaStream_t st) {
    if (s.n == 0) return;
    const size_t smem = force_smem_bytes(0, half, with_energy, tile_cap);
    if (!half) {
        // CTAs per block: one where blocks suffice (two per SM), else the fewest that leave no SM with more
        // than 1.2 times its share of the atoms (64 blocks over 152 SMs: 2 each).  Lanes per atom:
        // eight while a CTA then takes its atoms in one pass, else four below one block per SM
        // (23,328 atoms: 73 us, 89 with two); from there on two, and CTAs for one pass of
        // them.  Against the same split with an own queue and whole 16-byte chunks per lane (both with a
        // warp per tile cell in the staging, which cost 1 to 9 us more than it does now): 4,000 atoms
        // (8 blocks) 29 us instead of 46, 10,976 (64) 47 / 75, 32,000 (64) 106 / 171, 55,296 (216)
        // 173 / 212, 360,703 (2,016) 776 / 799.
        const int sms = g.sms;
        const int64_t per_block = (s.n + g.nblock - 1) / g.nblock;
        int64_t split = 1;
        int lpa = 2;
        if (g.nblock < 2 * sms) {
            const auto share = [&](int64_t k) { return (g.nblock * k + sms - 1) / sms * (double)per_block / k; };
            const double even = (double)s.n / sms;
            while (split < 32 && share(split) > 1.2 * even) ++split;
            split = std::max<int64_t>(split, sms / g.nblock);  // (up to a CTA per SM: blocks differ in size)
            if (per_block * 8 <= F_THREADS * split) lpa = 8;
            else if (g.nblock < sms) lpa = 4;
            else split = std::max(split, (per_block * 9 / 8 * lpa + F_THREADS - 1) / F_THREADS);  // (blocks differ)
        }
        // the FP32 test's error: coordinates up to two cells from the block centre, cut to 20 bits
        const double wmax = std::max({g.w[0], g.w[1], g.w[2]});
        double rc2 = 0.0;
        for (int t = 0; t < pt.nsp * pt.nsp; ++t) rc2 = std::max(rc2, pt.rc2_d[t]);
        const double e_d = 3.0 * wmax * 0x1p-19;
        const double rc = std::sqrt(rc2);
        const float rc2_test = (float)((rc2 + 2.0 * std::sqrt(3.0) * rc * e_d + 3.0 * e_d * e_d) * (1.0 + 1e-6));
        launch_full(s, g, pt, tile_cap, (int)split, lpa, with_energy, rc2_test, smem, st);
        return;
    }
    cudaMemsetAsync(s.f, 0, sizeof(double) * 3 * (size_t)s.n, st);
    const int per = g.nblock / 8;
    for (int col = 0; col < 8; ++col) {
        if (with_energy) {
            k_force_fp64_half<true><<<per, F_THREADS, smem, st>>>(s, g, pt, tile_cap, col * per);
        } else {
            k_force_fp64_half<false><<<per, F_THREADS, smem, st>>>(s, g, pt, tile_cap, col * per);
        }
    }
}

void init_force_fp64_kernels(int half, int single) {
    if (half) {
        allow_max_smem(k_force_fp64_half<false>);
        allow_max_smem(k_force_fp64_half<true>);
        return;
    }
    for (int k = 0; k < 4; ++k)
        for (int lpa = 2; lpa <= 8; lpa *= 2) allow_max_smem(full_kernel(single, k & 1, k & 2, lpa));
}

}  // namespace mdgb
