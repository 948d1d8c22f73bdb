// k_tbsma.cu - many-body forces of the tight-binding second-moment potential (Cleri and
// Rosato 1993), the potential of all of the paper's benchmarks (Sec. III), in two passes
// over the same cell tasks and full neighbour lists as the pair forces (Sec. II.A).
//
//   E = sum_i [ sum_j phi(r_ij) - sqrt(rho_i) ],  rho_i = sum_j psi(r_ij)
//   phi(r) = A exp(-p (r/r0 - 1)),  psi(r) = xi^2 exp(-2q (r/r0 - 1))
//   F_i = sum_j [ (2p/r0) phi - (q/r0) psi (1/sqrt(rho_i) + 1/sqrt(rho_j)) ] d / r
//
// Pass 1 (density) sums psi over each atom's list; pass 2 (force) needs 1/sqrt(rho_j) of every
// neighbour, so it starts its sums after pass 1 has finished, as its own launch, and stages those
// values into the .w of the tile entries (one species: the species bits are not needed there),
// so one 128-bit load brings a neighbour's coordinates and its 1/sqrt(rho).  Each atom is
// written by its own lanes only in both passes (full lists), so neither needs atomics.  In
// md_step pass 2 also updates velocities and positions, as the pair forces do.
//
// Two list entries are evaluated together in packed FP32x2 arithmetic.  What bounds the passes at
// 500,000 atoms is neither instruction issue (57 and 53 % busy) nor shared memory (64 and 47 %,
// half of it bank conflicts of the gathers) alone but their alternation with the staging of
// the tiles; fewer registers and more CTAs per SM do not help (68 us at 4 CTAs, 73 at 5 and 6).  A
// step's kernels took 65 + 104 us and 16.6 for the separate integration, and take 68 + 95; the
// second pass starts while the last CTAs of the first are running, for 1 us more.
//
// Mixed precision, as the pair kernels: block-frame FP32 coordinates, FP32 pair terms
// (the exponentials as 2^(k dr + l) on the hardware's base-2 exponential), densities and
// forces summed in Q31.32 fixed point (exact, order independent).  A pair whose FP32 r^2
// lies in the band around r_cut^2 is decided by the FP64 definition: its atom is
// finished after the loop by the whole warp, against the tile still in shared memory.
#include "full_task.cuh"
#include "launch.cuh"

#include <algorithm>

namespace mdgb {

namespace {

constexpr int TB_THREADS = 256;

__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// phi and psi at distance r = r2 * rinv (rinv = 1/r)
__device__ __forceinline__ void tb_terms(const TBTable& tb, float r2, float rinv, float& phi, float& psi) {
    const float dr = __fmaf_rn(r2, rinv, -tb.r0);
    phi = ex2_approx(__fmaf_rn(tb.kp, dr, tb.lp));
    psi = ex2_approx(__fmaf_rn(tb.kq, dr, tb.lq));
}

__device__ __forceinline__ float4 tb_disp(const float4& pi, const float4& pj, float& r2) {
    const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
    r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    return make_float4(dx, dy, dz, 0.f);
}

// The larger of big, |a| and |b|; a NaN stays.
__device__ __forceinline__ float max_abs_nan(float big, float a, float b) {
    asm("max.NaN.f32 %0, %0, %1, %2;" : "+f"(big) : "f"(fabsf(a)), "f"(fabsf(b)));
    return big;
}

// Two list entries of one atom at a time, in packed FP32x2 arithmetic: every operation rounds as its
// scalar counterpart, so that a term has the same bits in the exact finish.
struct TbPairs {
    f2_t dx, dy, dz;
    float r2a, r2b;
    f2_t rinv, dr;
    bool ina, inb;
};

__device__ __forceinline__ TbPairs tb_pairs(const TBTable& tb, const float4& pi, const float4& pa, const float4& pb,
                                            float& mdist) {
    TbPairs d;
    d.dx = f2_pack(__fsub_rn(pi.x, pa.x), __fsub_rn(pi.x, pb.x));
    d.dy = f2_pack(__fsub_rn(pi.y, pa.y), __fsub_rn(pi.y, pb.y));
    d.dz = f2_pack(__fsub_rn(pi.z, pa.z), __fsub_rn(pi.z, pb.z));
    const f2_t r2 = f2_fma(d.dz, d.dz, f2_fma(d.dy, d.dy, f2_mul(d.dx, d.dx)));
    f2_unpack(r2, d.r2a, d.r2b);
    d.rinv = f2_pack(rsqrt_approx(d.r2a), rsqrt_approx(d.r2b));
    d.dr = f2_fma(r2, d.rinv, f2_pack(-tb.r0, -tb.r0));
    d.ina = d.r2a < tb.rc2hi_f;
    d.inb = d.r2b < tb.rc2hi_f;
    float ca, cb;  // distance of r^2 from the cutoff's band
    f2_unpack(f2_sub(r2, f2_pack(tb.rc2_f, tb.rc2_f)), ca, cb);
    mdist = fminf(mdist, fminf(fabsf(ca), fabsf(cb)));
    return d;
}

// 2^(k dr + l), both entries
__device__ __forceinline__ f2_t tb_exp2(f2_t dr, float k, float l) {
    float a, b;
    f2_unpack(f2_fma(f2_pack(k, k), dr, f2_pack(l, l)), a, b);
    return f2_pack(ex2_approx(a), ex2_approx(b));
}

// cutoff test of a pair: FP32 outside the band, the FP64 definition inside it
__device__ __forceinline__ bool tb_inside_exact(const DevState& s, const Geometry& g, const TBTable& tb,
                                                const TileMeta& m, int gi, int u, float r2) {
    if (r2 < tb.rc2lo_f) return true;
    if (!(r2 < tb.rc2hi_f)) return false;
    return fp64_pair_test(s.x, s.y, s.z, g.L[0], g.L[1], g.L[2], gi, tile_global_index(m, u), tb.rc2_d);
}

// What an atom's lanes read of its list: its 16-byte chunks side by side, LPA 2: two words each, 4: one
// word each, 8: one word of every other chunk.  The first AHEAD chunks are requested by the
// constructor, before their number is known to the lane.
template <int LPA>
struct LaneList {
    static constexpr int STEP = LPA == 8 ? 2 : 1, WORDS = LPA == 2 ? 2 : 1, AHEAD = 4;
    const unsigned* words;
    size_t stride;
    int cq;
    unsigned e[AHEAD][WORDS];

    __device__ __forceinline__ unsigned load(int c, int h) const { return __ldcs(words + (size_t)c * stride + h); }

    __device__ __forceinline__ LaneList(const DevState& s, int gi, int lq) {
        words = reinterpret_cast<const unsigned*>(s.nl) + (size_t)gi * 4 + (LPA == 2 ? 2 * lq : (lq & 3));
        stride = (size_t)s.np * 4;
        cq = LPA == 8 ? lq >> 2 : 0;
#pragma unroll
        for (int k = 0; k < AHEAD; ++k)
#pragma unroll
            for (int h = 0; h < WORDS; ++h) e[k][h] = cq + k * STEP < s.nl_chunks ? load(cq + k * STEP, h) : 0u;
    }

    // body(u0, u1) for every two entries of the lane's share of nch chunks
    template <typename Body>
    __device__ __forceinline__ void walk(int nch, Body&& body) {
        for (int c0 = cq; c0 < nch; c0 += AHEAD * STEP) {
            unsigned cur[AHEAD][WORDS];
#pragma unroll
            for (int k = 0; k < AHEAD; ++k)
#pragma unroll
                for (int h = 0; h < WORDS; ++h) {
                    cur[k][h] = e[k][h];
                    const int c = c0 + (AHEAD + k) * STEP;
                    if (c < nch) e[k][h] = load(c, h);
                }
#pragma unroll
            for (int k = 0; k < AHEAD; ++k)
                if (c0 + k * STEP < nch) {
#pragma unroll
                    for (int h = 0; h < WORDS; ++h) body((int)(cur[k][h] & 0xffffu), (int)(cur[k][h] >> 16));
                }
        }
    }
};

template <>
struct LaneList<1> {
    const uint4* row;
    size_t stride;
    __device__ __forceinline__ LaneList(const DevState& s, int gi, int) {
        row = reinterpret_cast<const uint4*>(s.nl) + gi;
        stride = s.np;
    }
    template <typename Body>
    __device__ __forceinline__ void walk(int nch, Body&& body) {
        for_each_neighbour_pair(row, stride, nch, body);
    }
};

template <int LPA>
__device__ __forceinline__ void lanes_sum(FixAcc& a) {
#pragma unroll
    for (int o = LPA / 2; o > 0; o >>= 1) {
        a.hi += __shfl_xor_sync(0xffffffffu, a.hi, o);
        a.lo += __shfl_xor_sync(0xffffffffu, a.lo, o);
    }
}

// The lanes of the warp whose atom has a pair for the exact finish (bad on any of its lanes).
template <int LPA>
__device__ __forceinline__ bool lanes_any(unsigned bad, int lane) {
    constexpr unsigned GROUP = (1u << LPA) - 1u;
    return (bad >> (lane & ~(LPA - 1)) & GROUP) != 0u;
}

// The CTA's block and its share of it; false when it has nothing to do (a tile that does not fit is
// flagged).
template <int PER>
__device__ __forceinline__ bool tb_begin(const DevState& s, const Geometry& g, int tile_cap, int split, int& part,
                                         TileMeta& m) {
    part = blockIdx.x % split;
    tile_meta(g, s.cell_start, spatial_block(g, blockIdx.x / split), m);
    if (m.prefix[64] + 1 > tile_cap) {
        if (threadIdx.x == 0) atomicOr(s.err, ERR_TILE_OVERFLOW);
        return false;
    }
    return part * PER < m.prefix[8];
}

__device__ __forceinline__ void tb_store_density(const DevState& s, int gi, long long q, float rep, float* emb,
                                                 bool energy) {
    const float rho = __ll2float_rn(q) * 0x1p-32f;  // (one rounding: the sum is below 2^53)
    const float inv = rho > 0.f ? rsqrt_approx(rho) : 0.f;
    emb[gi] = inv;
    if (energy) s.pe_atom_f[gi] = rep - rho * inv;  // sum phi - sqrt(rho)
}

}  // namespace

// ---------------------------------------------------------------- pass 1: densities
// Exact finish of one atom by one warp: cutoff decisions by the definition, any list length.
template <bool EV>
__device__ __forceinline__ void tb_finish_density(const DevState& s, const Geometry& g, const TBTable& tb,
                                                  const TileMeta& m, const float4* __restrict__ tile, int ui,
                                                  float* __restrict__ emb) {
    const int lane = threadIdx.x & 31;
    const int gi = m.start[0] + ui;
    const float4 pi = tile[ui];
    const int T = m.prefix[64];
    const int nent = ((s.nl_cnt[gi] + 7) >> 3) * 8;
    long long q = 0;  // exact 64-bit sum
    float rep = 0.f;
    for (int e = lane; e < nent; e += 32) {
        const int u = s.nl[((size_t)(e >> 3) * s.np + gi) * 8 + (e & 7)];
        if (u >= T) continue;
        float r2;
        tb_disp(pi, tile[u], r2);
        const bool in = tb_inside_exact(s, g, tb, m, gi, u, r2);
        float phi, psi;
        tb_terms(tb, r2, rsqrt_approx(r2), phi, psi);
        q += fix_term(in ? psi * FS_SCALE : 0.f, 1.0f);
        if (EV) rep += in ? phi : 0.f;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        q += __shfl_xor_sync(0xffffffffu, q, o);
        if (EV) rep += __shfl_xor_sync(0xffffffffu, rep, o);
    }
    if (lane == 0) tb_store_density(s, gi, q, rep, emb, EV);
}

template <bool EV, int LPA>
__global__ void __launch_bounds__(TB_THREADS) k_tbsma_density(DevState s, Geometry g, TBTable tb, TileOffsets to,
                                                              int tile_cap, float* __restrict__ emb, int split) {
    static_assert(!EV || LPA == 1, "energy sums are FP32: one lane adds them in list order");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    float4* tile = reinterpret_cast<float4*>(smem);
    constexpr int PER = TB_THREADS / LPA;  // own atoms at a time
    int part;
    asm volatile("griddepcontrol.launch_dependents;");
    if (!tb_begin<PER>(s, g, tile_cap, split, part, m)) return;
    const unsigned tile_s = (unsigned)__cvta_generic_to_shared(tile);
    const int blk0 = m.start[0], nown = m.prefix[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lq = threadIdx.x % LPA;
    bool staged = false;
    for (int u0 = part * PER; u0 < nown; u0 += split * PER) {
        const int ui = u0 + (int)threadIdx.x / LPA;
        const bool active = ui < nown;
        const int uc = active ? ui : 0, gi = blk0 + uc;
        const int cnt = s.nl_cnt[gi];
        LaneList<LPA> list(s, gi, lq);
        if (!staged) {
            tile_stage_f32_cells(m, s.xr, to, tile);
            if (threadIdx.x == 0) tile[m.prefix[64]] = make_float4(1.0e4f, 1.0e4f, 1.0e4f, 0.f);
            __syncthreads();
            staged = true;
        }
        const float4 pi = tile[uc];
        const int nch = active ? (cnt + 7) >> 3 : 0;
        FixAcc acc{0u, 0u};
        float rep = 0.f, mdist = 1.0e30f;
        const f2_t magic2 = f2_pack(MAGIC, MAGIC), two21 = f2_pack(TWO21, TWO21);
        list.walk(nch, [&](int v0, int v1) {
            const TbPairs d = tb_pairs(tb, pi, lds_tile(tile_s, v0), lds_tile(tile_s, v1), mdist);
            float pa, pb;
            f2_unpack(f2_mul(tb_exp2(d.dr, tb.kq, tb.lq), f2_pack(FS_SCALE, FS_SCALE)), pa, pb);
            // psi <= xi^2 e^(2q) < 2048: inside the split
            fix_add2_one(acc, f2_pack(d.ina ? pa : 0.f, d.inb ? pb : 0.f), magic2, two21);
            if (EV) {
                float fa, fb;
                f2_unpack(tb_exp2(d.dr, tb.kp, tb.lp), fa, fb);
                rep += d.ina ? fa : 0.f;
                rep += d.inb ? fb : 0.f;
            }
        });
        lanes_sum<LPA>(acc);
        // (lists beyond the split's terms: the warp's 64-bit sums)
        unsigned left = __ballot_sync(0xffffffffu, active && (nch * 8 > FIX_SPLIT_MAX_TERMS || !(mdist > tb.band_f)));
        if (active && lq == 0 && !lanes_any<LPA>(left, lane))
            tb_store_density(s, gi, fix_final(acc, nch * 8), rep, emb, EV);
        while (left) {
            const int grp = (__ffs(left) - 1) / LPA;
            left &= ~(((1u << LPA) - 1u) << (grp * LPA));
            tb_finish_density<EV>(s, g, tb, m, tile, u0 + warp * (32 / LPA) + grp, emb);
        }
    }
}

// ---------------------------------------------------------------- pass 2: forces
// Exact finish of one atom by one warp.
template <bool EV, int MODE>
__device__ __forceinline__ void tb_finish_force(const DevState& s, const Geometry& g, const PairTable& pt,
                                                const TBTable& tb, const TileMeta& m, const float4* __restrict__ tile,
                                                int ui, float fs2_max, const StepOut& out, double dt, float lim2_f) {
    const int lane = threadIdx.x & 31;
    const int gi = m.start[0] + ui;
    const int64_t n = s.n;
    const float4 pi = tile[ui];
    const float inv_i = pi.w;
    const int T = m.prefix[64];
    const int nent = ((s.nl_cnt[gi] + 7) >> 3) * 8;
    long long qx = 0, qy = 0, qz = 0;  // exact 64-bit sums (any list length)
    int nwide = 0;
    float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
    for (int e = lane; e < nent; e += 32) {
        const int u = s.nl[((size_t)(e >> 3) * s.np + gi) * 8 + (e & 7)];
        if (u >= T) continue;
        float r2;
        const float4 pj = tile[u];
        const float4 d = tb_disp(pi, pj, r2);
        const bool in = tb_inside_exact(s, g, tb, m, gi, u, r2);
        const float rinv = rsqrt_approx(r2);
        float phi, psi;
        tb_terms(tb, r2, rinv, phi, psi);
        const float fr = __fmaf_rn(tb.c_rep, phi, -tb.c_band * psi * (inv_i + pj.w));
        const float fs2 = in ? fr * rinv * FS_SCALE : 0.f;
        qx += fix_term_any(fs2, d.x, fs2_max, s.err);
        qy += fix_term_any(fs2, d.y, fs2_max, s.err);
        qz += fix_term_any(fs2, d.z, fs2_max, s.err);
        nwide += fabsf(fs2) < fs2_max ? 0 : 1;
        if (EV) {
            const float gq = fs2 * (1.0f / FS_SCALE);
            w0 += d.x * (gq * d.x);
            w1 += d.y * (gq * d.y);
            w2 += d.z * (gq * d.z);
            w3 += d.x * (gq * d.y);
            w4 += d.x * (gq * d.z);
            w5 += d.y * (gq * d.z);
        }
    }
    nwide = __reduce_add_sync(0xffffffffu, (unsigned)nwide);
    if (lane == 0) fix_wide_count_ok(nwide, s.err);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        qx += __shfl_xor_sync(0xffffffffu, qx, o);
        qy += __shfl_xor_sync(0xffffffffu, qy, o);
        qz += __shfl_xor_sync(0xffffffffu, qz, o);
        if (EV) {
            w0 += __shfl_xor_sync(0xffffffffu, w0, o);
            w1 += __shfl_xor_sync(0xffffffffu, w1, o);
            w2 += __shfl_xor_sync(0xffffffffu, w2, o);
            w3 += __shfl_xor_sync(0xffffffffu, w3, o);
            w4 += __shfl_xor_sync(0xffffffffu, w4, o);
            w5 += __shfl_xor_sync(0xffffffffu, w5, o);
        }
    }
    if (lane == 0) {
        full_epilogue<true, MODE>(s, pt, gi, 0, qx, qy, qz, out, dt, lim2_f);
        if (EV) {
            s.vir_atom_f[gi] = 0.5f * w0;
            s.vir_atom_f[n + gi] = 0.5f * w1;
            s.vir_atom_f[2 * n + gi] = 0.5f * w2;
            s.vir_atom_f[3 * n + gi] = 0.5f * w3;
            s.vir_atom_f[4 * n + gi] = 0.5f * w4;
            s.vir_atom_f[5 * n + gi] = 0.5f * w5;
        }
    }
}

// The end of the densities' launch.  This pass may start before it (programmatic dependent launch, as
// soon as the last density CTA is running): up to here it reads what both passes read.
__device__ __forceinline__ void densities_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// MODE as in the pair kernels: forces; forces and the closing kick; forces, both kicks and the drift
// into the other coordinate buffer.
template <bool EV, int MODE, int LPA>
__global__ void __launch_bounds__(TB_THREADS) k_tbsma_force(DevState s, Geometry g, PairTable pt, TBTable tb,
                                                            TileOffsets to, int tile_cap,
                                                            const float* __restrict__ emb, float fs2_max, StepOut out,
                                                            double dt, float lim2_f, int split) {
    static_assert(!EV || (MODE == FM_FORCE && LPA == 1), "energy sums are FP32: one lane adds them in list order");
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    float4* tile = reinterpret_cast<float4*>(smem);  // .w: 1/sqrt(rho) of the atom
    constexpr int PER = TB_THREADS / LPA;            // own atoms at a time
    int part;
    if (!tb_begin<PER>(s, g, tile_cap, split, part, m)) {
        densities_wait();
        return;
    }
    const unsigned tile_s = (unsigned)__cvta_generic_to_shared(tile);
    const int blk0 = m.start[0], nown = m.prefix[8];
    const int64_t n = s.n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lq = threadIdx.x % LPA;
    bool staged = false;
    for (int u0 = part * PER; u0 < nown; u0 += split * PER) {
        const int ui = u0 + (int)threadIdx.x / LPA;
        const bool active = ui < nown;
        const int uc = active ? ui : 0, gi = blk0 + uc;
        const int cnt = s.nl_cnt[gi];
        LaneList<LPA> list(s, gi, lq);
        LaneState<MODE, LPA> st;
        if (LPA > 1) st.load(s, gi, lq);
        if (!staged) {
            densities_wait();
            tile_stage_f32_cells<true>(m, s.xr, to, tile, emb);
            if (threadIdx.x == 0) tile[m.prefix[64]] = make_float4(1.0e4f, 1.0e4f, 1.0e4f, 0.f);
            __syncthreads();
            staged = true;
        }
        const float4 pi = tile[uc];
        const float inv_i = pi.w;
        const int nch = active ? (cnt + 7) >> 3 : 0;
        FixAcc ax{0u, 0u}, ay{0u, 0u}, az{0u, 0u};
        float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
        float mdist = 1.0e30f, big = 0.f;
        const f2_t magic2 = f2_pack(MAGIC, MAGIC), two21 = f2_pack(TWO21, TWO21);
        // (|f| / r) * 2^11: the power of two in the coefficients
        const float c_rep = tb.c_rep * FS_SCALE, c_band = -tb.c_band * FS_SCALE;
        list.walk(nch, [&](int v0, int v1) {
            const float4 pa = lds_tile(tile_s, v0), pb = lds_tile(tile_s, v1);
            const TbPairs d = tb_pairs(tb, pi, pa, pb, mdist);
            const f2_t phi = tb_exp2(d.dr, tb.kp, tb.lp), psi = tb_exp2(d.dr, tb.kq, tb.lq);
            const f2_t inv_ij = f2_pack(__fadd_rn(inv_i, pa.w), __fadd_rn(inv_i, pb.w));
            const f2_t fr = f2_fma(f2_pack(c_rep, c_rep), phi, f2_mul(f2_mul(f2_pack(c_band, c_band), psi), inv_ij));
            float fa, fb;
            f2_unpack(f2_mul(fr, d.rinv), fa, fb);
            fa = d.ina ? fa : 0.f;
            fb = d.inb ? fb : 0.f;
            big = max_abs_nan(big, fa, fb);
            const f2_t fs2 = f2_pack(fa, fb);
            fix_add2(ax, fs2, d.dx, magic2, two21);
            fix_add2(ay, fs2, d.dy, magic2, two21);
            fix_add2(az, fs2, d.dz, magic2, two21);
            if (EV) {
                float x[2], y[2], z[2];
                f2_unpack(d.dx, x[0], x[1]);
                f2_unpack(d.dy, y[0], y[1]);
                f2_unpack(d.dz, z[0], z[1]);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const float gq = (k ? fb : fa) * (1.0f / FS_SCALE);
                    w0 += x[k] * (gq * x[k]);
                    w1 += y[k] * (gq * y[k]);
                    w2 += z[k] * (gq * z[k]);
                    w3 += x[k] * (gq * y[k]);
                    w4 += x[k] * (gq * z[k]);
                    w5 += y[k] * (gq * z[k]);
                }
            }
        });
        lanes_sum<LPA>(ax);
        lanes_sum<LPA>(ay);
        lanes_sum<LPA>(az);
        // (lists beyond the split's terms: the warp's 64-bit sums)
        unsigned left = __ballot_sync(0xffffffffu, active && (nch * 8 > FIX_SPLIT_MAX_TERMS || !(mdist > tb.band_f) ||
                                                              !(big < fs2_max)));
        const bool write = active && !lanes_any<LPA>(left, lane);
        const int nterms = nch * 8;
        const long long q[3] = {fix_final(ax, nterms), fix_final(ay, nterms), fix_final(az, nterms)};
        if (LPA > 1) {
            full_epilogue_lanes<true, MODE, LPA>(s, pt, gi, 0, q, st, lq, write, out, dt, lim2_f);
        } else if (write) {
            full_epilogue<true, MODE>(s, pt, gi, 0, q[0], q[1], q[2], out, dt, lim2_f);
            if (EV) {  // full lists see every pair twice: each atom keeps half of each pair virial
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
            left &= ~(((1u << LPA) - 1u) << (grp * LPA));
            tb_finish_force<EV, MODE>(s, g, pt, tb, m, tile, u0 + warp * (32 / LPA) + grp, fs2_max, out, dt, lim2_f);
        }
    }
}

// ---------------------------------------------------------------- launchers
// The limit on a system's tile (the kernels themselves keep only the tile).
size_t tbsma_smem_bytes(int tile_cap) {
    return (size_t)tile_cap * sizeof(float4) + (((size_t)tile_cap * sizeof(uint16_t) + 15) & ~(size_t)15);
}

namespace {

using TbDensity = void (*)(DevState, Geometry, TBTable, TileOffsets, int, float*, int);
using TbForce = void (*)(DevState, Geometry, PairTable, TBTable, TileOffsets, int, const float*, float, StepOut, double,
                         float, int);

TbDensity tb_density(bool ev, int lpa) {
    if (ev) return k_tbsma_density<true, 1>;
    switch (lpa) {
        case 1: return k_tbsma_density<false, 1>;
        case 2: return k_tbsma_density<false, 2>;
        case 4: return k_tbsma_density<false, 4>;
        default: return k_tbsma_density<false, 8>;
    }
}

template <int MODE>
TbForce tb_force_of(int lpa) {
    switch (lpa) {
        case 1: return k_tbsma_force<false, MODE, 1>;
        case 2: return k_tbsma_force<false, MODE, 2>;
        case 4: return k_tbsma_force<false, MODE, 4>;
        default: return k_tbsma_force<false, MODE, 8>;
    }
}

TbForce tb_force(bool ev, int mode, int lpa) {
    if (ev) return k_tbsma_force<true, FM_FORCE, 1>;
    return mode == FM_FORCE ? tb_force_of<FM_FORCE>(lpa)
                            : (mode == FM_KICK ? tb_force_of<FM_KICK>(lpa) : tb_force_of<FM_KKD>(lpa));
}

}  // namespace

void init_tbsma_kernels() {
    allow_max_smem(tb_density(true, 1));
    allow_max_smem(tb_force(true, FM_FORCE, 1));
    for (int lpa = 1; lpa <= 8; lpa *= 2) {
        allow_max_smem(tb_density(false, lpa));
        for (int mode = FM_FORCE; mode <= FM_KKD; ++mode) allow_max_smem(tb_force(false, mode, lpa));
    }
}

void launch_tbsma(const DevState& s, const LaunchGeometry& g, const PairTable& pt, const TBTable& tb, const TileOffsets& to,
                  int tile_cap, float* emb, int with_energy, int mode, StepOut out, double dt, double lim2,
                  cudaStream_t st) {
    if (s.n == 0) return;
    const size_t smem = (size_t)tile_cap * sizeof(float4);
    // |fs2 * d| < 2^22 (the exact range of the two-part split) holds when |fs2| < 2^22 / r_cut
    const float fs2_max = (float)(4194304.0 / std::sqrt(tb.rc2_d) * 0.999);
    // the FP32 displacement test is slightly stricter than skin/2 (as in k_integrate)
    const float lim2_f = (float)(lim2 * (1.0 - 1e-4));
    // As in the pair forces of small systems: below two blocks per SM, the fewest lanes per atom (two
    // at least) that give every SM a CTA.  Both passes: 6,912 atoms (27 blocks) 31.9 us with one
    // lane and a CTA per block, 21.4 with eight lanes; 55,296 atoms (216 blocks) 41.2 and 38.0 (two
    // lanes); at 500,000 atoms (2,744 blocks) two lanes take 172, one lane 163.
    const int sms = g.sms;
    const int64_t per_block = (s.n + g.nblock - 1) / g.nblock;
    int lpa = 1;
    int64_t split = 1;
    if (!with_energy && g.nblock < 2 * sms) {
        for (lpa = 2;; lpa *= 2) {
            split = std::max<int64_t>(1, (per_block * lpa + TB_THREADS - 1) / TB_THREADS);
            if (lpa == 8 || g.nblock * split >= sms) break;
        }
    }
    const unsigned grid = (unsigned)(g.nblock * split);
    tb_density(with_energy, lpa)<<<grid, TB_THREADS, smem, st>>>(s, g, tb, to, tile_cap, emb, (int)split);
    cudaLaunchAttribute early{};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(TB_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, tb_force(with_energy, mode, lpa), s, g, pt, tb, to, tile_cap, (const float*)emb, fs2_max, out,
                       dt, lim2_f, (int)split);
}

}  // namespace mdgb
