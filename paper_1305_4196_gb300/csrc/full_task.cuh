// full_task.cuh - device code shared by the full-list mixed force kernels: one thread per atom
// (k_force.cu) and, for small systems, several lanes per atom (k_force_split.cu).  Both apply
// exactly the same operations to a pair and after an atom's force, and add its terms as
// integers, so their results agree bit for bit.
#pragma once

#include "fixpt.cuh"
#include "tile.cuh"

namespace mdgb {

enum { FM_FORCE = 0, FM_KICK = 1, FM_KKD = 2 };  // what the full-list mixed kernel does after the force

__device__ __forceinline__ void stage_dummy_f32(float4* tile, int T) {
    if (threadIdx.x == 0) tile[T] = make_float4(1.0e4f, 1.0e4f, 1.0e4f, __int_as_float(0));
}

// Species constants of a CTA in shared memory (dynamic indexing of kernel parameters
// would go through local memory); with one species they are read as parameters.
struct SpeciesTable {
    float sig2[MAX_PAIR], c48[MAX_PAIR], c24[MAX_PAIR], c4[MAX_PAIR], rc2[MAX_PAIR];
    float rc2lo[MAX_PAIR], rc2hi[MAX_PAIR];  // r_cut^2 (1 -/+ cut_band): the FP64 decision band
    double rc2d[MAX_PAIR];                   // FP64 r_cut^2
};

__device__ __forceinline__ void load_species_table(const PairTable& pt, SpeciesTable& st) {
    const int t = threadIdx.x;
    if (t < MAX_PAIR) {
        st.sig2[t] = pt.sig2_f[t];
        st.c48[t] = pt.c48_f[t];
        st.c24[t] = pt.c24_f[t];
        st.c4[t] = pt.c4_f[t];
        st.rc2[t] = pt.rc2_f[t];
        st.rc2lo[t] = pt.rc2lo_f[t];
        st.rc2hi[t] = pt.rc2hi_f[t];
        st.rc2d[t] = pt.rc2_d[t];
    }
}

// What follows an atom's force in the full-list mixed kernels (MODE as below); one
// function so that every kernel applies exactly the same operations.
template <bool SINGLE, int MODE>
__device__ __forceinline__ void full_epilogue(const DevState& s, const PairTable& pt, int gi, int si, long long qx,
                                              long long qy, long long qz, const StepOut& out, double dt,
                                              float lim2_f) {
    const int64_t n = s.n;
    if (MODE != FM_KKD) {
        s.fq[gi] = qx;
        s.fq[n + gi] = qy;
        s.fq[2 * n + gi] = qz;
    }
    if (MODE != FM_FORCE) {
        const double hq = pt.hdtm_q[SINGLE ? 0 : si];
        const double kq = MODE == FM_KKD ? 2.0 * hq : hq;
        const double vx = fma(kq, (double)qx, s.vx[gi]);
        const double vy = fma(kq, (double)qy, s.vy[gi]);
        const double vz = fma(kq, (double)qz, s.vz[gi]);
        s.vx[gi] = vx;
        s.vy[gi] = vy;
        s.vz[gi] = vz;
        if (MODE == FM_KKD) {
            const double x = fma(dt, vx, s.x[gi]), y = fma(dt, vy, s.y[gi]), z = fma(dt, vz, s.z[gi]);
            out.x[gi] = x;
            out.y[gi] = y;
            out.z[gi] = z;
            const int c = s.cell_of[gi];
            const float4 r = s.xr_ref[gi];
            float4 q;
            q.x = __double2float_rn(x - s.centre[c]);
            q.y = __double2float_rn(y - s.centre[s.ncell + c]);
            q.z = __double2float_rn(z - s.centre[2 * s.ncell + c]);
            q.w = r.w;
            out.xr[gi] = q;
            const float ex = q.x - r.x, ey = q.y - r.y, ez = q.z - r.z;
            if (!(fmaf(ez, ez, fmaf(ey, ey, ex * ex)) <= lim2_f)) *s.rebuild_flag = 1;
        }
    }
}

// The state of an atom's velocity Verlet update as LPA lanes share it, lane q with components q,
// q + LPA, ...: loaded before the pairs, so that the loads and their chains (cell, then its centre)
// run beside them.
template <int MODE, int LPA>
struct LaneState {
    static constexpr int NC = (3 + LPA - 1) / LPA;
    double v[NC], x[NC], centre[NC];
    float4 ref;

    __device__ __forceinline__ void load(const DevState& s, int gi, int lq) {
        if (MODE == FM_FORCE) return;
        int c = 0;
        if (MODE == FM_KKD) {
            c = s.cell_of[gi];
            ref = s.xr_ref[gi];
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            const int d = lq + k * LPA;
            v[k] = x[k] = centre[k] = 0.0;
            if (d < 3) {
                v[k] = (d == 0 ? s.vx : (d == 1 ? s.vy : s.vz))[gi];
                if (MODE == FM_KKD) {
                    x[k] = (d == 0 ? s.x : (d == 1 ? s.y : s.z))[gi];
                    centre[k] = s.centre[d * s.ncell + c];
                }
            }
        }
    }
};

// full_epilogue by the LPA >= 2 lanes of an atom, which all hold its force (q) and their share of
// its state: the same operations, a third or half of the FP64 instructions per warp.  Every lane
// of the warp takes part; write: this atom is to be written.
template <bool SINGLE, int MODE, int LPA>
__device__ __forceinline__ void full_epilogue_lanes(const DevState& s, const PairTable& pt, int gi, int si,
                                                    const long long (&q)[3], const LaneState<MODE, LPA>& st, int lq,
                                                    bool write, const StepOut& out, double dt, float lim2_f) {
    const int64_t n = s.n;
    if (MODE != FM_KKD && write)
        for (int d = lq; d < 3; d += LPA) s.fq[d * n + gi] = d == 0 ? q[0] : (d == 1 ? q[1] : q[2]);
    if (MODE == FM_FORCE) return;
    const double hq = pt.hdtm_q[SINGLE ? 0 : si];
    const double kq = MODE == FM_KKD ? 2.0 * hq : hq;
    float xr[LaneState<MODE, LPA>::NC];
#pragma unroll
    for (int k = 0; k < LaneState<MODE, LPA>::NC; ++k) {
        const int d = lq + k * LPA;
        const double v = fma(kq, (double)(d == 0 ? q[0] : (d == 1 ? q[1] : q[2])), st.v[k]);
        if (write && d < 3) (d == 0 ? s.vx : (d == 1 ? s.vy : s.vz))[gi] = v;
        if (MODE == FM_KKD) {
            const double x = fma(dt, v, st.x[k]);
            if (write && d < 3) (d == 0 ? out.x : (d == 1 ? out.y : out.z))[gi] = x;
            xr[k] = __double2float_rn(x - st.centre[k]);
        }
    }
    if (MODE == FM_KKD) {
        const int l0 = (int)(threadIdx.x & 31) - lq;  // the atom's first lane
        float4 p;
        p.x = __shfl_sync(0xffffffffu, xr[0], l0);
        p.y = __shfl_sync(0xffffffffu, xr[0], l0 + 1);
        p.z = LPA == 2 ? __shfl_sync(0xffffffffu, xr[LPA == 2 ? 1 : 0], l0) : __shfl_sync(0xffffffffu, xr[0], l0 + 2);
        p.w = st.ref.w;
        if (write && lq == 0) {
            out.xr[gi] = p;
            const float ex = p.x - st.ref.x, ey = p.y - st.ref.y, ez = p.z - st.ref.z;
            if (!(fmaf(ez, ez, fmaf(ey, ey, ex * ex)) <= lim2_f)) *s.rebuild_flag = 1;
        }
    }
}

// Exact finish of one atom by one warp (all 32 lanes), for an atom that the FP32 loop
// below cannot finish: a pair whose FP32 r^2 lies within the band around r_cut^2 (the
// cutoff is decided by the FP64 definition) or a pair force component that may reach
// 2048 eps/sigma (beyond the two-part split; or not finite).  About one atom in 1,500 of
// a liquid.  The neighbours come from the CTA's tile, so every other pair gets exactly
// the term the FP32 loop adds; band pairs are decided in FP64 in the oracle's operation
// order; large terms are rounded in FP64 (fix_term_wide).  Each lane keeps the 32-bit
// split sums of the FP32 loop, and the terms they cannot take - large terms, and the
// lane's split sums every FIX_SPLIT_MAX_TERMS terms - go to the warp's exact 64-bit sums
// in shared memory (WarpWide), so this rare path adds no 64-bit registers to the kernel
// it is inlined into.  All sums are exact integers, so the warp total does not depend on
// how the list is spread over the lanes.  The same epilogue follows.  This runs after the
// loop, not inside it: a call from the loop cost the kernel half its speed.
struct WarpWide {
    unsigned long long q[3];
    int nwide;
};

template <bool SINGLE, bool EV, int MODE>
__device__ __forceinline__ void finish_atom_warp(const DevState& s, const Geometry& g, const PairTable& pt,
                                                 const float4* __restrict__ tile, const SpeciesTable& stab,
                                                 const TileMeta& m, int ui, float fs2_max, const StepOut& out,
                                                 double dt, float lim2_f, WarpWide& ww) {
    const int lane = threadIdx.x & 31;
    const int T = m.prefix[64];
    const int gi = m.start[0] + ui;
    const float4 pi = tile[ui];
    const int si = __float_as_int(pi.w);
    const int nsp = pt.nsp;
    const int nent = ((s.nl_cnt[gi] + 7) >> 3) * 8;
    if (lane == 0) {
        ww.q[0] = ww.q[1] = ww.q[2] = 0ull;
        ww.nwide = 0;
    }
    __syncwarp();
    FixAcc ax{0u, 0u}, ay{0u, 0u}, az{0u, 0u};
    int nterms = 0;
    float pe = 0.f, w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f, w4 = 0.f, w5 = 0.f;
    for (int k = lane; k < nent; k += 32) {
        const int u = s.nl[((size_t)(k >> 3) * s.np + gi) * 8 + (k & 7)];
        if (u >= T) continue;  // padding (the tile's dummy slot): no force
        const float4 pj = tile[u];
        const float dx = pi.x - pj.x, dy = pi.y - pj.y, dz = pi.z - pj.z;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        const int t = SINGLE ? 0 : si * nsp + __float_as_int(pj.w);
        const float inv = rcp_approx(r2);
        float fs, s6;  // the FP32 loop's operations, term for term
        if (SINGLE) {
            const float inv2 = __fmul_rn(inv, inv), inv3 = __fmul_rn(inv2, inv);
            fs = __fmul_rn(__fmaf_rn(pt.lj_a_f, inv3, -pt.lj_b_f), __fmul_rn(inv2, inv2));
            s6 = __fmul_rn(pt.sig6_f, inv3);
        } else {
            const float s2 = __fmul_rn(stab.sig2[t], inv);
            s6 = __fmul_rn(__fmul_rn(s2, s2), s2);
            fs = __fmul_rn(__fmul_rn(__fmaf_rn(stab.c48[t], s6, -stab.c24[t]), s6), inv);
        }
        bool inside = r2 < (SINGLE ? pt.rc2lo_f[0] : stab.rc2lo[t]);
        if (!inside && r2 < (SINGLE ? pt.rc2hi_f[0] : stab.rc2hi[t]))
            inside = fp64_pair_test(s.x, s.y, s.z, g.L[0], g.L[1], g.L[2], gi, tile_global_index(m, u),
                                    SINGLE ? pt.rc2_d[0] : stab.rc2d[t]);
        const float fs2 = inside ? fs : 0.0f;
        if (fabsf(fs2) < fs2_max) {
            fix_add(ax, fs2, dx);
            fix_add(ay, fs2, dy);
            fix_add(az, fs2, dz);
            if (++nterms == FIX_SPLIT_MAX_TERMS) {  // only for lists of more than 16,000 entries
                atomicAdd(&ww.q[0], (unsigned long long)fix_final(ax, nterms));
                atomicAdd(&ww.q[1], (unsigned long long)fix_final(ay, nterms));
                atomicAdd(&ww.q[2], (unsigned long long)fix_final(az, nterms));
                ax = ay = az = FixAcc{0u, 0u};
                nterms = 0;
            }
        } else {
            atomicAdd(&ww.q[0], (unsigned long long)fix_term_wide(fs2, dx, s.err));
            atomicAdd(&ww.q[1], (unsigned long long)fix_term_wide(fs2, dy, s.err));
            atomicAdd(&ww.q[2], (unsigned long long)fix_term_wide(fs2, dz, s.err));
            atomicAdd(&ww.nwide, 1);
        }
        if (EV && inside) {
            const float gq = fs2 * (1.0f / FS_SCALE);
            pe += (SINGLE ? pt.c4_f[0] : stab.c4[t]) * s6 * (s6 - 1.0f);
            w0 += dx * (gq * dx);
            w1 += dy * (gq * dy);
            w2 += dz * (gq * dz);
            w3 += dx * (gq * dy);
            w4 += dx * (gq * dz);
            w5 += dy * (gq * dz);
        }
    }
    long long qx = fix_final(ax, nterms), qy = fix_final(ay, nterms), qz = fix_final(az, nterms);
    __syncwarp();
    if (lane == 0) {
        fix_wide_count_ok(ww.nwide, s.err);
        qx += (long long)ww.q[0];
        qy += (long long)ww.q[1];
        qz += (long long)ww.q[2];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        qx += __shfl_xor_sync(0xffffffffu, qx, o);
        qy += __shfl_xor_sync(0xffffffffu, qy, o);
        qz += __shfl_xor_sync(0xffffffffu, qz, o);
        if (EV) {  // a fixed butterfly: the FP32 sums are reproducible
            pe += __shfl_xor_sync(0xffffffffu, pe, o);
            w0 += __shfl_xor_sync(0xffffffffu, w0, o);
            w1 += __shfl_xor_sync(0xffffffffu, w1, o);
            w2 += __shfl_xor_sync(0xffffffffu, w2, o);
            w3 += __shfl_xor_sync(0xffffffffu, w3, o);
            w4 += __shfl_xor_sync(0xffffffffu, w4, o);
            w5 += __shfl_xor_sync(0xffffffffu, w5, o);
        }
    }
    if (lane == 0) {
        full_epilogue<SINGLE, MODE>(s, pt, gi, si, qx, qy, qz, out, dt, lim2_f);
        if (EV) {
            const int64_t n = s.n;
            s.pe_atom_f[gi] = 0.5f * pe;
            s.vir_atom_f[gi] = 0.5f * w0;
            s.vir_atom_f[n + gi] = 0.5f * w1;
            s.vir_atom_f[2 * n + gi] = 0.5f * w2;
            s.vir_atom_f[3 * n + gi] = 0.5f * w3;
            s.vir_atom_f[4 * n + gi] = 0.5f * w4;
            s.vir_atom_f[5 * n + gi] = 0.5f * w5;
        }
    }
}

// Two list entries of one atom (tile coordinates pi, species si), in packed FP32x2 arithmetic;
// each neighbour is one 128-bit shared-memory load.  The sums are single references: as the
// members of a struct they cost the kernel at its register cap 1.3 % (285.6 against 281.8 us
// at 2,048,000 atoms).  bad, and for one species the minima mdist and mr2, send an atom to the
// exact finish.
template <bool SINGLE, bool EV>
__device__ __forceinline__ void full_pair(const PairTable& pt, const SpeciesTable& stab, unsigned tile_s,
                                          const float4& pi, int si, int nsp, float fs2_max, f2_t magic2, f2_t two21,
                                          int u0, int u1, FixAcc& ax, FixAcc& ay, FixAcc& az, float& pe, float& w0,
                                          float& w1, float& w2, float& w3, float& w4, float& w5, bool& bad, float& mdist,
                                          float& mr2) {
    const float4 pa = lds_tile(tile_s, u0);
    const float4 pb = lds_tile(tile_s, u1);
    // scalar differences land directly in the register pairs of the packed operands
    const f2_t dx = f2_pack(__fsub_rn(pi.x, pa.x), __fsub_rn(pi.x, pb.x));
    const f2_t dy = f2_pack(__fsub_rn(pi.y, pa.y), __fsub_rn(pi.y, pb.y));
    const f2_t dz = f2_pack(__fsub_rn(pi.z, pa.z), __fsub_rn(pi.z, pb.z));
    const f2_t r2 = f2_fma(dz, dz, f2_fma(dy, dy, f2_mul(dx, dx)));
    float r2a, r2b;
    f2_unpack(r2, r2a, r2b);
    const f2_t inv = f2_pack(rcp_approx(r2a), rcp_approx(r2b));
    float fa, fb;
    f2_t s6;  // (sigma^2 / r^2)^3, for the energy
    bool ina, inb;
    if (SINGLE) {
        // fs2 = inv^4 (a inv^3 - b): the constants are kernel parameters
        const f2_t inv2 = f2_mul(inv, inv);
        const f2_t inv3 = f2_mul(inv2, inv);
        const f2_t t = f2_fma(f2_pack(pt.lj_a_f, pt.lj_a_f), inv3, f2_pack(-pt.lj_b_f, -pt.lj_b_f));
        f2_unpack(f2_mul(t, f2_mul(inv2, inv2)), fa, fb);
        if (EV) s6 = f2_mul(f2_pack(pt.sig6_f, pt.sig6_f), inv3);
        // inside for certain below the band, tentatively inside up to its top: a pair
        // in the band leaves the atom to finish_atom_warp (FP64 cutoff decision)
        ina = r2a < pt.rc2hi_f[0];
        inb = r2b < pt.rc2hi_f[0];
        float dca, dcb;
        f2_unpack(f2_sub(r2, f2_pack(pt.rc2_f[0], pt.rc2_f[0])), dca, dcb);  // exact near r_cut
        mdist = fminf(mdist, fminf(fabsf(dca), fabsf(dcb)));
        mr2 = fminf(mr2, fminf(r2a, r2b));
    } else {
        const int ta = si * nsp + __float_as_int(pa.w);
        const int tb = si * nsp + __float_as_int(pb.w);
        const f2_t s2 = f2_mul(f2_pack(stab.sig2[ta], stab.sig2[tb]), inv);
        s6 = f2_mul(f2_mul(s2, s2), s2);
        f2_unpack(f2_mul(f2_mul(f2_fma(f2_pack(stab.c48[ta], stab.c48[tb]), s6,
                                       f2_pack(-stab.c24[ta], -stab.c24[tb])),
                                s6),
                         inv),
                  fa, fb);
        ina = r2a < stab.rc2hi[ta];
        inb = r2b < stab.rc2hi[tb];
        bad |= !(fabsf(fa) < fs2_max) | !(fabsf(fb) < fs2_max) | (ina != (r2a < stab.rc2lo[ta])) |
               (inb != (r2b < stab.rc2lo[tb]));
    }
    fa = ina ? fa : 0.0f;
    fb = inb ? fb : 0.0f;
    const f2_t fs2 = f2_pack(fa, fb);
    fix_add2(ax, fs2, dx, magic2, two21);
    fix_add2(ay, fs2, dy, magic2, two21);
    fix_add2(az, fs2, dz, magic2, two21);
    if (EV) {
        float s6a, s6b, dxa, dxb, dya, dyb, dza, dzb;
        f2_unpack(s6, s6a, s6b);
        f2_unpack(dx, dxa, dxb);
        f2_unpack(dy, dya, dyb);
        f2_unpack(dz, dza, dzb);
        const int ta = SINGLE ? 0 : si * nsp + __float_as_int(pa.w);
        const int tb = SINGLE ? 0 : si * nsp + __float_as_int(pb.w);
        const float c4a = SINGLE ? pt.c4_f[0] : stab.c4[ta], c4b = SINGLE ? pt.c4_f[0] : stab.c4[tb];
        const float ua = ina ? c4a * s6a * (s6a - 1.0f) : 0.0f;
        const float ub = inb ? c4b * s6b * (s6b - 1.0f) : 0.0f;
        const float ga = fa * (1.0f / FS_SCALE), gb = fb * (1.0f / FS_SCALE);
        pe += ua + ub;
        w0 += dxa * (ga * dxa) + dxb * (gb * dxb);
        w1 += dya * (ga * dya) + dyb * (gb * dyb);
        w2 += dza * (ga * dza) + dzb * (gb * dzb);
        w3 += dxa * (ga * dya) + dxb * (gb * dyb);
        w4 += dxa * (ga * dza) + dxb * (gb * dzb);
        w5 += dya * (ga * dza) + dyb * (gb * dzb);
    }
}

}  // namespace mdgb
