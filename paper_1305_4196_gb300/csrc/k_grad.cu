// k_grad.cu - reverse-mode derivatives of the Lennard-Jones forces (force matching).
//
// For a scalar loss L of the forces with G = dL/dF given, the chain rule over the
// pairs inside their cutoffs (the pair set held fixed: the cutoff contributes no
// derivative) gives, per pair (i, j) with d = x_i - x_j, f_ij = g(r^2) d and
// w = G_i - G_j:
//     dL/dx_i += g w + 2 g' (w . d) d          (and the negative on x_j)
//     dL/deps_ab += (w . d) g / eps
//     dL/dsig_ab += (w . d) * 144 eps (4 s6^2 - s6) / (sig r^2)
// with s6 = (sig^2/r^2)^3, g = 24 eps (2 s6^2 - s6) / r^2 and
// g' = dg/d(r^2) = 24 eps (4 s6 - 14 s6^2) / r^4.  The energy's parameter
// derivatives, dE/deps_ab = sum 4 (s6^2 - s6) and dE/dsig_ab = sum 24 eps
// (2 s6^2 - s6) / sig, come from the same pass.
//
// One CTA per 2x2x2-cell block with the block's 4x4x4-cell tile in shared memory, as in the
// full-list force kernels; an atom accumulates only its own dL/dx_i (each pair is seen from
// both sides, which also gives the negative term on x_j).  T = double on FP64 systems, float
// (FP32 pair arithmetic, block-frame coordinates) on mixed-precision ones.
//  * Four lanes share an atom, lane q with word q (entries 2q, 2q + 1) of every 16-byte chunk of the
//    list, so a warp reads its lists in whole sectors and a system of a few 10^4 atoms fills
//    the SMs.
//  * The parameter terms leave out the factors that their species pair shares and are
//    summed in the CTA, to one row of partial sums per CTA instead of one per atom.
//  * The summation order is fixed, so every result is deterministic.
// The pass is bound by instruction issue and the latency of the gathered G_j.  For 32,000 atoms of a
// binary mixture it took 217 us with one lane per atom, 2-byte list reads and FP64 sums, and 47 us
// for the column sums of a row per atom; it takes 45 us (28 for the energy's derivatives) and 3.
#include "tile.cuh"

#include <algorithm>
#include <type_traits>

#include "fixpt.cuh"
#include "float_sum.cuh"
#include "launch.cuh"

namespace mdgb {

constexpr int G_LPA = 4;  // lanes per own atom
constexpr int G_THREADS = 512;
constexpr int G_ATOMS = G_THREADS / G_LPA;  // own atoms at a time
constexpr int G_QUANT = 2;                  // per species pair: the derivatives by eps and by sig

// G of one atom in the arithmetic of the pairs.
template <typename T>
struct alignas(4 * sizeof(T)) Grad4 {
    T x, y, z, w;
};

// A lane's sums of a pair's two terms: FP64 terms in FP64, FP32 terms in three floats (FloatSum: no less
// exact than FP64 sums; an FP64 addition and the conversion before it would hold a warp as long as
// some 100 FP32 operations).
template <typename T>
using ParamSums = std::conditional_t<sizeof(T) == 8, DoubleSum2, FloatSum2>;

// The sums of a warp by species pair and quantity, of lanes that hold them for an atom of species si by
// its neighbours' species.  Half of them to each half of an atom's lanes, twice: a lane keeps VPL;
// then the warp's atoms of one species after the other, whose sums stay with the lanes 4 c .. 4 c + 3
// of species c.
template <int NSP>
struct WarpColumns {
    static constexpr int NV = NSP * G_QUANT, VPL = (NV + 3) / 4, PAIRS = 2 * VPL;

    template <typename S>
    static __device__ __forceinline__ S over_species(const S& mine, int si) {
        const int lane = threadIdx.x & 31;
        S kept;
#pragma unroll
        for (int c = 0; c < NSP; ++c) {
            S v = NSP == 1 || si == c ? mine : S();
#pragma unroll
            for (int o = G_LPA; o < 32; o <<= 1) v.add(lane_xor(v, o));
            if (lane >> 2 == c) kept = v;
        }
        return kept;
    }

    template <typename P>
    static __device__ __forceinline__ void get(P (&val)[PAIRS], int si, double (&out)[VPL]) {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int o = 2, m = VPL; m > 0 && o > 0; o >>= 1, m >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int k = 0; k < m; ++k) {
                const P give = up ? val[k] : val[k + m];
                if (up) val[k] = val[k + m];
                val[k].add(lane_xor(give, o));
            }
        }
        if constexpr (VPL == 1) {
            const bool up = (lane & 1) != 0;
            auto v = val[0].half(up);
            v.add(lane_xor(val[0].half(!up), 1));
            out[0] = over_species(v, si).get();
        } else {
            const P v = over_species(val[0], si);
            out[0] = v.half(false).get();
            out[1] = v.half(true).get();
        }
    }
    // the column (species pair t, quantity q: 2 t + q) of this lane's j-th sum; negative: none
    static __device__ __forceinline__ int column(int j) {
        const int lane = threadIdx.x & 31, c = lane >> 2, v = (lane & 3) * VPL + j;
        return c < NSP && v < NV ? c * NV + v : -1;
    }
};

// 1/x, correctly rounded.  FP32: one Newton step from the approximate one (compared with the division over
// all significands at exponents -30 .. 30), 5 % of the pass's time less than a division; FP64: the division,
// 2 % (the loss's derivatives) and 4 % (the energy's) more than a cubic step from an FP32 seed, which is an
// ulp off for two numbers in a million.
__device__ __forceinline__ float grad_rcp(float x) {
    const float y = rcp_approx(x);
    return __fmaf_rn(y, __fmaf_rn(-x, y, 1.0f), y);
}
__device__ __forceinline__ double grad_rcp(double x) { return 1.0 / x; }

// Per species pair, in shared memory: the lanes of a warp read several entries at once, which the
// constant bank would serve one after another.  (FP64 keeps 24 eps there: the tile takes the rest.)
template <typename T, int NT>
struct GradTable;

template <int NT>
struct GradTable<float, NT> {
    float sig2[NT], e24[NT], in[NT], out[NT];  // inside below `in`, outside from `out` on
};

template <int NT>
struct GradTable<double, NT> {
    double sig2[NT], out[NT];
};

// part_out: column by column (species pair t, quantity q: 2 t + q), each CTA's sum of its own atoms'
// terms.  Each unordered pair is visited from both sides, so every term is halved.
// EN: the energy's parameter derivatives (G_ is not read); otherwise those of the loss.
template <typename T, int NSP, bool EN>
__global__ void __launch_bounds__(G_THREADS, 2) k_force_backward(DevState s, Geometry g, PairTable pt, TileOffsets to,
                                                                 int tile_cap, const void* __restrict__ G_,
                                                                 double* __restrict__ gx_out,
                                                                 double* __restrict__ part_out, int split) {
    constexpr bool FP64 = sizeof(T) == 8;
    constexpr int NC = NSP * NSP * G_QUANT;  // sums per CTA
    static_assert(NC <= 32, "one lane per sum");
    const Grad4<T>* __restrict__ G = reinterpret_cast<const Grad4<T>*>(G_);
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileMeta m;
    __shared__ GradTable<T, NSP * NSP> tab;
    // split CTAs share one block: each stages the whole tile and takes every split-th group of
    // own atoms, so that a small system still spreads over the SMs
    const int b = spatial_block(g, blockIdx.x / split), part = blockIdx.x % split;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int nw = G_THREADS / 32;
    if (threadIdx.x < NSP * NSP) {
        if constexpr (FP64) {
            tab.sig2[threadIdx.x] = pt.sig2_d[threadIdx.x];
            tab.out[threadIdx.x] = pt.rc2_d[threadIdx.x];
        } else {
            tab.sig2[threadIdx.x] = pt.sig2_f[threadIdx.x];
            tab.e24[threadIdx.x] = 6.0f * pt.c4_f[threadIdx.x];
            tab.in[threadIdx.x] = pt.rc2lo_f[threadIdx.x];
            tab.out[threadIdx.x] = pt.rc2hi_f[threadIdx.x];
        }
    }
    tile_meta(g, s.cell_start, b, m);
    const int T_ = m.prefix[64], nown = m.prefix[8];
    if (T_ + 1 > tile_cap || part * G_ATOMS >= nown) {
        if (threadIdx.x == 0 && T_ + 1 > tile_cap) atomicOr(s.err, ERR_TILE_OVERFLOW);
        if (threadIdx.x < NC) part_out[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = 0.0;
        return;
    }
    // the tile: FP64 as x | y | z | species, FP32 as (x, y, z, species); behind it the atoms' global
    // indices
    double* tx = reinterpret_cast<double*>(smem);
    double *ty = tx + tile_cap, *tz = ty + tile_cap;
    int* tsp = reinterpret_cast<int*>(tz + tile_cap);
    float4* tp = reinterpret_cast<float4*>(smem);
    int* gid = FP64 ? tsp + tile_cap : reinterpret_cast<int*>(tp + tile_cap);
    if (FP64) {
        tile_stage_f64(s, g, m, b, tx, ty, tz, tsp, m.prefix);
    } else {
        tile_stage_f32_cells(m, s.xr, to, tp);
        if (threadIdx.x == 0) tp[T_] = make_float4(1.0e4f, 1.0e4f, 1.0e4f, __int_as_float(0));
    }
    for (int slot = warp; slot < 64; slot += nw) {
        const int u0 = m.prefix[slot], cnt = m.prefix[slot + 1] - u0, j0 = m.start[slot];
        for (int e = lane; e < cnt; e += 32) gid[u0 + e] = j0 + e;
    }
    __syncthreads();
    const int blk0 = m.start[0];
    const size_t np = s.np;
    const int lq = threadIdx.x % G_LPA;
    using Columns = WarpColumns<NSP>;
    constexpr int VPL = Columns::VPL;
    double mine[VPL] = {};  // the warp's sums, by the lanes that Columns says
    for (int u0 = part * G_ATOMS; u0 < nown; u0 += split * G_ATOMS) {
        const int ui = u0 + (int)threadIdx.x / G_LPA;
        const bool active = ui < nown;
        const int uc = active ? ui : 0, gi = blk0 + uc;
        T xi, yi, zi;
        int si;
        if (FP64) {
            xi = (T)tx[uc], yi = (T)ty[uc], zi = (T)tz[uc];
            si = tsp[uc];
        } else {
            const float4 p = tp[uc];
            xi = p.x, yi = p.y, zi = p.z;
            si = __float_as_int(p.w);
        }
        Grad4<T> Gi{};
        if (!EN) Gi = G[gi];
        T a[3] = {T(0), T(0), T(0)};
        ParamSums<T> sum[Columns::PAIRS];  // by the neighbour's species
        // neighbour u; take(its species, the pair's two terms, its part of dL/dx) if it is inside the cutoff
        const auto visit = [&](int u, auto&& take) {
            T dx, dy, dz;
            int sj;
            if (FP64) {
                dx = xi - (T)tx[u], dy = yi - (T)ty[u], dz = zi - (T)tz[u];
                sj = tsp[u];
            } else {
                const float4 p = tp[u];
                dx = xi - p.x, dy = yi - p.y, dz = zi - p.z;
                sj = __float_as_int(p.w);
            }
            const T r2 = dx * dx + dy * dy + dz * dz;
            const int t = NSP == 1 ? 0 : si * NSP + sj;
            if (!(r2 < tab.out[t])) return;
            if constexpr (!FP64) {
                if (!(r2 < tab.in[t]) &&  // rare: decide the cutoff in FP64
                    !fp64_pair_test(s.x, s.y, s.z, g.L[0], g.L[1], g.L[2], gi, gid[u], pt.rc2_d[t]))
                    return;
            }
            const T inv = grad_rcp(r2);
            const T sr2 = tab.sig2[t] * inv;
            const T s6 = sr2 * sr2 * sr2;
            const T v = T(2) * s6 * s6 - s6;
            if (EN) {  // dE/deps / 4, dE/dsig sig / (24 eps)
                take(sj, s6 * s6 - s6, v, T(0), T(0), T(0));
            } else {
                const Grad4<T> Gj = G[gid[u]];
                const T wx = Gi.x - Gj.x, wy = Gi.y - Gj.y, wz = Gi.z - Gj.z;
                const T wd = wx * dx + wy * dy + wz * dz;
                T e24;
                if constexpr (FP64) e24 = 24.0 * pt.eps_d[t];
                else e24 = tab.e24[t];
                const T gq = e24 * v * inv;
                const T h = T(2) * (e24 * (T(4) * s6 - T(14) * s6 * s6) * inv * inv) * wd;
                const T wi = wd * inv;  // dL/deps / 24, dL/dsig sig / (144 eps)
                take(sj, wi * v, wi * (T(4) * s6 * s6 - s6), gq * wx + h * dx, gq * wy + h * dy, gq * wz + h * dz);
            }
        };
        const int nch = active ? (s.nl_cnt[gi] + 7) >> 3 : 0;
        const unsigned* words = reinterpret_cast<const unsigned*>(s.nl) + (size_t)gi * 4 + lq;
        const auto walk = [&](auto&& take) {
            unsigned nxt = nch > 0 ? __ldcs(words) : 0u;
            for (int c = 0; c < nch; ++c) {
                const unsigned w = nxt;
                if (c + 1 < nch) nxt = __ldcs(words + (size_t)(c + 1) * np * 4);
                visit((int)(w & 0xffffu), take);
                visit((int)(w >> 16), take);
            }
        };
        walk([&](int sj, T q0, T q1, T ax, T ay, T az) {
            a[0] += ax;
            a[1] += ay;
            a[2] += az;
#pragma unroll
            for (int k = 0; k < NSP; ++k) {
                const bool take = NSP == 1 || sj == k;
                sum[k].add(take ? q0 : T(0), take ? q1 : T(0));
            }
        });
        __syncwarp();
        if (!EN) {
#pragma unroll
            for (int o = 1; o < G_LPA; o <<= 1) {
#pragma unroll
                for (int d = 0; d < 3; ++d) a[d] += __shfl_xor_sync(0xffffffffu, a[d], o);
            }
            if (gx_out && active && lq < 3) {
                const T v = lq == 0 ? a[0] : (lq == 1 ? a[1] : a[2]);
                gx_out[3 * (size_t)s.orig[gi] + lq] = (double)v;
            }
        }
        double columns[VPL];
        Columns::get(sum, si, columns);
        if constexpr (!FP64) {
            bool bad = false;
#pragma unroll
            for (int j = 0; j < VPL; ++j) bad |= !isfinite(columns[j]);
            if (__any_sync(0xffffffffu, bad)) {  // (FloatSum) the warp's atoms again, in FP64
                DoubleSum2 wide[Columns::PAIRS];
                walk([&](int sj, T q0, T q1, T, T, T) {
#pragma unroll
                    for (int k = 0; k < NSP; ++k)
                        if (NSP == 1 || sj == k) wide[k].add((double)q0, (double)q1);
                });
                __syncwarp();
                Columns::get(wide, si, columns);
            }
        }
#pragma unroll
        for (int j = 0; j < VPL; ++j) mine[j] += columns[j];
    }
    __syncthreads();
    double* red = reinterpret_cast<double*>(smem);  // the tile is done with: NC sums of each warp
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const int c = Columns::column(j);
        if (c >= 0) red[warp * NC + c] = mine[j];
    }
    __syncthreads();
    if (threadIdx.x < NC) {
        double v = 0.0;
        for (int k = 0; k < nw; ++k) v += red[k * NC + threadIdx.x];
        // the factors left out above, halved
        const int t = threadIdx.x / G_QUANT, q = threadIdx.x % G_QUANT;
        const double f = EN ? (q ? 12.0 * pt.eps_d[t] / pt.sig_d[t] : 2.0)
                            : (q ? 72.0 * pt.eps_d[t] / pt.sig_d[t] : 12.0);
        part_out[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = f * v;
    }
}

// Column sums of the CTAs' partial sums (column by column), one CTA per column, in a fixed order.
constexpr int CS_THREADS = 256;

__global__ void __launch_bounds__(CS_THREADS) k_colsum(const double* __restrict__ part, int nparts,
                                                       double* __restrict__ out) {
    __shared__ double sh[CS_THREADS];
    double acc = 0.0;
    for (int p = threadIdx.x; p < nparts; p += CS_THREADS) acc += part[(size_t)blockIdx.x * nparts + p];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int w = CS_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

// G (N x 3, original order) -> cell order, one (x, y, z, -) entry per atom
template <typename T>
__global__ void k_grad_in(DevState s, const double* __restrict__ G, Grad4<T>* __restrict__ Gc) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int64_t o = s.orig[i];
    Gc[i] = Grad4<T>{(T)G[3 * o], (T)G[3 * o + 1], (T)G[3 * o + 2], T(0)};
}

size_t backward_smem_bytes(int fp64, int tile_cap) {
    // (the reduction at the end reuses the tile's memory)
    return std::max((size_t)tile_cap * (3 * (fp64 ? sizeof(double) : sizeof(float)) + 2 * sizeof(int)),
                    sizeof(double) * G_THREADS);
}

BackwardPlan backward_plan(const LaunchGeometry& g, int nsp, int fp64, int64_t n) {
    BackwardPlan p;
    const int64_t per_block = (n + g.nblock - 1) / g.nblock;
    const int64_t split =
        std::min<int64_t>((per_block + G_ATOMS - 1) / G_ATOMS, (2 * g.sms + g.nblock - 1) / g.nblock);
    p.split = (int)std::max<int64_t>(1, std::min<int64_t>(split, 8));
    const size_t ncol = (size_t)nsp * nsp * G_QUANT;
    p.sums = (ncol * (1 + (size_t)g.nblock * p.split) + 3) & ~(size_t)3;
    p.doubles = p.sums + (size_t)n * (fp64 ? 4 : 2);
    return p;
}

using Backward = void (*)(DevState, Geometry, PairTable, TileOffsets, int, const void*, double*, double*, int);

template <typename T, bool EN>
static Backward backward_of(int nsp) {
    switch (nsp) {
        case 1: return k_force_backward<T, 1, EN>;
        case 2: return k_force_backward<T, 2, EN>;
        case 3: return k_force_backward<T, 3, EN>;
        default: return k_force_backward<T, 4, EN>;
    }
}

static Backward backward_kernel(int fp64, int energy, int nsp) {
    if (fp64) return energy ? backward_of<double, true>(nsp) : backward_of<double, false>(nsp);
    return energy ? backward_of<float, true>(nsp) : backward_of<float, false>(nsp);
}

// With G: dL/deps and dL/dsig (columns 2 t and 2 t + 1 of the totals at the start of the scratch), and
// dL/dx in the caller's order into gx.  Without: dE/deps and dE/dsig.
void launch_force_backward(const DevState& s, const Geometry& g, const PairTable& pt, const TileOffsets& to,
                           int tile_cap, int fp64, const BackwardPlan& plan, const double* G, double* gx,
                           double* scratch, cudaStream_t st) {
    const int64_t n = s.n;
    const int ncol = pt.nsp * pt.nsp * G_QUANT;
    const unsigned grid = (unsigned)g.nblock * (unsigned)plan.split;
    double* part = scratch + ncol;
    double* Gc = scratch + plan.sums;
    const int bs = 256;
    const unsigned nb = (unsigned)((n + bs - 1) / bs);
    if (G) {
        if (fp64) k_grad_in<<<nb, bs, 0, st>>>(s, G, reinterpret_cast<Grad4<double>*>(Gc));
        else k_grad_in<<<nb, bs, 0, st>>>(s, G, reinterpret_cast<Grad4<float>*>(Gc));
    }
    backward_kernel(fp64, G == nullptr, pt.nsp)<<<grid, G_THREADS, backward_smem_bytes(fp64, tile_cap), st>>>(
        s, g, pt, to, tile_cap, Gc, gx, part, plan.split);
    k_colsum<<<ncol, CS_THREADS, 0, st>>>(part, (int)grid, scratch);
}

void init_grad_kernels(int fp64, int nsp) {
    for (int energy = 0; energy < 2; ++energy) allow_max_smem(backward_kernel(fp64, energy, nsp));
}

}  // namespace mdgb
