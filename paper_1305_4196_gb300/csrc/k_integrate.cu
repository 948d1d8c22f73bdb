// k_integrate.cu - velocity Verlet, displacement test, FP64 reductions and state I/O.
//
// The paper integrates the equations of motion with a plain particle-parallel
// loop (Sec. II.A, Sec. II.C).  The integrator is textbook velocity Verlet:
//     v += (dt/2m) F;  x += dt v;  [rebuild test];  F = F(x);  v += (dt/2m) F
// with every operation rounded exactly as written (no contraction), so that
// given identical forces the FP64 trajectory matches the definition bit for bit.
// Consecutive steps fuse the closing half kick of one step with the opening
// half kick and drift of the next (the same operations, one kernel).
//
// Energies use the paper's thread-local accumulators (Sec. II.C) in a fixed
// order: per-atom shares, then per-CTA FP64 partials, then the last CTA sums those.
#include "float_sum.cuh"
#include "mdgb_internal.cuh"

#include <algorithm>
#include <type_traits>

namespace mdgb {

__device__ __forceinline__ double force_of(const DevState& s, int mixed, int64_t i) {
    return mixed ? (double)s.fq[i] * 2.3283064365386963e-10 /* 2^-32 */ : s.f[i];
}

// mode: INT_KICK_DRIFT (first step), INT_KICK_KICK_DRIFT (close step, open next), INT_KICK (close)
//
// FP64 path: every operation rounded exactly as written, as the definition.
// Mixed path: the same update in fused form (one FMA per kick of the fixed-point
// force, one per drift, a fused double kick between steps); GB300 runs FP64 at
// 1/64 of the FP32 rate, so the FP64 instruction count sets this kernel's time.
__global__ void k_integrate(DevState s, Geometry g, PairTable pt, int mode, int mixed, double dt, double lim2,
                            float lim2_f) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int64_t n = s.n;
    const int sp = s.species[i];
    double v[3] = {s.vx[i], s.vy[i], s.vz[i]};
    if (mixed) {
        const double hq = pt.hdtm_q[sp];
        const double kq = mode == INT_KICK_KICK_DRIFT ? 2.0 * hq : hq;
        const double F[3] = {(double)s.fq[i], (double)s.fq[n + i], (double)s.fq[2 * n + i]};
#pragma unroll
        for (int d = 0; d < 3; ++d) v[d] = fma(kq, F[d], v[d]);
    } else {
        const double h = pt.hdtm[sp];
        const double F[3] = {s.f[i], s.f[n + i], s.f[2 * n + i]};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            if (mode != INT_KICK_DRIFT) v[d] = __dadd_rn(v[d], __dmul_rn(h, F[d]));
            if (mode != INT_KICK) v[d] = __dadd_rn(v[d], __dmul_rn(h, F[d]));
        }
    }
    s.vx[i] = v[0];
    s.vy[i] = v[1];
    s.vz[i] = v[2];
    if (mode == INT_KICK) return;
    double x[3] = {s.x[i], s.y[i], s.z[i]};
    bool moved;
    if (mixed) {
#pragma unroll
        for (int d = 0; d < 3; ++d) x[d] = fma(dt, v[d], x[d]);
        // FP32 coordinates relative to the build cell's centre, and the displacement test on them
        const int c = s.cell_of[i];
        float4 p;
        p.x = __double2float_rn(x[0] - s.centre[c]);
        p.y = __double2float_rn(x[1] - s.centre[s.ncell + c]);
        p.z = __double2float_rn(x[2] - s.centre[2 * s.ncell + c]);
        const float4 r = s.xr_ref[i];
        p.w = r.w;
        s.xr[i] = p;
        const float dx = p.x - r.x, dy = p.y - r.y, dz = p.z - r.z;
        moved = fmaf(dz, dz, fmaf(dy, dy, dx * dx)) > lim2_f;
    } else {
#pragma unroll
        for (int d = 0; d < 3; ++d) x[d] = __dadd_rn(x[d], __dmul_rn(dt, v[d]));
        const double dx = __dsub_rn(x[0], s.rx[i]);
        const double dy = __dsub_rn(x[1], s.ry[i]);
        const double dz = __dsub_rn(x[2], s.rz[i]);
        const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
        moved = d2 > lim2;
    }
    s.x[i] = x[0];
    s.y[i] = x[1];
    s.z[i] = x[2];
    if (moved) *s.rebuild_flag = 1;
}

void launch_integrate(const DevState& s, const Geometry& g, const PairTable& pt, int mode, int mixed,
                      double dt, double lim2, cudaStream_t st) {
    if (s.n == 0) return;
    int bs = 256;
    // the FP32 test is made slightly stricter so that FP32 rounding can never let an atom
    // move further than skin/2 without a rebuild
    float lim2_f = (float)(lim2 * (1.0 - 1e-4));
    k_integrate<<<(unsigned)((s.n + bs - 1) / bs), bs, 0, st>>>(s, g, pt, mode, mixed, dt, lim2, lim2_f);
}

// ---------------------------------------------------------------- step control (graph mode)
// One thread decides whether this step rebuilds the lists: the skin/2 flag raised
// by k_integrate, or every k-th step.  It sets the graph's IF-node condition,
// clears the flag for the next step and advances the device step counter.
__global__ void k_step_ctrl(int policy, int every_k, int32_t* rebuild_flag, long long* step_counter,
                            uint32_t* err, cudaGraphConditionalHandle handle) {
    const long long step = *step_counter + 1;
    const int moved = *rebuild_flag;
    int rebuild;
    if (policy == 1) {
        rebuild = (step % every_k) == 0;
        if (moved && !rebuild) atomicOr(err, ERR_SKIN);
    } else {
        rebuild = moved != 0;
    }
    *rebuild_flag = 0;
    *step_counter = step;
    cudaGraphSetConditional(handle, rebuild ? 1u : 0u);
}

// The while node over a chunk's steps: another pass as long as some are left; done: the passes
// that just ended.
__global__ void k_loop_ctrl(long long* passes_left, int done, cudaGraphConditionalHandle handle) {
    const long long left = *passes_left - done;
    *passes_left = left;
    cudaGraphSetConditional(handle, left > 0 ? 1u : 0u);
}

void launch_loop_ctrl(long long* passes_left, int done, cudaGraphConditionalHandle handle, cudaStream_t st) {
    k_loop_ctrl<<<1, 1, 0, st>>>(passes_left, done, handle);
}

void launch_step_ctrl(int policy, int every_k, int32_t* rebuild_flag, long long* step_counter,
                      uint32_t* err, cudaGraphConditionalHandle handle, cudaStream_t st) {
    k_step_ctrl<<<1, 1, 0, st>>>(policy, every_k, rebuild_flag, step_counter, err, handle);
}

// snapshot copy of the permuted state (positions, velocities, images, species, ids)
__global__ void k_copy_state(DevState d, DevState s) {
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (t >= s.n) return;
    d.x[t] = s.x[t];
    d.y[t] = s.y[t];
    d.z[t] = s.z[t];
    d.vx[t] = s.vx[t];
    d.vy[t] = s.vy[t];
    d.vz[t] = s.vz[t];
    d.ix[t] = s.ix[t];
    d.iy[t] = s.iy[t];
    d.iz[t] = s.iz[t];
    d.species[t] = s.species[t];
    d.orig[t] = s.orig[t];
}

void launch_copy_state(const DevState& dst, const DevState& src, cudaStream_t st) {
    if (src.n == 0) return;
    int bs = 256;
    k_copy_state<<<(unsigned)((src.n + bs - 1) / bs), bs, 0, st>>>(dst, src);
}

// ---------------------------------------------------------------- reductions
// (PE, KE, W_xx, W_yy, W_zz, W_xy, W_xz, W_yz): partial[b][0..7] over a contiguous chunk, each thread
// summing a fixed strided subset in order, then the lanes of a warp, then the warps, in a fixed
// shape; the CTA that finishes last sums the partials.
//
// The FP64 pipe would bound this (an SM takes 16 cycles for a warp's FP64 addition or conversion), so
// FP32 shares are added in three floats up to the warp's sums (FloatSum: no less exact than FP64
// sums), and the lanes of a warp add each column in a part of the warp only.  At 1,048,576 atoms
// 54 us with FP64 sums per thread and a second launch, 18 so; at 2,048 atoms 14 and 4.9, at 360,703 in
// FP64 24.5 (a tree over all threads) and 18.7.
constexpr int RED_THREADS = 256, RED_WARPS = RED_THREADS / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

template <bool MIXED>
__global__ void __launch_bounds__(RED_THREADS, 4) k_reduce_energy(DevState s, PairTable pt, int64_t chunk,
                                                                  double* __restrict__ partials,
                                                                  unsigned* __restrict__ finished,
                                                                  double* __restrict__ out8) {
    __shared__ double sh[RED_WARPS][8];
    __shared__ bool last;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t n = s.n;
    const int64_t lo = blockIdx.x * chunk;
    const int64_t hi = lo + chunk < n ? lo + chunk : n;
    double ke = 0.0;
    std::conditional_t<MIXED, FloatSum, DoubleSum> f[8];  // PE, the six of W, one left empty
    for (int64_t i = lo + threadIdx.x; i < hi; i += RED_THREADS) {
        const double vx = s.vx[i], vy = s.vy[i], vz = s.vz[i];
        if (pt.nsp == 1) ke = fma(vx, vx, fma(vy, vy, fma(vz, vz, ke)));
        else ke += 0.5 * pt.mass[s.species[i]] * (vx * vx + vy * vy + vz * vz);
        if constexpr (MIXED) {
            f[0].add(s.pe_atom_f[i]);
#pragma unroll
            for (int c = 0; c < 6; ++c) f[1 + c].add(s.vir_atom_f[c * n + i]);
        } else {
            f[0].add(s.pe_atom_d[i]);
#pragma unroll
            for (int c = 0; c < 6; ++c) f[1 + c].add(s.vir_atom_d[c * n + i]);
        }
    }
    if (pt.nsp == 1) ke *= 0.5 * pt.mass[0];
    // half of the columns to each half of the lanes, three times, then the four lanes of a column
#pragma unroll
    for (int o = 16, m = 4; m > 0; o >>= 1, m >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < m; ++k) {
            const auto give = up ? f[k] : f[k + m];
            if (up) f[k] = f[k + m];
            f[k].add(lane_xor(give, o));
        }
    }
    f[0].add(lane_xor(f[0], 2));
    f[0].add(lane_xor(f[0], 1));
    const int c = lane >> 2;  // this lane's column
    const double t = f[0].get();  // (shares beyond FP32's range come with a force error, so FloatSum suffices)
    ke = warp_sum(ke);
    if ((lane & 3) == 0 && c < 7) sh[warp][c == 0 ? 0 : 1 + c] = t;
    if (lane == 0) sh[warp][1] = ke;
    __syncthreads();
    if (threadIdx.x < 8) {
        double v = 0.0;
#pragma unroll
        for (int w = 0; w < RED_WARPS; ++w) v += sh[w][threadIdx.x];
        __stcg(partials + blockIdx.x * 8 + threadIdx.x, v);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(finished, gridDim.x - 1) == gridDim.x - 1;  // (back to 0 for the next launch)
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (int b = threadIdx.x >> 3; b < (int)gridDim.x; b += RED_THREADS / 8)
        v += __ldcg(partials + b * 8 + (threadIdx.x & 7));
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    if (lane < 8) sh[warp][lane] = v;
    __syncthreads();
    if (threadIdx.x < 8) {
        double u = 0.0;
#pragma unroll
        for (int w = 0; w < RED_WARPS; ++w) u += sh[w][threadIdx.x];
        out8[threadIdx.x] = u;
    }
}

void launch_reduce_energy(const DevState& s, const PairTable& pt, int mixed, double* partials, unsigned* finished,
                          int nparts, double* out8, cudaStream_t st) {
    const int64_t want = (s.n + RED_THREADS - 1) / RED_THREADS;  // small systems: an atom per thread
    const int parts = (int)std::max<int64_t>(1, std::min<int64_t>(nparts, want));
    const int64_t chunk = std::max<int64_t>(1, (s.n + parts - 1) / parts);
    (mixed ? k_reduce_energy<true> : k_reduce_energy<false>)<<<parts, RED_THREADS, 0, st>>>(s, pt, chunk, partials,
                                                                                       finished, out8);
}

// ---------------------------------------------------------------- state I/O
__global__ void k_set_state(DevState s, Geometry g, const double* __restrict__ pos, const double* __restrict__ vel,
                            const int32_t* __restrict__ species, int nsp) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    double q[6] = {pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], vel ? vel[3 * i] : 0.0, vel ? vel[3 * i + 1] : 0.0,
                   vel ? vel[3 * i + 2] : 0.0};
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (!isfinite(q[k])) {  // refused by md_set_state; kept finite meanwhile
            atomicOr(s.err, 0x40000000u);
            q[k] = 0.0;
        }
    // below -L or at 2 L and beyond, by the upper words (a position just above -L counts too): k_map_far
    bool far = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int h = __double2hiint(q[d]), hL = __double2hiint(g.L[d]);
        far |= h >= 0 ? h >= hL + (1 << 20) : (h & 0x7fffffff) >= hL;
    }
    if (far) atomicOr(s.err, 0x20000000u);
    s.x[i] = q[0];
    s.y[i] = q[1];
    s.z[i] = q[2];
    s.vx[i] = q[3];
    s.vy[i] = q[4];
    s.vz[i] = q[5];
    s.ix[i] = 0;
    s.iy[i] = 0;
    s.iz[i] = 0;
    int sp = species ? species[i] : 0;
    if (sp < 0 || sp >= nsp) {
        atomicOr(s.err, 0x80000000u);
        sp = 0;
    }
    s.species[i] = sp;
    s.orig[i] = (int32_t)i;
}

void launch_set_state(const DevState& s, const Geometry& g, const double* pos, const double* vel, const int32_t* species, int nsp,
                      cudaStream_t st) {
    if (s.n == 0) return;
    int bs = 256;
    k_set_state<<<(unsigned)((s.n + bs - 1) / bs), bs, 0, st>>>(s, g, pos, vel, species, nsp);
}

__global__ void k_get_state(DevState s, double* __restrict__ pos, double* __restrict__ vel,
                            int32_t* __restrict__ image) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int64_t o = s.orig[i];
    if (pos) {
        pos[3 * o] = s.x[i];
        pos[3 * o + 1] = s.y[i];
        pos[3 * o + 2] = s.z[i];
    }
    if (vel) {
        vel[3 * o] = s.vx[i];
        vel[3 * o + 1] = s.vy[i];
        vel[3 * o + 2] = s.vz[i];
    }
    if (image) {
        image[3 * o] = s.ix[i];
        image[3 * o + 1] = s.iy[i];
        image[3 * o + 2] = s.iz[i];
    }
}

void launch_get_state(const DevState& s, double* pos, double* vel, int32_t* image, cudaStream_t st) {
    if (s.n == 0) return;
    int bs = 256;
    k_get_state<<<(unsigned)((s.n + bs - 1) / bs), bs, 0, st>>>(s, pos, vel, image);
}

__global__ void k_forces_out(DevState s, int mixed, double* __restrict__ out) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    const int64_t o = s.orig[i];
    const int64_t n = s.n;
    out[3 * o] = force_of(s, mixed, i);
    out[3 * o + 1] = force_of(s, mixed, n + i);
    out[3 * o + 2] = force_of(s, mixed, 2 * n + i);
}

void launch_forces_out(const DevState& s, int mixed, double* f_out, cudaStream_t st) {
    if (s.n == 0) return;
    int bs = 256;
    k_forces_out<<<(unsigned)((s.n + bs - 1) / bs), bs, 0, st>>>(s, mixed, f_out);
}

__global__ void k_cells_out(DevState s, Geometry g, int32_t* __restrict__ cells) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s.n) return;
    int cx, cy, cz;
    cell_coords(g, s.cell_of[i], cx, cy, cz);
    cells[s.orig[i]] = cx + g.nc[0] * (cy + g.nc[1] * cz);
}

void launch_cells_out(const DevState& s, const Geometry& g, int32_t* cells, cudaStream_t st) {
    if (s.n == 0) return;
    int bs = 256;
    k_cells_out<<<(unsigned)((s.n + bs - 1) / bs), bs, 0, st>>>(s, g, cells);
}

}  // namespace mdgb
