// api_batch.cu - C ABI of ensembles of independent systems (include/mdgb_batch.h).
//
// Every call that advances or evaluates the ensemble is one persistent launch of
// k_ensemble_run over a work table of all systems (k_batch.cu): systems of at most
// one_cta_max atoms (or with too small a box for 2x2x2-cell blocks) are one task each, run
// by one CTA for the whole call, or, where that would take longer than a CTA's share of the
// work, in phases of tasks; larger ones are split into phases of block and chunk tasks
// that any CTA may take.  The launch is captured into a CUDA graph per (steps, flags),
// together with the resets of its scheduler words, and replayed.
#include "mdgb.h"
#include "mdgb_batch.h"
#include "mdgb_batch_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

using namespace mdgb;

namespace {

constexpr int NBUCKET = 5;  // one-CTA systems: [.., 512), [512, 1024), [1024, 2048), [2048, 4096), [4096, 8192]
const int BUCKET_HI[NBUCKET] = {512, 1024, 2048, 4096, BATCH_MAX_ATOMS + 1};
constexpr long long DEFAULT_BUDGET = 1LL << 34;  // cycles without work before a CTA gives up (~9 s)
constexpr int DEFAULT_ONE_CTA_MAX = 2048;
constexpr int ENS_SHARE_CTAS = 2;  // CTAs per SM that a launch usually has

int bucket_of(int64_t n) {
    for (int k = 0; k < NBUCKET; ++k)
        if (n < BUCKET_HI[k]) return k;
    return -1;
}

}  // namespace

struct md_batch {
    int device = 0;
    int sms = 0;
    cudaStream_t stream = nullptr;
    cudaStream_t cap_stream = nullptr;  // capture only records; the legacy stream cannot capture
    int nsys = 0;
    std::vector<int64_t> n, a0;
    std::vector<double> box;  // 3 per system
    double r_cut = 0, skin = 0, dt = 0;
    double eps = 1, sigma = 1, mass = 1;
    PairTable pt{};
    int64_t ntot = 0;
    BatchState st{};
    EnsArrays ea{};
    double *d_pe = nullptr, *d_ke = nullptr;
    double* d_aos = nullptr;  // N_total x 3 staging for AoS input/output
    int32_t* d_sys_of = nullptr;  // system of each atom (output wrap)
    double* d_box = nullptr;      // 3 per system
    // launch shape (md_batch_autotune may change it)
    int threads = 256;
    int one_cta_max = DEFAULT_ONE_CTA_MAX;
    int R[NBUCKET] = {1, 1, 1, 1, 1};
    // the work table for the current shape
    std::vector<int> path;  // 0: one CTA, 1: block tasks
    std::vector<BatchSys> one;
    std::vector<EnsBlockSys> blk;
    std::vector<EnsEntry> ent;
    BatchSys* d_one = nullptr;
    EnsBlockSys* d_blk = nullptr;
    EnsEntry* d_ent = nullptr;
    unsigned long long* d_ctl_init = nullptr;
    int64_t ncell_blk = 0;  // cells of the block systems
    int nmax = 0, cmax = 0, tile_slots = 0, per_sm = 0, grid = 0;
    size_t smem = 0;
    // test hook: a held entry and a budget (launched without a graph)
    int hold = -1;
    long long budget = DEFAULT_BUDGET;
    bool has_state = false, have_forces = false;
    cudaGraphExec_t gexec = nullptr;
    int g_steps = -1, g_flags = -1;
    std::vector<void*> allocs;
    char msg[512] = "";
};

namespace {

int bfail(md_batch* b, int code, const char* fmt, ...) {
    if (b) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(b->msg, sizeof(b->msg), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define BCK(call)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) return bfail(b, MD_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
    } while (0)

template <typename T>
int balloc(md_batch* b, T** p, size_t count) {
    *p = nullptr;
    void* q = nullptr;
    BCK(cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T)));
    b->allocs.push_back(q);
    *p = static_cast<T*>(q);
    return MD_OK;
}

// Geometry of one one-CTA system with cells at least r_cut / R wide (at most 16 per side).
BatchSys make_sys(const md_batch* b, int k, int R) {
    BatchSys y{};
    y.a0 = b->a0[k];
    y.id = k;
    y.n = (int)b->n[k];
    y.R = R;
    y.ncell = 1;
    for (int d = 0; d < 3; ++d) {
        const double L = b->box[3 * k + d];
        int nc = (int)std::floor(L * R / (b->r_cut * (1.0 + 1e-12)));
        nc = std::max(1, std::min(nc, 16));
        y.nc[d] = nc;
        y.L[d] = L;
        y.w[d] = L / nc;
        y.inv_w[d] = nc / L;
        y.wf[d] = (float)y.w[d];
        y.ncell *= nc;
    }
    return y;
}

// Block-task geometry: per side the largest even number of cells at least r_cut + skin
// wide (at most 1024).  False if some side has fewer than 6: with 4 the tile would be the
// whole box, with cells up to 3/2 (r_cut + skin) wide and about 3 times the atoms of the
// narrowest ones, which would set every CTA's shared memory.
bool make_blk(const md_batch* b, int k, EnsBlockSys& y) {
    y = EnsBlockSys{};
    y.a0 = b->a0[k];
    y.id = k;
    y.n = (int)b->n[k];
    y.ncell = 1;
    for (int d = 0; d < 3; ++d) {
        const double L = b->box[3 * k + d];
        int nc = (int)std::min(std::floor(L / ((b->r_cut + b->skin) * (1.0 + 1e-12))), 1024.0);
        nc -= nc % 2;
        if (nc < 6) return false;
        y.nc[d] = nc;
        y.nb[d] = nc / 2;
        y.L[d] = L;
        y.w[d] = L / nc;
        y.inv_w[d] = nc / L;
        for (int t = 0; t < 4; ++t) y.off[d][t] = (float)((t - 1.5) * y.w[d]);
        y.ncell *= nc;
    }
    y.nblock = y.nb[0] * y.nb[1] * y.nb[2];
    return true;
}

// Tile slots a block task of system y may need: 64 cells of up to 1.6 times the mean
// occupancy plus a margin.
int tile_need(const EnsBlockSys& y) {
    const double rho = y.n / (y.L[0] * y.L[1] * y.L[2]);
    return 64 * ((int)std::ceil(1.6 * rho * y.w[0] * y.w[1] * y.w[2]) + 4);
}

bool is_block(const md_batch* b, int k) {
    EnsBlockSys y;
    return b->n[k] > 0 && make_blk(b, k, y) && (b->n[k] > b->one_cta_max || b->n[k] > BATCH_MAX_ATOMS);
}

void drop_graph(md_batch* b) {
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    b->gexec = nullptr;
    b->g_steps = b->g_flags = -1;
}

// Work table, geometry and launch shape for the current threads / one_cta_max / R; the
// device arrays were sized at create for the largest table (every system an entry, every
// blockable system a block system).
int build_table(md_batch* b) {
    drop_graph(b);
    b->path.assign(b->nsys, 0);
    b->one.clear();
    b->blk.clear();
    b->ent.clear();
    b->nmax = b->cmax = 0;
    b->ncell_blk = 0;
    int tile = 0;
    std::vector<int> order(b->nsys);
    for (int k = 0; k < b->nsys; ++k) order[k] = k;
    // the longest tasks first: one-CTA systems by size, then block systems by size
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return b->n[x] > b->n[y]; });
    // A one-CTA system of more than half of a CTA's share of all atoms is shared out as tasks (an
    // atom costs about the same on every path), if that makes more than one.  128 systems of 273 to
    // 32,684 atoms, ten steps, forces and energies: 11.2 ms when the 4,264 atoms of the largest one-CTA
    // system set the length of the launch, 6.0 with it and 29 others shared out; 8 systems of up
    // to 2,000 atoms 2.4 and 1.3 ms.
    const int64_t share = b->ntot / std::max(1, ENS_SHARE_CTAS * b->sms) / 2;
    int64_t s0 = 0;
    std::vector<EnsEntry> e_one, e_shared, e_blk;
    for (int k : order) {
        if (b->n[k] == 0) continue;
        if (is_block(b, k)) {
            EnsBlockSys y;
            make_blk(b, k, y);
            y.c0 = b->ncell_blk;
            y.s0 = b->ncell_blk + (int64_t)b->blk.size();
            b->ncell_blk += y.ncell;
            tile = std::max(tile, tile_need(y));
            e_blk.push_back(EnsEntry{1, (int)b->blk.size(), (y.n + ENS_ATOM_CHUNK - 1) / ENS_ATOM_CHUNK,
                                     (y.ncell + ENS_CELL_CHUNK - 1) / ENS_CELL_CHUNK, y.nblock});
            b->blk.push_back(y);
            b->path[k] = 1;
        } else {
            if (b->n[k] > BATCH_MAX_ATOMS)
                return bfail(b, MD_ERR_BOX_TOO_SMALL, "system %d: %lld atoms in a box of fewer than 6 (r_cut + skin) per side",
                             k, (long long)b->n[k]);
            BatchSys y1 = make_sys(b, k, b->R[bucket_of(b->n[k])]);
            if (y1.ncell > BATCH_MAX_CELLS) return bfail(b, MD_ERR_CELL_OVERFLOW, "system %d: too many cells", k);
            b->nmax = std::max(b->nmax, y1.n);
            b->cmax = std::max(b->cmax, y1.ncell);
            if (y1.n > share && y1.n > ENS_SHARED_CHUNK) {
                y1.s0 = s0;
                s0 += y1.ncell + 1;
                e_shared.push_back(
                    EnsEntry{2, (int)b->one.size(), (y1.n + ENS_SHARED_CHUNK - 1) / ENS_SHARED_CHUNK, 0, 0});
            } else {
                e_one.push_back(EnsEntry{0, (int)b->one.size(), 0, 0, 0});
            }
            b->one.push_back(y1);
        }
    }
    b->nmax = (b->nmax + 7) & ~7;
    b->ent = e_shared;
    b->ent.insert(b->ent.end(), e_one.begin(), e_one.end());
    b->ent.insert(b->ent.end(), e_blk.begin(), e_blk.end());
    // shared memory: the larger of the one-CTA layout and the tile; the tile takes what is left
    size_t smem = b->one.empty() ? 0 : batch_smem_bytes(b->nmax, b->cmax);
    if (!b->blk.empty()) smem = std::max(smem, std::max(ens_tile_smem_bytes(tile), ens_list_smem(tile)));
    smem = (smem + 15) & ~(size_t)15;
    int optin = 0;
    BCK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, b->device));
    if (smem + 8192 > (size_t)optin)
        return bfail(b, MD_ERR_CELL_OVERFLOW, "an ensemble task needs %zu B of shared memory", smem);
    b->smem = smem;
    b->tile_slots = (int)(smem / sizeof(float4)) - 1;
    b->per_sm = ensemble_ctas_per_sm(b->threads, smem);
    if (b->per_sm < 1) return bfail(b, MD_ERR_CUDA, "the ensemble kernel does not fit an SM at %d threads", b->threads);
    b->grid = b->per_sm * b->sms;
    // initial scheduler words: one-CTA systems at their task, the others at START
    std::vector<unsigned long long> init(b->ent.size(), 0ull);
    for (size_t e = 0; e < b->ent.size(); ++e)
        if (b->ent[e].kind != 0) init[e] = (unsigned long long)ENS_START << 32;
    // the block systems' lists and coordinates belong to the old table
    if (b->ea.valid) BCK(cudaMemsetAsync(b->ea.valid, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream));
    if (b->ea.rebuild) BCK(cudaMemsetAsync(b->ea.rebuild, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream));
    if (!b->ent.empty()) {
        BCK(cudaMemcpy(b->d_ent, b->ent.data(), sizeof(EnsEntry) * b->ent.size(), cudaMemcpyHostToDevice));
        BCK(cudaMemcpy(b->d_ctl_init, init.data(), sizeof(unsigned long long) * init.size(), cudaMemcpyHostToDevice));
    }
    if (!b->one.empty()) BCK(cudaMemcpy(b->d_one, b->one.data(), sizeof(BatchSys) * b->one.size(), cudaMemcpyHostToDevice));
    if (!b->blk.empty())
        BCK(cudaMemcpy(b->d_blk, b->blk.data(), sizeof(EnsBlockSys) * b->blk.size(), cudaMemcpyHostToDevice));
    return MD_OK;
}

// Reset the scheduler words (and the block systems' cell counts) and launch, on stream s.
int enqueue_ensemble(md_batch* b, int n_steps, int flags, cudaStream_t s) {
    const int nent = (int)b->ent.size();
    if (nent == 0) return MD_OK;
    BCK(cudaMemcpyAsync(b->ea.ctl, b->d_ctl_init, sizeof(unsigned long long) * nent, cudaMemcpyDeviceToDevice, s));
    BCK(cudaMemsetAsync(b->ea.done, 0, sizeof(int32_t) * nent, s));
    BCK(cudaMemsetAsync(b->ea.g_done, 0, sizeof(int32_t), s));
    if (b->ncell_blk > 0) BCK(cudaMemsetAsync(b->ea.count, 0, sizeof(int32_t) * b->ncell_blk, s));
    if (b->hold >= 0 && b->hold < nent) {
        const unsigned long long w = (unsigned long long)ENS_HOLD << 32;
        BCK(cudaMemcpyAsync(b->ea.ctl + b->hold, &w, sizeof(w), cudaMemcpyHostToDevice, s));
        BCK(cudaStreamSynchronize(s));  // w lives on this stack frame
    }
    EnsArrays ea = b->ea;
    ea.budget = b->budget;
    launch_ensemble(b->d_ent, nent, b->d_one, b->d_blk, b->st, ea, b->pt, n_steps, flags, b->dt, b->threads, b->grid,
                    b->nmax, b->cmax, b->tile_slots, b->smem, b->d_pe, b->d_ke, s);
    BCK(cudaGetLastError());
    return MD_OK;
}

int run_ensemble(md_batch* b, int n_steps, int flags) {
    if (b->ent.empty()) return MD_OK;
    if (b->hold >= 0 || b->budget != DEFAULT_BUDGET) {  // the test hook: a direct launch
        drop_graph(b);
        return enqueue_ensemble(b, n_steps, flags, b->stream);
    }
    if (!(b->gexec && b->g_steps == n_steps && b->g_flags == flags)) {
        drop_graph(b);
        cudaGraph_t g = nullptr;
        BCK(cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal));
        const int rc = enqueue_ensemble(b, n_steps, flags, b->cap_stream);
        const cudaError_t ec = cudaStreamEndCapture(b->cap_stream, &g);
        if (rc) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        if (ec != cudaSuccess) return bfail(b, MD_ERR_CUDA, "graph capture: %s", cudaGetErrorString(ec));
        cudaError_t e = cudaGraphInstantiate(&b->gexec, g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return bfail(b, MD_ERR_CUDA, "graph instantiate: %s", cudaGetErrorString(e));
        b->g_steps = n_steps;
        b->g_flags = flags;
    }
    BCK(cudaGraphLaunch(b->gexec, b->stream));
    return MD_OK;
}

__global__ void k_aos_in(int64_t ntot, const double* __restrict__ pos, const double* __restrict__ vel,
                         const int32_t* __restrict__ sp, BatchState st) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ntot) return;
    st.x[i] = pos[3 * i];
    st.y[i] = pos[3 * i + 1];
    st.z[i] = pos[3 * i + 2];
    st.vx[i] = vel[3 * i];
    st.vy[i] = vel[3 * i + 1];
    st.vz[i] = vel[3 * i + 2];
    st.ix[i] = st.iy[i] = st.iz[i] = 0;
    st.species[i] = sp ? sp[i] : 0;
}

// One coordinate wrapped into [0, L) (one box length at most, as the binning does) and its
// image counter: positions of block systems are wrapped only when they are binned.
__device__ __forceinline__ void wrap_out(double& x, int32_t& img, double L) {
    if (x >= L) {
        x -= L;
        img += 1;
    } else if (x < 0.0) {
        x += L;
        img -= 1;
    }
}

__global__ void k_aos_out(int64_t ntot, BatchState st, const int32_t* __restrict__ sys_of,
                          const double* __restrict__ box, int what, double* __restrict__ out,
                          int32_t* __restrict__ img) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= ntot) return;
    if (what == 0 || what == 3) {
        const double* B = box + 3 * (int64_t)sys_of[i];
        double x = st.x[i], y = st.y[i], z = st.z[i];
        int32_t ix = st.ix[i], iy = st.iy[i], iz = st.iz[i];
        wrap_out(x, ix, B[0]);
        wrap_out(y, iy, B[1]);
        wrap_out(z, iz, B[2]);
        if (what == 0) {
            out[3 * i] = x;
            out[3 * i + 1] = y;
            out[3 * i + 2] = z;
        } else {
            img[3 * i] = ix;
            img[3 * i + 1] = iy;
            img[3 * i + 2] = iz;
        }
    } else if (what == 1) {
        out[3 * i] = st.vx[i];
        out[3 * i + 1] = st.vy[i];
        out[3 * i + 2] = st.vz[i];
    } else if (what == 2) {
        const double q = 2.3283064365386963e-10;  // 2^-32
        out[3 * i] = (double)st.fq[i] * q;
        out[3 * i + 1] = (double)st.fq[st.ntot + i] * q;
        out[3 * i + 2] = (double)st.fq[2 * st.ntot + i] * q;
    }
}

int check_batch_err(md_batch* b) {
    uint32_t e = 0;
    BCK(cudaMemcpy(&e, b->st.err, sizeof(uint32_t), cudaMemcpyDeviceToHost));
    if (!e) return MD_OK;
    cudaMemset(b->st.err, 0, sizeof(uint32_t));
    cudaMemsetAsync(b->ea.valid, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream);
    cudaStreamSynchronize(b->stream);
    b->have_forces = false;
    if (e & ERR_TIMEOUT)
        return bfail(b, MD_ERR_TIMEOUT, "a CTA of the ensemble launch found no work for its whole wait budget");
    if (e & ERR_NONFINITE) return bfail(b, MD_ERR_NONFINITE, "non-finite force or coordinate");
    if (e & ERR_ESCAPE) return bfail(b, MD_ERR_NONFINITE, "an atom moved more than one box length in a step");
    if (e & ERR_TILE_OVERFLOW) return bfail(b, MD_ERR_CELL_OVERFLOW, "a cell neighbourhood exceeded shared memory");
    if (e & ERR_LIST_OVERFLOW) return bfail(b, MD_ERR_LIST_OVERFLOW, "a neighbour list exceeded its capacity");
    return bfail(b, MD_ERR_CUDA, "device error 0x%x", e);
}

// Time 10 steps of the whole ensemble with the current shape (warm-up step first), with the
// state saved before and restored after.
struct Snapshot {
    double* d = nullptr;
    int32_t* i = nullptr;
    long long* f = nullptr;
};

void snap(md_batch* b, Snapshot& sn, bool restore) {
    const size_t n = (size_t)b->ntot;
    double* D[6] = {b->st.x, b->st.y, b->st.z, b->st.vx, b->st.vy, b->st.vz};
    int32_t* I[3] = {b->st.ix, b->st.iy, b->st.iz};
    for (int c = 0; c < 6; ++c)
        cudaMemcpyAsync(restore ? D[c] : sn.d + c * n, restore ? sn.d + c * n : D[c], sizeof(double) * n,
                        cudaMemcpyDeviceToDevice, b->stream);
    for (int c = 0; c < 3; ++c)
        cudaMemcpyAsync(restore ? I[c] : sn.i + c * n, restore ? sn.i + c * n : I[c], sizeof(int32_t) * n,
                        cudaMemcpyDeviceToDevice, b->stream);
    cudaMemcpyAsync(restore ? b->st.fq : sn.f, restore ? sn.f : b->st.fq, sizeof(long long) * 3 * n,
                    cudaMemcpyDeviceToDevice, b->stream);
}

float time_shape(md_batch* b, Snapshot& sn, cudaEvent_t e0, cudaEvent_t e1) {
    if (build_table(b)) return 1e30f;
    if (enqueue_ensemble(b, 1, 0, b->stream)) return 1e30f;
    cudaEventRecord(e0, b->stream);
    if (enqueue_ensemble(b, 10, BATCH_HAVE_FORCES, b->stream)) return 1e30f;
    cudaEventRecord(e1, b->stream);
    if (cudaEventSynchronize(e1) != cudaSuccess) return 1e30f;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    snap(b, sn, true);
    cudaMemsetAsync(b->ea.valid, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream);
    cudaMemsetAsync(b->ea.rebuild, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream);
    uint32_t e = 0;
    cudaMemcpy(&e, b->st.err, sizeof(uint32_t), cudaMemcpyDeviceToHost);
    if (e) {
        cudaMemset(b->st.err, 0, sizeof(uint32_t));
        return 1e30f;
    }
    return ms;
}

}  // namespace

extern "C" {

int md_batch_create(int32_t n_systems, const int64_t* n_atoms, const double* boxes, double r_cut, double skin,
                    const md_params* p, md_batch** out) {
    if (!out) return MD_ERR_ARG;
    *out = nullptr;
    if (n_systems < 1 || !n_atoms || !boxes || !p || !(r_cut > 0.0) || !(skin >= 0.0)) return MD_ERR_ARG;
    if (p->n_species != 1 || p->precision != MD_MIXED || !p->eps || !p->sigma || !p->mass || !(p->dt > 0.0))
        return MD_ERR_ARG;
    md_batch* b = new md_batch();
    auto bail = [&](int code) {
        md_batch_destroy(b);
        return code;
    };
    cudaGetDevice(&b->device);
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->device);
    b->stream = static_cast<cudaStream_t>(p->stream);
    if (cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess) return bail(MD_ERR_CUDA);
    b->nsys = n_systems;
    b->r_cut = r_cut;
    b->skin = skin;
    b->dt = p->dt;
    b->eps = p->eps[0];
    b->sigma = p->sigma[0];
    b->mass = p->mass[0];
    // pair constants as the main path builds them (one species)
    b->pt.nsp = 1;
    b->pt.sig2_f[0] = (float)(b->sigma * b->sigma);
    b->pt.c48_f[0] = (float)(48.0 * b->eps * 2048.0);
    b->pt.c24_f[0] = (float)(24.0 * b->eps * 2048.0);
    b->pt.c4_f[0] = (float)(4.0 * b->eps);
    b->pt.rc2_f[0] = (float)(r_cut * r_cut);
    b->pt.rc2_d[0] = r_cut * r_cut;
    b->pt.mass[0] = b->mass;
    b->pt.hdtm[0] = (0.5 * p->dt) / b->mass;
    b->pt.hdtm_q[0] = b->pt.hdtm[0] * 0x1p-32;
    init_batch_kernels();
    b->n.assign(n_atoms, n_atoms + n_systems);
    b->box.assign(boxes, boxes + 3 * n_systems);
    b->a0.resize(n_systems);
    int64_t cells_max = 0, nblk_max = 0, starts_max = 0;
    double band = 0.0, rho_max = 0.0;
    for (int k = 0; k < n_systems; ++k) {
        if (b->n[k] < 0 || b->n[k] > 0x7fffffffLL) return bail(MD_ERR_ARG);
        b->a0[k] = b->ntot;
        b->ntot += b->n[k];
        for (int d = 0; d < 3; ++d)
            if (!(boxes[3 * k + d] >= 2.0 * r_cut) || !std::isfinite(boxes[3 * k + d])) {
                bfail(b, MD_ERR_BOX_TOO_SMALL, "system %d: box side %g < 2 r_cut", k, boxes[3 * k + d]);
                return bail(MD_ERR_BOX_TOO_SMALL);
            }
        // FP64 decision band: the widest any system needs, on either path and cell divisor
        for (int R = 1; R <= 2; ++R) {
            const BatchSys y = make_sys(b, k, R);
            band = std::max(band, cell_frame_cut_band(std::max(y.w[0], std::max(y.w[1], y.w[2])), R, r_cut));
            if (R == 2 && b->n[k] > ENS_SHARED_CHUNK && b->n[k] <= BATCH_MAX_ATOMS) starts_max += y.ncell + 1;
        }
        EnsBlockSys y;
        if (make_blk(b, k, y)) {
            band = std::max(band,
                            tile_frame_cut_band(std::max(y.w[0], std::max(y.w[1], y.w[2])), 0.5 * skin, r_cut));
            cells_max += y.ncell;
            nblk_max += 1;
            rho_max = std::max(rho_max, b->n[k] / (y.L[0] * y.L[1] * y.L[2]));
        }
    }
    b->pt.cut_band = (float)band;
    set_band_thresholds(b->pt);
    int rc;
    BatchState& st = b->st;
    EnsArrays& ea = b->ea;
    st.ntot = b->ntot;
    // Verlet lists of the block systems: 1.5 times the mean count in the list sphere at the
    // densest such system, plus 32, in chunks of 8 (a longer list reports MD_ERR_LIST_OVERFLOW)
    const double rl = r_cut + skin;
    ea.list_chunks = (int)((std::ceil(1.5 * 4.0 / 3.0 * M_PI * rl * rl * rl * rho_max) + 32 + 7) / 8);
    ea.rl2 = rl * rl;
    ea.rl2_lo = (float)(ea.rl2 * (1.0 - 1e-4));
    ea.rl2_hi = (float)(ea.rl2 * (1.0 + 1e-4));
    ea.lim2_f = (float)(0.25 * skin * skin);
    const size_t nt = (size_t)b->ntot, ns = (size_t)n_systems;
    if ((rc = balloc(b, &st.x, nt)) || (rc = balloc(b, &st.y, nt)) || (rc = balloc(b, &st.z, nt)) ||
        (rc = balloc(b, &st.vx, nt)) || (rc = balloc(b, &st.vy, nt)) || (rc = balloc(b, &st.vz, nt)) ||
        (rc = balloc(b, &st.ix, nt)) || (rc = balloc(b, &st.iy, nt)) || (rc = balloc(b, &st.iz, nt)) ||
        (rc = balloc(b, &st.species, nt)) || (rc = balloc(b, &st.fq, 3 * nt)) || (rc = balloc(b, &st.err, 1)) ||
        (rc = balloc(b, &b->d_pe, ns)) || (rc = balloc(b, &b->d_ke, ns)) || (rc = balloc(b, &b->d_aos, 3 * nt)) ||
        (rc = balloc(b, &ea.xa, nt)) || (rc = balloc(b, &ea.ya, nt)) || (rc = balloc(b, &ea.za, nt)) ||
        (rc = balloc(b, &ea.cell_of, nt)) || (rc = balloc(b, &ea.perm_u, nt)) || (rc = balloc(b, &ea.perm_s, nt)) ||
        (rc = balloc(b, &ea.xs, nt)) || (rc = balloc(b, &ea.xsb, nt)) ||
        (rc = balloc(b, &ea.xs_ref, nt)) || (rc = balloc(b, &ea.nl_cnt, nt)) ||
        (rc = balloc(b, &ea.nl, nt * (size_t)ea.list_chunks)) || (rc = balloc(b, &ea.rebuild, ns)) ||
        (rc = balloc(b, &ea.valid, ns)) || (rc = balloc(b, &b->d_sys_of, nt)) || (rc = balloc(b, &b->d_box, 3 * ns)) ||
        (rc = balloc(b, &ea.pe_atom, nt)) ||
        (rc = balloc(b, &ea.count, (size_t)cells_max)) || (rc = balloc(b, &ea.cursor, (size_t)cells_max)) ||
        (rc = balloc(b, &ea.cstart, (size_t)(cells_max + nblk_max))) ||
        (rc = balloc(b, &ea.cstart1, (size_t)starts_max)) || (rc = balloc(b, &ea.ctl, ns)) ||
        (rc = balloc(b, &ea.done, ns)) || (rc = balloc(b, &ea.g_done, 1)) || (rc = balloc(b, &b->d_ctl_init, ns)) ||
        (rc = balloc(b, &b->d_ent, ns)) || (rc = balloc(b, &b->d_one, ns)) || (rc = balloc(b, &b->d_blk, ns)))
        return bail(rc);
    // slot maps start as valid indices, so that a step that gave up after an error reads
    // only inside its system
    if (cudaMemset(st.err, 0, sizeof(uint32_t)) != cudaSuccess || cudaMemset(b->d_pe, 0, sizeof(double) * ns) ||
        cudaMemset(b->d_ke, 0, sizeof(double) * ns) || cudaMemset(ea.valid, 0, sizeof(int32_t) * ns) ||
        cudaMemset(ea.rebuild, 0, sizeof(int32_t) * ns) || cudaMemset(ea.perm_u, 0, sizeof(int32_t) * nt) ||
        cudaMemset(ea.perm_s, 0, sizeof(int32_t) * nt))
        return bail(MD_ERR_CUDA);
    {
        std::vector<int32_t> sys_of(nt);
        for (int k = 0; k < n_systems; ++k)
            for (int64_t i = 0; i < b->n[k]; ++i) sys_of[b->a0[k] + i] = k;
        if (nt && cudaMemcpy(b->d_sys_of, sys_of.data(), sizeof(int32_t) * nt, cudaMemcpyHostToDevice) != cudaSuccess)
            return bail(MD_ERR_CUDA);
        if (cudaMemcpy(b->d_box, boxes, sizeof(double) * 3 * ns, cudaMemcpyHostToDevice) != cudaSuccess)
            return bail(MD_ERR_CUDA);
    }
    // default launch shape; md_batch_autotune may change it
    if ((rc = build_table(b))) return bail(rc);
    *out = b;
    return MD_OK;
}

int md_batch_set_state(md_batch* b, const double* pos, const double* vel, const int32_t* species, int device_ptrs) {
    if (!b || !pos || !vel) return MD_ERR_ARG;
    const size_t n3 = 3 * (size_t)b->ntot;
    const double *P = pos, *V = vel;
    const int32_t* S = species;
    double* tmp = nullptr;
    int32_t* tsp = nullptr;
    if (!device_ptrs) {
        BCK(cudaMalloc(&tmp, sizeof(double) * 2 * std::max<size_t>(n3, 1)));
        BCK(cudaMemcpy(tmp, pos, sizeof(double) * n3, cudaMemcpyHostToDevice));
        BCK(cudaMemcpy(tmp + n3, vel, sizeof(double) * n3, cudaMemcpyHostToDevice));
        P = tmp;
        V = tmp + n3;
        if (species) {
            BCK(cudaMalloc(&tsp, sizeof(int32_t) * std::max<int64_t>(b->ntot, 1)));
            BCK(cudaMemcpy(tsp, species, sizeof(int32_t) * b->ntot, cudaMemcpyHostToDevice));
            S = tsp;
        }
    }
    if (b->ntot > 0) k_aos_in<<<(unsigned)((b->ntot + 255) / 256), 256, 0, b->stream>>>(b->ntot, P, V, S, b->st);
    BCK(cudaGetLastError());
    BCK(cudaStreamSynchronize(b->stream));
    if (tmp) cudaFree(tmp);
    if (tsp) cudaFree(tsp);
    BCK(cudaMemset(b->st.err, 0, sizeof(uint32_t)));
    BCK(cudaMemsetAsync(b->ea.valid, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream));
    BCK(cudaMemsetAsync(b->ea.rebuild, 0, sizeof(int32_t) * (size_t)b->nsys, b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    b->has_state = true;
    b->have_forces = false;
    return MD_OK;
}

int md_batch_step(md_batch* b, int32_t n_steps) {
    if (!b || n_steps < 0) return MD_ERR_ARG;
    if (!b->has_state) return bfail(b, MD_ERR_STATE, "no state: call md_batch_set_state first");
    if (n_steps == 0) return MD_OK;
    int rc = run_ensemble(b, n_steps, b->have_forces ? BATCH_HAVE_FORCES : 0);
    if (rc) return rc;
    BCK(cudaStreamSynchronize(b->stream));
    if ((rc = check_batch_err(b))) return rc;
    b->have_forces = true;
    return MD_OK;
}

int md_batch_forces(md_batch* b, double* f_out, int device_ptrs) {
    if (!b) return MD_ERR_ARG;
    if (!b->has_state) return bfail(b, MD_ERR_STATE, "no state");
    int rc;
    if (!b->have_forces) {
        if ((rc = run_ensemble(b, 0, 0))) return rc;
        BCK(cudaStreamSynchronize(b->stream));
        if ((rc = check_batch_err(b))) return rc;
        b->have_forces = true;
    }
    if (!f_out) return MD_OK;
    double* dst = device_ptrs ? f_out : b->d_aos;
    if (b->ntot > 0) k_aos_out<<<(unsigned)((b->ntot + 255) / 256), 256, 0, b->stream>>>(b->ntot, b->st, b->d_sys_of, b->d_box, 2,
                                                                           dst, nullptr);
    BCK(cudaGetLastError());
    BCK(cudaStreamSynchronize(b->stream));
    if (!device_ptrs) BCK(cudaMemcpy(f_out, b->d_aos, sizeof(double) * 3 * b->ntot, cudaMemcpyDeviceToHost));
    return MD_OK;
}

int md_batch_energies(md_batch* b, double* pe, double* ke) {
    if (!b || !pe || !ke) return MD_ERR_ARG;
    if (!b->has_state) return bfail(b, MD_ERR_STATE, "no state");
    int rc;
    if ((rc = run_ensemble(b, 0, BATCH_ENERGY))) return rc;
    BCK(cudaMemcpyAsync(pe, b->d_pe, sizeof(double) * b->nsys, cudaMemcpyDeviceToHost, b->stream));
    BCK(cudaMemcpyAsync(ke, b->d_ke, sizeof(double) * b->nsys, cudaMemcpyDeviceToHost, b->stream));
    BCK(cudaStreamSynchronize(b->stream));
    if ((rc = check_batch_err(b))) return rc;
    b->have_forces = true;
    return MD_OK;
}

int md_batch_get_state(md_batch* b, double* pos, double* vel, int32_t* image, int device_ptrs) {
    if (!b) return MD_ERR_ARG;
    if (!b->has_state) return bfail(b, MD_ERR_STATE, "no state");
    double* outs[2] = {pos, vel};
    for (int w = 0; w < 3; ++w) {
        double* o = w < 2 ? outs[w] : nullptr;
        if (w < 2 && !o) continue;
        if (w == 2 && !image) continue;
        double* dst = device_ptrs ? o : b->d_aos;
        int32_t* idst = device_ptrs ? image : reinterpret_cast<int32_t*>(b->d_aos);
        if (b->ntot > 0)
            k_aos_out<<<(unsigned)((b->ntot + 255) / 256), 256, 0, b->stream>>>(b->ntot, b->st, b->d_sys_of, b->d_box,
                                                                                w == 2 ? 3 : w, dst, idst);
        BCK(cudaGetLastError());
        BCK(cudaStreamSynchronize(b->stream));
        if (!device_ptrs) {
            if (w < 2) BCK(cudaMemcpy(o, b->d_aos, sizeof(double) * 3 * b->ntot, cudaMemcpyDeviceToHost));
            else BCK(cudaMemcpy(image, b->d_aos, sizeof(int32_t) * 3 * b->ntot, cudaMemcpyDeviceToHost));
        }
    }
    return MD_OK;
}

int md_batch_layout(md_batch* b, int32_t* path, int32_t* threads, int32_t* cell_range) {
    if (!b) return MD_ERR_ARG;
    for (int k = 0; k < b->nsys; ++k) {
        const bool one = b->path[k] == 0 && b->n[k] > 0;
        if (path) path[k] = b->path[k];
        if (threads) threads[k] = b->threads;
        if (cell_range) cell_range[k] = one ? b->R[bucket_of(b->n[k])] : 1;
    }
    return MD_OK;
}

int md_batch_launch_shape(md_batch* b, int32_t* form, int32_t* ctas_per_sm, int64_t* smem_bytes) {
    if (!b) return MD_ERR_ARG;
    if (form) {
        std::fill(form, form + b->nsys, -1);
        for (const EnsEntry& en : b->ent) form[en.kind == 1 ? b->blk[en.idx].id : b->one[en.idx].id] = en.kind;
    }
    if (ctas_per_sm) *ctas_per_sm = b->per_sm;
    if (smem_bytes) *smem_bytes = (int64_t)b->smem;
    return MD_OK;
}

int md_batch_set_wait_budget(md_batch* b, int64_t budget_cycles, int32_t held_system) {
    if (!b || budget_cycles < 0 || held_system < -1 || held_system >= b->nsys) return MD_ERR_ARG;
    b->budget = budget_cycles == 0 ? DEFAULT_BUDGET : budget_cycles;
    b->hold = -1;
    if (held_system >= 0)
        for (size_t e = 0; e < b->ent.size(); ++e) {
            const EnsEntry& en = b->ent[e];
            const int id = en.kind == 1 ? b->blk[en.idx].id : b->one[en.idx].id;
            if (id == held_system) b->hold = (int)e;
        }
    drop_graph(b);
    return MD_OK;
}

int md_batch_autotune(md_batch* b, const char* cache_path) {
    if (!b) return MD_ERR_ARG;
    if (!b->has_state) return bfail(b, MD_ERR_STATE, "no state: the autotuner times real steps");
    cudaDeviceProp prop;
    BCK(cudaGetDeviceProperties(&prop, b->device));
    bool present[NBUCKET] = {};
    for (int k = 0; k < b->nsys; ++k) {
        const int bu = bucket_of(b->n[k]);
        if (b->n[k] > 0 && bu >= 0) present[bu] = true;
    }
    // a cached shape for this GPU: threads, one-CTA limit and R per bucket
    if (cache_path) {
        FILE* f = std::fopen(cache_path, "r");
        if (f) {
            char buf[4096];
            const size_t len = std::fread(buf, 1, sizeof(buf) - 1, f);
            std::fclose(f);
            buf[len] = 0;
            const std::string s(buf);
            int th = 0, lim = 0, R[NBUCKET] = {0, 0, 0, 0, 0};
            bool ok = s.find(std::string("\"gpu\": \"") + prop.name + "\"") != std::string::npos;
            const size_t at = s.find("\"shape\": [");
            ok = ok && at != std::string::npos &&
                 std::sscanf(s.c_str() + at + 10, "%d, %d, %d, %d, %d, %d, %d", &th, &lim, &R[0], &R[1], &R[2], &R[3],
                             &R[4]) == 7 &&
                 (th == 128 || th == 256 || th == 512) && (lim == 1024 || lim == 2048 || lim == 4096);
            for (int k = 0; k < NBUCKET; ++k) ok = ok && (R[k] == 1 || R[k] == 2);
            if (ok) {
                b->threads = th;
                b->one_cta_max = lim;
                for (int k = 0; k < NBUCKET; ++k) b->R[k] = R[k];
                if (build_table(b) == MD_OK) return MD_OK;
            }
        }
    }
    // time 10 steps per candidate on a copy of the state, restored afterwards: the launch
    // size, then the one-CTA limit, then the cell divisor of each size bucket present
    const size_t n = (size_t)b->ntot;
    Snapshot sn;
    BCK(cudaMalloc(&sn.d, sizeof(double) * 6 * std::max<size_t>(n, 1)));
    BCK(cudaMalloc(&sn.i, sizeof(int32_t) * 3 * std::max<size_t>(n, 1)));
    BCK(cudaMalloc(&sn.f, sizeof(long long) * 3 * std::max<size_t>(n, 1)));
    snap(b, sn, false);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int hold = b->hold;
    const long long budget = b->budget;
    b->hold = -1;
    b->budget = DEFAULT_BUDGET;
    float best = time_shape(b, sn, e0, e1);
    for (int th : {128, 512}) {
        const int keep = b->threads;
        b->threads = th;
        const float ms = time_shape(b, sn, e0, e1);
        if (ms < best) best = ms;
        else b->threads = keep;
    }
    for (int lim : {1024, 4096}) {
        const int keep = b->one_cta_max;
        b->one_cta_max = lim;
        const float ms = time_shape(b, sn, e0, e1);
        if (ms < best) best = ms;
        else b->one_cta_max = keep;
    }
    for (int k = 0; k < NBUCKET; ++k) {
        if (!present[k]) continue;
        b->R[k] = 2;
        const float ms = time_shape(b, sn, e0, e1);
        if (ms < best) best = ms;
        else b->R[k] = 1;
    }
    b->hold = hold;
    b->budget = budget;
    const int rc = build_table(b);
    snap(b, sn, true);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    BCK(cudaStreamSynchronize(b->stream));
    cudaFree(sn.d);
    cudaFree(sn.i);
    cudaFree(sn.f);
    if (rc) return rc;
    BCK(cudaMemset(b->st.err, 0, sizeof(uint32_t)));
    b->have_forces = false;
    if (cache_path) {
        FILE* f = std::fopen(cache_path, "w");
        if (f) {
            std::fprintf(f, "{\"gpu\": \"%s\", \"shape\": [%d, %d, %d, %d, %d, %d, %d]}\n", prop.name, b->threads,
                         b->one_cta_max, b->R[0], b->R[1], b->R[2], b->R[3], b->R[4]);
            std::fclose(f);
        }
    }
    return MD_OK;
}

int md_batch_last_error(md_batch* b, char* buf, int64_t len) {
    if (!b || !buf || len <= 0) return MD_ERR_ARG;
    std::snprintf(buf, (size_t)len, "%s", b->msg);
    return MD_OK;
}

void md_batch_destroy(md_batch* b) {
    if (!b) return;
    if (b->gexec) cudaGraphExecDestroy(b->gexec);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    for (void* p : b->allocs) cudaFree(p);
    delete b;
}

}  // extern "C"
