// Laguerre cell clipping: volumes, first moments and facet areas of every cell, in up
// to three passes per evaluation (the per-cell work is in cell.cuh):
//   pass 1  every cell: clipped by its first candidates (its facets in the previous
//           diagram, else its k nearest seeds) and certified by the security walk;
//           a cell with a possible unseen cutter is re-queued;
//   pass 2  the re-queued cells: the walk clips every seed that cuts;
//   pass 3  FP64 re-clip, with the large polytope capacity, of the cells that failed
//           the FP32 consistency check or overflowed the small capacity.
#include <float.h>
#include <math.h>

#include <string>
#include <vector>

#include "cell.cuh"

namespace sdot {

// carry.cu: the cells a carried certificate certifies; the others go to queue (count cnt)
int launch_carry(const ClipParams& cp, int32_t* queue, int32_t* cnt, int32_t* work, cudaStream_t s);

// A block's warps go through the phases of a cell together (see process_cell). Larger
// blocks keep the instruction cache better, smaller ones wait less for their slowest cell.
// 1, 2, 4, 8 blocks per SM (32 to 4 warps each): first diagram 97^3, whose cells differ
// most, 177, 132, 113, 119 ms; early Newton step 100^3 95, 90, 105, 131 ms; late step 129^3
// (1% of its cells left to these kernels) 17.4, 17.2, 17.3, 17.4 ms; FP64 step 45^3 15.2, 14.0,
// 14.3, 16.4 ms.
constexpr int CLIP_BLOCKS_PER_SM = 4;

// Warps of a full clipping block: as many as shared memory holds polytopes for with
// CLIP_BLOCKS_PER_SM blocks on an SM, and at most 32 warps an SM (64 registers a thread).
template <typename R, class C>
constexpr int clip_warps() {
    return (int)((226u * 1024u / CLIP_BLOCKS_PER_SM - 1024u) / sizeof(Poly<R, C>)) <
                   32 / CLIP_BLOCKS_PER_SM
               ? (int)((226u * 1024u / CLIP_BLOCKS_PER_SM - 1024u) / sizeof(Poly<R, C>))
               : 32 / CLIP_BLOCKS_PER_SM;
}

template <typename R, class C, int MODE>
__global__ void __launch_bounds__(clip_warps<R, C>() * 32, CLIP_BLOCKS_PER_SM)
    clip_kernel(const __grid_constant__ ClipParams cp) {
    __shared__ int64_t first;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const float psimax_glob = top_psimax(cp, lane);
    const float halfLmin = 0.5f * fminf(cp.Lt[0], fminf(cp.Lt[1], cp.Lt[2]));
    const int64_t nwork = cp.nwork_dev ? *cp.nwork_dev : cp.nwork;
    int carried = 0;  // cells certified by a carried certificate
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) first = atomicAdd(cp.work_counter, nwarp);
        __syncthreads();
        const int64_t w = first + warp;
        if (first >= nwork) break;
        carried += process_cell<R, C, MODE>(warp, cp, w < nwork, w, psimax_glob, halfLmin, lane)
                       ? 1
                       : 0;
    }
    if (lane == 0 && carried) atomicAdd(cp.cert_carried, carried);
}

// The same pass over the work items of several contexts in one persistent launch (a
// batch of server jobs): item w of the batch belongs to the job j with
// start[j] <= w < start[j + 1] and is that job's item w - start[j].
struct ClipBatch {
    const ClipParams* jobs;       // njobs entries, device memory
    const int64_t* start;         // njobs + 1 prefix sums of the jobs' nwork
    unsigned long long* counter;  // next batch item
    int njobs;
};

template <typename R, class C, int MODE>
__global__ void __launch_bounds__(clip_warps<R, C>() * 32, CLIP_BLOCKS_PER_SM) clip_batch_kernel(ClipBatch bt) {
    __shared__ long long first;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const long long total = bt.start[bt.njobs];
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) first = (long long)atomicAdd(bt.counter, (unsigned long long)nwarp);
        __syncthreads();
        const long long w = first + warp;
        if (first >= total) break;
        // the last job j with start[j] <= w (jobs without items are skipped)
        int lo = 0, hi = bt.njobs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (bt.start[mid] <= w) lo = mid;
            else hi = mid - 1;
        }
        const ClipParams& cp = bt.jobs[lo];
        const float psimax_glob = top_psimax(cp, lane);
        const float halfLmin = 0.5f * fminf(cp.Lt[0], fminf(cp.Lt[1], cp.Lt[2]));
        process_cell<R, C, MODE>(warp, cp, w < total, (int64_t)(w - bt.start[lo]), psimax_glob,
                                 halfLmin, lane);
    }
}

// ---------------------------------------------------------------------------
// per-evaluation preparation: normalised float positions and the psi pyramid
// ---------------------------------------------------------------------------
// The seeds' grid cells and offsets in them: once per context (its first evaluation).
__global__ void posf_kernel(const Pos4* __restrict__ pos, int64_t N, double inv_a, double hx,
                            double hy, double hz, int Gx, int Gy, int Gz,
                            float4* __restrict__ posf, int32_t* __restrict__ leafc,
                            uint4* __restrict__ ioff) {
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    Pos4 y = pos[s];
    double h[3] = {hx, hy, hz};
    int G[3] = {Gx, Gy, Gz};
    double p[3] = {y.x, y.y, y.z};
    int c[3];
    float off[3];
    uint32_t io[3];
    for (int a = 0; a < 3; a++) {
        int cc = (int)floor(p[a] / h[a]);
        cc = cc < 0 ? 0 : (cc >= G[a] ? G[a] - 1 : cc);
        c[a] = cc;
        double f = p[a] - cc * h[a];
        off[a] = (float)(f * inv_a);
        double fx = floor(f / h[a] * 4294967296.0);
        fx = fx < 0.0 ? 0.0 : (fx > 4294967295.0 ? 4294967295.0 : fx);
        io[a] = (uint32_t)fx;
    }
    posf[s] = make_float4(off[0], off[1], off[2], 0.f);
    leafc[s] = c[0] | (c[1] << 10) | (c[2] << 20);
    ioff[s] = make_uint4(io[0], io[1], io[2], 0u);
}

// Level 0 of the pyramid from the ordered maxima psi_kernel left (0: no seed).
__global__ void leaf_max_kernel(float* __restrict__ psimax, int64_t ncell) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    const uint32_t u = __float_as_uint(psimax[c]);
    psimax[c] = u ? ord2f(u) : -INFINITY;
}

__global__ void level_max_kernel(const float* __restrict__ in, int dx, int dy, int dz,
                                 float* __restrict__ out, int ox, int oy, int oz) {
    int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= (int64_t)ox * oy * oz) return;
    int X = (int)(n % ox), Y = (int)((n / ox) % oy), Z = (int)(n / ((int64_t)ox * oy));
    float m = -INFINITY;
    for (int c = 0; c < 64; c++) {
        int x = 4 * X + (c & 3), y = 4 * Y + ((c >> 2) & 3), z = 4 * Z + (c >> 4);
        if (x < dx && y < dy && z < dz) m = fmaxf(m, in[((int64_t)z * dy + y) * dx + x]);
    }
    out[n] = m;
}

// The pyramid's levels from l on in one block: they are small, and a launch each cost more
// than they do.
__global__ void __launch_bounds__(1024) top_levels_kernel(Pyramid P, int l) {
    for (; l < P.nlev; l++) {
        const float* in = P.psimax + P.off[l - 1];
        float* out = P.psimax + P.off[l];
        const int dx = P.dim[l - 1][0], dy = P.dim[l - 1][1], dz = P.dim[l - 1][2];
        const int ox = P.dim[l][0], oy = P.dim[l][1], oz = P.dim[l][2];
        // 8 lanes a node, 8 children each
        const int part = threadIdx.x & 7;
        for (int n = threadIdx.x >> 3; n < (ox * oy * oz + 3) / 4 * 4; n += blockDim.x >> 3) {
            const int X = n % ox, Y = (n / ox) % oy, Z = n / (ox * oy);
            float m = -INFINITY;
            for (int c = part; c < 64; c += 8) {
                const int x = 4 * X + (c & 3), y = 4 * Y + ((c >> 2) & 3), z = 4 * Z + (c >> 4);
                if (x < dx && y < dy && z < dz) m = fmaxf(m, in[(z * dy + y) * dx + x]);
            }
            for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULLMASK, m, o));
            if (part == 0 && Z < oz) out[n] = m;
        }
        __syncthreads();
    }
}

// What changes with psi, in one pass over the seeds:
//  - psi/a^2 as hi + lo floats;
//  - the upper bound of psi/a^2 over each grid cell (an integer maximum of ordered bits: a
//    clump's grid cell holds hundreds of seeds, which one thread used to scan);
//  - the change of psi since the previous evaluation of the context: the largest and
//    smallest psi - psi_prev in units of a^2 (rounded outward, as order-preserving integers
//    for the atomics: mm[0] the maximum, mm[1] the minimum); psi_prev then takes psi. Only
//    differences of psi shape the diagram, so a carried certificate consumes max - min.
// 2.1 M seeds: 70 us, where three passes, one of which recomputed the grid offsets with six
// FP64 divisions a seed, took 440 us; 38 k clumped seeds 49 -> 6 us.
__global__ void psi_kernel(const double* __restrict__ psi, double* __restrict__ prev, int64_t N,
                           double inv_a2, int Gx, int Gy, const int32_t* __restrict__ leafc,
                           float4* __restrict__ posf, float* __restrict__ pslo,
                           uint32_t* __restrict__ leafmax, uint32_t* __restrict__ mm) {
    float hi = -INFINITY, lo = INFINITY;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double p = psi[i];
        const double dv = (p - prev[i]) * inv_a2;
        hi = fmaxf(hi, __double2float_ru(dv));
        lo = fminf(lo, __double2float_rd(dv));
        prev[i] = p;
        const double q = p * inv_a2;
        const float qh = (float)q;
        posf[i].w = qh;
        pslo[i] = (float)(q - (double)qh);
        const int lc = leafc[i];
        const int64_t leaf =
            ((int64_t)((lc >> 20) & 1023) * Gy + ((lc >> 10) & 1023)) * Gx + (lc & 1023);
        atomicMax(&leafmax[leaf], f2ord(__double2float_ru(q * (1.0 + 1e-15 * (p > 0 ? 1 : -1)))));
    }
    uint32_t h = f2ord(hi), l = f2ord(lo);
    h = __reduce_max_sync(FULLMASK, h);
    l = __reduce_min_sync(FULLMASK, l);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&mm[0], h);
        atomicMin(&mm[1], l);
    }
}

int build_pyramid(DeviceState& d, const double* psi, cudaStream_t s) {
    const int64_t N = d.N;
    uint32_t* mm = reinterpret_cast<uint32_t*>(d.counters + 30);
    Pyramid& P = d.pyr;
    if (!d.posf_valid) {
        posf_kernel<<<(unsigned)((N + 255) / 256), 256, 0, s>>>(
            d.pos, N, 1.0 / d.a, d.grid.h[0], d.grid.h[1], d.grid.h[2], d.grid.G[0], d.grid.G[1],
            d.grid.G[2], d.posf, d.leafc, d.ioff);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        d.posf_valid = 1;
    }
    SDOT_CUDA_TRY(cudaMemsetAsync(mm, 0, 4, s));
    SDOT_CUDA_TRY(cudaMemsetAsync(mm + 1, 0xff, 4, s));
    SDOT_CUDA_TRY(cudaMemsetAsync(P.psimax + P.off[0], 0, (size_t)d.grid.ncell * 4, s));
    const int64_t nb = (N + 255) / 256, most = 8 * (int64_t)num_sms();
    psi_kernel<<<(unsigned)(nb < most ? nb : most), 256, 0, s>>>(
        psi, d.psi_prev, N, 1.0 / (d.a * d.a), d.grid.G[0], d.grid.G[1], d.leafc, d.posf, d.pslo,
        reinterpret_cast<uint32_t*>(P.psimax + P.off[0]), mm);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    leaf_max_kernel<<<(unsigned)((d.grid.ncell + 255) / 256), 256, 0, s>>>(P.psimax + P.off[0],
                                                                          d.grid.ncell);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    int l = 1;
    for (; l < P.nlev; l++) {
        const int64_t n = (int64_t)P.dim[l][0] * P.dim[l][1] * P.dim[l][2];
        if (n <= 4096) break;  // 32 nodes a pass of top_levels_kernel's block
        level_max_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
            P.psimax + P.off[l - 1], P.dim[l - 1][0], P.dim[l - 1][1], P.dim[l - 1][2],
            P.psimax + P.off[l], P.dim[l][0], P.dim[l][1], P.dim[l][2]);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
    }
    if (l < P.nlev) {
        top_levels_kernel<<<1, 1024, 0, s>>>(P, l);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
    }
    return SDOT_OK;
}

// ---------------------------------------------------------------------------
// reductions over the cells
// ---------------------------------------------------------------------------
constexpr int RED_BLOCKS = 256;

__global__ void cell_reduce_kernel(const double* __restrict__ vol, const double* __restrict__ nu,
                                   const uint8_t* __restrict__ status, int64_t N,
                                   double* __restrict__ part) {
    double sv = 0, mr = 0, l2 = 0, mv = INFINITY, ne = 0;
    uint32_t fl = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
        double v = vol[i], g = nu[i] - v;
        sv += v;
        mr = fmax(mr, fabs(g) / nu[i]);
        l2 += g * g;
        mv = fmin(mv, v);
        if (!(v > 0)) ne += 1;
        fl |= status[i];
    }
    __shared__ double sh[6][8];
    for (int o = 16; o > 0; o >>= 1) {
        sv += __shfl_xor_sync(FULLMASK, sv, o);
        mr = fmax(mr, __shfl_xor_sync(FULLMASK, mr, o));
        l2 += __shfl_xor_sync(FULLMASK, l2, o);
        mv = fmin(mv, __shfl_xor_sync(FULLMASK, mv, o));
        ne += __shfl_xor_sync(FULLMASK, ne, o);
        fl |= __shfl_xor_sync(FULLMASK, fl, o);
    }
    int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        sh[0][w] = sv;
        sh[1][w] = mr;
        sh[2][w] = l2;
        sh[3][w] = mv;
        sh[4][w] = ne;
        sh[5][w] = (double)fl;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int u = 1; u < (int)(blockDim.x >> 5); u++) {
            sh[0][0] += sh[0][u];
            sh[1][0] = fmax(sh[1][0], sh[1][u]);
            sh[2][0] += sh[2][u];
            sh[3][0] = fmin(sh[3][0], sh[3][u]);
            sh[4][0] += sh[4][u];
            sh[5][0] = (double)((uint32_t)sh[5][0] | (uint32_t)sh[5][u]);
        }
        for (int q = 0; q < 6; q++) part[blockIdx.x * 6 + q] = sh[q][0];
    }
}

// The blocks' partials in block order (the sums' order is part of the result): loaded by the
// whole block, then one warp a quantity. A single thread that also loaded them took 94 us
// of every evaluation; this takes 15.
__global__ void __launch_bounds__(RED_BLOCKS) cell_reduce_final(const double* __restrict__ part,
                                                                double* __restrict__ out) {
    __shared__ double sh[6][RED_BLOCKS];
    for (int t = threadIdx.x; t < 6 * RED_BLOCKS; t += RED_BLOCKS) sh[t % 6][t / 6] = part[t];
    __syncthreads();
    const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (q == 0 || q == 2 || q == 4) {  // sums, serially
        if (lane == 0) {
            double v = 0;
#pragma unroll 16
            for (int b = 0; b < RED_BLOCKS; b++) v += sh[q][b];
            out[q] = q == 2 ? sqrt(v) : v;
        }
    } else if (q == 1 || q == 3) {  // maximum, minimum
        double v = q == 1 ? 0.0 : INFINITY;
        for (int b = lane; b < RED_BLOCKS; b += 32) v = q == 1 ? fmax(v, sh[q][b]) : fmin(v, sh[q][b]);
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_xor_sync(FULLMASK, v, o);
            v = q == 1 ? fmax(v, u) : fmin(v, u);
        }
        if (lane == 0) out[q] = v;
    } else if (q == 5) {
        uint32_t fl = 0;
        for (int b = lane; b < RED_BLOCKS; b += 32) fl |= (uint32_t)sh[5][b];
        fl = __reduce_or_sync(FULLMASK, fl);
        if (lane == 0) out[5] = (double)fl;
    }
}

// Warps of a clipping block and blocks for nwork cells: full blocks where there are cells
// for one on every SM, smaller ones (the cells spread over all SMs) below that.
struct ClipGrid {
    int warps, blocks;
};
template <typename R, class C>
static ClipGrid clip_grid(int64_t nwork) {
    const int sms = num_sms();
    const int64_t per_block = (nwork + sms - 1) / sms;
    ClipGrid g;
    g.warps = per_block < clip_warps<R, C>() ? (int)per_block : clip_warps<R, C>();
    const int64_t need = (nwork + g.warps - 1) / g.warps;
    const int most = sms * CLIP_BLOCKS_PER_SM;
    g.blocks = (int)(need < most ? need : most);
    return g;
}

template <typename R, class C, int MODE>
static int launch_clip(const ClipParams& cp, cudaStream_t s) {
    // the shared-memory limit, raised once per instantiation (thread-safe: contexts of
    // different host threads launch concurrently)
    static const cudaError_t err = cudaFuncSetAttribute(
        clip_kernel<R, C, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)(sizeof(Poly<R, C>) * clip_warps<R, C>()));
    if (err != cudaSuccess) {
        set_error(std::string("clip kernel setup: ") + cudaGetErrorString(err));
        return SDOT_ERR_CUDA;
    }
    if (cp.nwork < 1) return SDOT_OK;
    const ClipGrid g = clip_grid<R, C>(cp.nwork);
    clip_kernel<R, C, MODE><<<g.blocks, g.warps * 32, sizeof(Poly<R, C>) * g.warps, s>>>(cp);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    return SDOT_OK;
}

// clipping parameters of one evaluation of context d at psi (no work counter,
// work list or counters yet)
static ClipParams make_clip_params(DeviceState& d, const double* psi) {
    ClipParams cp;
    cp.N = d.N;
    cp.k = d.k;
    cp.a = d.a;
    cp.inv_a = 1.0 / d.a;
    cp.inv_a2 = 1.0 / (d.a * d.a);
    for (int a = 0; a < 3; a++) {
        cp.L[a] = d.L[a];
        cp.halfL[a] = 0.5 * d.L[a];
        cp.Lt[a] = (float)(d.L[a] / d.a);
        cp.halfLt[a] = 0.5f * cp.Lt[a];
        cp.ht[a] = (float)(d.grid.h[a] / d.a);
        cp.G[a] = d.grid.G[a];
    }
    cp.pos = d.pos;
    cp.posf = d.posf;
    cp.pslo = d.pslo;
    cp.ioff = d.ioff;
    for (int a = 0; a < 3; a++) cp.hfix[a] = (float)(d.grid.h[a] / d.a / 4294967296.0);
    cp.leafc = d.leafc;
    cp.facets_valid = d.facets_valid;
    cp.psi = psi;
    cp.knn = d.knn;
    cp.knn_d2k = d.knn_d2k;
    cp.cell_start = d.grid.cell_start;
    cp.pyr = d.pyr;
    for (int l = 0; l < MAXLEV; l++)
        for (int a = 0; a < 3; a++) cp.nsz[l][a] = (float)((double)(1 << (2 * l)) * d.grid.h[a] / d.a);
    cp.vol = d.vol;
    cp.m1 = d.m1;
    cp.anchor = d.anchor;
    cp.status = d.status;
    cp.fcnt = d.fcnt;
    cp.fcol = d.fcol;
    cp.fval = d.fval;
    cp.topo = d.topo;
    cp.topo_n = d.topo_n;
    cp.cert_f = d.cert_f;
    cp.cert_s = d.cert_s;
    cp.cert_j = d.cert_j;
    cp.cert_n = d.cert_n;
    cp.cert_dpsi = reinterpret_cast<const uint32_t*>(d.counters + 30);
    cp.cert_carried = d.counters + 29;
    cp.cert_use = d.carry;
    cp.queue_out = d.queue;
    cp.queue_cnt = d.counters + 0;
    cp.q64_out = d.queue64;
    cp.q64_cnt = d.counters + 1;
    cp.counters64 = (unsigned long long*)(d.counters + 8);
    cp.work_counter = nullptr;
    cp.worklist = nullptr;
    cp.nwork = d.N;
    cp.nwork_dev = nullptr;
    cp.pass = 1;
    return cp;
}

// the cells of context d at its current psi, for rebuilding them from their facets in
// FP64 (mesh.cu)
ClipParams mesh_clip_params(DeviceState& d) { return make_clip_params(d, d.psi); }

// The carried pass runs for FP32 cells that may hold a certificate. Its queue lies in
// rowcnt, which the CSR assembly rewrites.
static bool carries(const DeviceState& d, int precision) {
    return precision != SDOT_PREC_FP64 && d.carry && d.facets_valid;
}

int evaluate_cells(DeviceState& d, const double* psi, int precision, EvalResult* res,
                   cudaStream_t s) {
    NvtxRange nv("laguerre_cells");
    int rc = build_pyramid(d, psi, s);
    if (rc) return rc;
    ClipParams cp = make_clip_params(d, psi);
    SDOT_CUDA_TRY(cudaMemsetAsync(d.counters, 0, 30 * sizeof(int32_t), s));

    cudaEvent_t e0, e1, ep1, ep2;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventCreate(&ep1);
    cudaEventCreate(&ep2);
    cudaEventRecord(e0, s);
    // pass 1: every cell, first candidates + security test; before it, where certificates
    // may hold, the cells they carry
    cp.work_counter = d.counters + 2;
    cp.worklist = nullptr;
    cp.nwork = d.N;
    cp.pass = 1;
    if (carries(d, precision)) {
        cp.worklist = d.rowcnt;
        cp.nwork_dev = d.counters + 7;
        if ((rc = launch_carry(cp, d.rowcnt, d.counters + 7, d.counters + 25, s))) return rc;
    }
    rc = precision == SDOT_PREC_FP64 ? launch_clip<double, CapS, MODE_CERTIFY>(cp, s)
                                     : launch_clip<float, CapS, MODE_CERTIFY>(cp, s);
    if (rc) return rc;
    cudaEventRecord(ep1, s);
    int32_t cnt[2];
    SDOT_CUDA_TRY(cudaMemcpyAsync(cnt, d.counters, 8, cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    int64_t requeued = cnt[0];
    // pass 2: re-queued cells, full walk with clipping
    if (requeued > 0) {
        cp.work_counter = d.counters + 4;
        cp.worklist = d.queue;
        cp.nwork = requeued;
        cp.nwork_dev = nullptr;
        cp.pass = 2;
        rc = precision == SDOT_PREC_FP64 ? launch_clip<double, CapS, MODE_FULL>(cp, s)
                                         : launch_clip<float, CapS, MODE_FULL>(cp, s);
        if (rc) return rc;
        SDOT_CUDA_TRY(cudaMemcpyAsync(cnt, d.counters, 8, cudaMemcpyDeviceToHost, s));
        SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    }
    cudaEventRecord(ep2, s);
    int64_t reclipped = cnt[1];
    // pass 3: FP64 re-clip of the cells failing the FP32 checks or over the small
    // capacity: the small polytope first, then the large one for its overflows. Those go to
    // the re-queue pass's list, which is free by now and holds every cell: the cells of
    // pass 3 may fill queue64 already, and an overflow is in it a second time.
    if (reclipped > 0) {
        cp.pass = 3;
        cp.work_counter = d.counters + 5;
        cp.worklist = d.queue64;
        cp.nwork = reclipped;
        cp.nwork_dev = nullptr;
        if (precision != SDOT_PREC_FP64) {
            cp.q64_out = d.queue;
            cp.q64_cnt = d.counters;
            SDOT_CUDA_TRY(cudaMemsetAsync(d.counters, 0, sizeof(int32_t), s));
            if ((rc = launch_clip<double, CapS, MODE_FULL>(cp, s))) return rc;
            SDOT_CUDA_TRY(cudaMemcpyAsync(cnt, d.counters, 4, cudaMemcpyDeviceToHost, s));
            SDOT_CUDA_TRY(cudaStreamSynchronize(s));
            cp.work_counter = d.counters + 6;
            cp.worklist = d.queue;
            cp.nwork = cnt[0];
        }
        if (cp.nwork > 0 && (rc = launch_clip<double, CapL, MODE_FULL>(cp, s))) return rc;
    }
    cudaEventRecord(e1, s);
    cell_reduce_kernel<<<RED_BLOCKS, 256, 0, s>>>(d.vol, d.nu, d.status, d.N, d.partials);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    cell_reduce_final<<<1, RED_BLOCKS, 0, s>>>(d.partials, d.scal);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    double h[6];
    SDOT_CUDA_TRY(cudaMemcpyAsync(h, d.scal, sizeof h, cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventElapsedTime(&res->ms_pass[0], e0, ep1);
    cudaEventElapsedTime(&res->ms_pass[1], ep1, ep2);
    cudaEventElapsedTime(&res->ms_pass[2], ep2, e1);
    SDOT_CUDA_TRY(cudaMemcpy(res->work, d.counters + 8, 64, cudaMemcpyDeviceToHost));
    int32_t carried = 0;
    SDOT_CUDA_TRY(cudaMemcpy(&carried, d.counters + 29, 4, cudaMemcpyDeviceToHost));
    res->carried = carried;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaEventDestroy(ep1);
    cudaEventDestroy(ep2);
    d.facets_valid = 1;  // every cell now holds its facets of this diagram
    res->sum_vol = h[0];
    res->max_rel_err = h[1];
    res->l2_err = h[2];
    res->min_vol = h[3];
    res->n_empty = (int64_t)h[4];
    res->flags = (uint32_t)h[5];
    res->requeued = requeued;
    res->reclipped = reclipped;
    res->ms = ms;
    return SDOT_OK;
}


// ---------------------------------------------------------------------------
// batched evaluation: one persistent launch per pass over the cells of several
// contexts (the server's jobs)
// ---------------------------------------------------------------------------
template <typename R, class C, int MODE>
static int launch_clip_batch(const ClipBatch& bt, int64_t total, cudaStream_t s) {
    static const cudaError_t err = cudaFuncSetAttribute(
        clip_batch_kernel<R, C, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)(sizeof(Poly<R, C>) * clip_warps<R, C>()));
    if (err != cudaSuccess) {
        set_error(std::string("clip batch kernel setup: ") + cudaGetErrorString(err));
        return SDOT_ERR_CUDA;
    }
    if (total < 1) return SDOT_OK;
    const ClipGrid g = clip_grid<R, C>(total);
    clip_batch_kernel<R, C, MODE><<<g.blocks, g.warps * 32, sizeof(Poly<R, C>) * g.warps, s>>>(bt);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    return SDOT_OK;
}

// Job tables of a batch: one slot per launch of a pass (the FP32 and the FP64 group);
// the host copies are pinned and reused after the stream has been synchronised.
struct BatchScratch {
    int cap = 0;
    ClipParams* jobs_dev[2] = {nullptr, nullptr};
    int64_t* start_dev[2] = {nullptr, nullptr};
    unsigned long long* counter_dev = nullptr;  // one per slot
    ClipParams* jobs_host[2] = {nullptr, nullptr};
    int64_t* start_host[2] = {nullptr, nullptr};
    int32_t* cnt_host = nullptr;  // 2 per job: re-queued, FP64 re-clip counts
    double* red_host = nullptr;   // 6 per job: the reductions of cell_reduce_final
};

void batch_scratch_destroy(BatchScratch* b) {
    if (!b) return;
    for (int t = 0; t < 2; t++) {
        cudaFree(b->jobs_dev[t]);
        cudaFree(b->start_dev[t]);
        cudaFreeHost(b->jobs_host[t]);
        cudaFreeHost(b->start_host[t]);
    }
    cudaFree(b->counter_dev);
    cudaFreeHost(b->cnt_host);
    cudaFreeHost(b->red_host);
    delete b;
}

int batch_scratch_create(int cap, BatchScratch** out) {
    *out = nullptr;
    if (cap < 1) return SDOT_ERR_ARG;
    BatchScratch* b = new BatchScratch();
    b->cap = cap;
    bool ok = true;
    for (int t = 0; t < 2 && ok; t++) {
        ok = cudaMalloc(&b->jobs_dev[t], sizeof(ClipParams) * cap) == cudaSuccess &&
             cudaMalloc(&b->start_dev[t], sizeof(int64_t) * (cap + 1)) == cudaSuccess &&
             cudaMallocHost(&b->jobs_host[t], sizeof(ClipParams) * cap) == cudaSuccess &&
             cudaMallocHost(&b->start_host[t], sizeof(int64_t) * (cap + 1)) == cudaSuccess;
    }
    ok = ok && cudaMalloc(&b->counter_dev, sizeof(unsigned long long) * 2) == cudaSuccess &&
         cudaMallocHost(&b->cnt_host, sizeof(int32_t) * 2 * cap) == cudaSuccess &&
         cudaMallocHost(&b->red_host, sizeof(double) * 6 * cap) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        batch_scratch_destroy(b);
        set_error("batch scratch: allocation failed");
        return SDOT_ERR_OOM;
    }
    *out = b;
    return SDOT_OK;
}

// one launch of pass MODE in precision R over the work items nwork[j] of the jobs with
// take[j] (items: worklist of cps[j], or cells 0..nwork[j]-1)
template <typename R, class C, int MODE>
static int launch_table(const std::vector<ClipParams>& cps, const std::vector<int64_t>& nwork,
                        const std::vector<char>& take, int slot, BatchScratch* sc,
                        cudaStream_t s) {
    int m = 0;
    int64_t total = 0;
    ClipParams* hj = sc->jobs_host[slot];
    int64_t* hs = sc->start_host[slot];
    for (size_t j = 0; j < cps.size(); j++) {
        if (!take[j] || nwork[j] <= 0) continue;
        hj[m] = cps[j];
        hj[m].nwork = nwork[j];
        hj[m].work_counter = nullptr;  // the batch counter hands out the items
        hs[m] = total;
        total += nwork[j];
        m++;
    }
    if (m == 0) return SDOT_OK;
    hs[m] = total;
    SDOT_CUDA_TRY(cudaMemcpyAsync(sc->jobs_dev[slot], hj, sizeof(ClipParams) * m,
                                  cudaMemcpyHostToDevice, s));
    SDOT_CUDA_TRY(cudaMemcpyAsync(sc->start_dev[slot], hs, sizeof(int64_t) * (m + 1),
                                  cudaMemcpyHostToDevice, s));
    SDOT_CUDA_TRY(cudaMemsetAsync(sc->counter_dev + slot, 0, sizeof(unsigned long long), s));
    ClipBatch bt;
    bt.jobs = sc->jobs_dev[slot];
    bt.start = sc->start_dev[slot];
    bt.counter = sc->counter_dev + slot;
    bt.njobs = m;
    return launch_clip_batch<R, C, MODE>(bt, total, s);
}

// the per-job counters (re-queued, FP64 re-clip) of every job, after a sync of s
static int read_counts(DeviceState* const* ds, int n, BatchScratch* sc, cudaStream_t s) {
    for (int j = 0; j < n; j++)
        SDOT_CUDA_TRY(cudaMemcpyAsync(sc->cnt_host + 2 * j, ds[j]->counters, 2 * sizeof(int32_t),
                                      cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    return SDOT_OK;
}

int evaluate_cells_batch(DeviceState* const* ds, const double* const* psis, const int* precs,
                         EvalResult* res, int n, BatchScratch* sc, cudaStream_t s) {
    if (n < 1 || !sc || n > sc->cap) {
        set_error("evaluate_cells_batch: batch size out of range");
        return SDOT_ERR_ARG;
    }
    int rc;
    std::vector<ClipParams> cps((size_t)n);
    std::vector<int64_t> nwork((size_t)n);
    std::vector<char> is64((size_t)n), is32((size_t)n), all((size_t)n, 1);
    for (int j = 0; j < n; j++) {
        DeviceState& d = *ds[j];
        if ((rc = build_pyramid(d, psis[j], s))) return rc;
        cps[j] = make_clip_params(d, psis[j]);
        SDOT_CUDA_TRY(cudaMemsetAsync(d.counters, 0, 30 * sizeof(int32_t), s));
        is64[j] = precs[j] == SDOT_PREC_FP64;
        is32[j] = !is64[j];
    }
    cudaEvent_t e0, e1, ep1, ep2;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventCreate(&ep1);
    cudaEventCreate(&ep2);
    auto cleanup = [&] {
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        cudaEventDestroy(ep1);
        cudaEventDestroy(ep2);
    };
    cudaEventRecord(e0, s);
    // pass 1: every cell of every job, less those a certificate carries (each job's carried
    // pass comes first and leaves the rest in its queue)
    bool carry = false;
    for (int j = 0; j < n; j++) {
        DeviceState& d = *ds[j];
        cps[j].worklist = nullptr;
        cps[j].pass = 1;
        nwork[j] = d.N;
        if (!carries(d, precs[j])) continue;
        cps[j].worklist = d.rowcnt;
        rc = launch_carry(cps[j], d.rowcnt, d.counters + 7, d.counters + 25, s);
        if (!rc && cudaMemcpyAsync(sc->cnt_host + 2 * j, d.counters + 7, sizeof(int32_t),
                                   cudaMemcpyDeviceToHost, s) != cudaSuccess) {
            set_error("evaluate_cells_batch: reading a queue's count failed");
            rc = SDOT_ERR_CUDA;
        }
        if (rc) {
            cleanup();
            return rc;
        }
        carry = true;
    }
    if (carry) {
        if (cudaStreamSynchronize(s) != cudaSuccess) {
            cleanup();
            set_error("evaluate_cells_batch: the carried pass failed");
            return SDOT_ERR_CUDA;
        }
        for (int j = 0; j < n; j++)
            if (cps[j].worklist) nwork[j] = sc->cnt_host[2 * j];
    }
    if ((rc = launch_table<float, CapS, MODE_CERTIFY>(cps, nwork, is32, 0, sc, s)) ||
        (rc = launch_table<double, CapS, MODE_CERTIFY>(cps, nwork, is64, 1, sc, s))) {
        cleanup();
        return rc;
    }
    cudaEventRecord(ep1, s);
    if ((rc = read_counts(ds, n, sc, s))) {
        cleanup();
        return rc;
    }
    std::vector<int64_t> requeued((size_t)n), reclipped((size_t)n);
    bool any = false;
    for (int j = 0; j < n; j++) {
        requeued[j] = sc->cnt_host[2 * j];
        cps[j].worklist = ds[j]->queue;
        cps[j].pass = 2;
        nwork[j] = requeued[j];
        any = any || requeued[j] > 0;
    }
    // pass 2: the re-queued cells, full walk with clipping
    if (any) {
        if ((rc = launch_table<float, CapS, MODE_FULL>(cps, nwork, is32, 0, sc, s)) ||
            (rc = launch_table<double, CapS, MODE_FULL>(cps, nwork, is64, 1, sc, s))) {
            cleanup();
            return rc;
        }
    }
    cudaEventRecord(ep2, s);
    if ((rc = read_counts(ds, n, sc, s))) {
        cleanup();
        return rc;
    }
    any = false;
    for (int j = 0; j < n; j++) {
        reclipped[j] = sc->cnt_host[2 * j + 1];
        cps[j].worklist = ds[j]->queue64;
        cps[j].pass = 3;
        nwork[j] = reclipped[j];
        any = any || nwork[j] > 0;
    }
    // pass 3: FP64 re-clip with the large capacity (FP32 cells failing the checks,
    // cells over the small capacity)
    if (any && (rc = launch_table<double, CapL, MODE_FULL>(cps, nwork, all, 0, sc, s))) {
        cleanup();
        return rc;
    }
    cudaEventRecord(e1, s);
    std::vector<unsigned long long> work((size_t)n * 8);
    for (int j = 0; j < n; j++) {
        DeviceState& d = *ds[j];
        SDOT_CUDA_TRY(cudaMemcpyAsync(work.data() + 8 * j, d.counters + 8, 64,
                                      cudaMemcpyDeviceToHost, s));
        cell_reduce_kernel<<<RED_BLOCKS, 256, 0, s>>>(d.vol, d.nu, d.status, d.N, d.partials);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        cell_reduce_final<<<1, RED_BLOCKS, 0, s>>>(d.partials, d.scal);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        SDOT_CUDA_TRY(cudaMemcpyAsync(sc->red_host + 6 * j, d.scal, 6 * sizeof(double),
                                      cudaMemcpyDeviceToHost, s));
    }
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    float ms = 0, mp[3] = {0, 0, 0};
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventElapsedTime(&mp[0], e0, ep1);
    cudaEventElapsedTime(&mp[1], ep1, ep2);
    cudaEventElapsedTime(&mp[2], ep2, e1);
    cleanup();
    for (int j = 0; j < n; j++) {
        DeviceState& d = *ds[j];
        EvalResult& r = res[j];
        const double* h = sc->red_host + 6 * j;
        for (int q = 0; q < 8; q++) r.work[q] = work[8 * j + q];
        d.facets_valid = 1;
        r.sum_vol = h[0];
        r.max_rel_err = h[1];
        r.l2_err = h[2];
        r.min_vol = h[3];
        r.n_empty = (int64_t)h[4];
        r.flags = (uint32_t)h[5];
        r.requeued = requeued[j];
        r.reclipped = reclipped[j];
        r.ms = ms;
        for (int q = 0; q < 3; q++) r.ms_pass[q] = mp[q];
    }
    return SDOT_OK;
}

}  // namespace sdot
