// Spatial hash of the seeds and the periodic k-nearest-neighbour lists.
//
// The seeds are binned into a G^3 grid of cells of ~seeds_per_leaf seeds, sorted by
// cell (counting sort; ties inside a cell by caller index, so the order is
// deterministic) and kept in that order on the device for every later kernel.
// Each query takes shells of grid cells until its k-th distance is below the distance
// to the first unvisited shell. The distance key is (d^2, caller index) with
// d^2 = (dx*dx + dy*dy) + dz*dz of the minimum-image difference, evaluated with
// explicit round-to-nearest products and sums (no FMA) so that it is bit-identical
// to a plain IEEE binary64 evaluation.
//
// The paper computes the Laguerre diagram exactly (Sec. "Monge-Ampere-Kantorovich
// Reconstruction", eq. laguerrecell) without saying how neighbours are found; the
// kNN list is the first candidate set of the clipping kernel.
#include <float.h>
#include <limits.h>

#include "internal.cuh"

namespace sdot {

static unsigned long long g_launches = 0;
void note_launch() { __atomic_add_fetch(&g_launches, 1ull, __ATOMIC_RELAXED); }
unsigned long long launch_count() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }

// SM count of the device current at the first call (initialised once, thread-safe)
int num_sms() {
    static const int n = [] {
        int dev = 0, m = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev);
        return m > 0 ? m : 1;
    }();
    return n;
}

// ---------------------------------------------------------------------------
// exclusive scan (three-phase, recursive over block sums)
// ---------------------------------------------------------------------------
constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int64_t SCAN_CHUNK = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__device__ T block_exclusive_scan(T v, T* total) {
    __shared__ T ws[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        T s = (lane < nw) ? ws[lane] : T(0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        ws[lane] = s;
    }
    __syncthreads();
    T pre = (w > 0) ? ws[w - 1] : T(0);
    *total = ws[nw - 1];
    __syncthreads();
    return pre + x - v;
}

template <typename Tin, typename Tout>
__global__ void scan_sums_kernel(const Tin* in, int64_t n, Tout* sums) {
    int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_ITEMS;
    Tout t = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++)
        if (base + k < n) t += (Tout)in[base + k];
    __shared__ Tout red[32];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        Tout s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : Tout(0);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) sums[blockIdx.x] = s;
    }
}

template <typename Tin, typename Tout>
__global__ void scan_apply_kernel(const Tin* in, Tout* out, int64_t n, const Tout* offsets) {
    int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_ITEMS;
    Tout v[SCAN_ITEMS];
    Tout t = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        v[k] = (base + k < n) ? (Tout)in[base + k] : Tout(0);
        t += v[k];
    }
    Tout total;
    Tout pre = block_exclusive_scan<Tout>(t, &total);
    if (offsets) pre += offsets[blockIdx.x];
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        if (base + k < n) out[base + k] = pre;
        pre += v[k];
    }
}

size_t scan_temp_bytes(int64_t n) {
    size_t b = 0;
    while (n > SCAN_CHUNK) {
        n = (n + SCAN_CHUNK - 1) / SCAN_CHUNK;
        b += (size_t)n * sizeof(int64_t) + 256;
    }
    return b + 256;
}

template <typename Tin, typename Tout>
static int scan_impl(const Tin* in, Tout* out, int64_t n, char* temp, cudaStream_t s) {
    if (n <= 0) return SDOT_OK;
    int64_t nb = (n + SCAN_CHUNK - 1) / SCAN_CHUNK;
    if (nb == 1) {
        scan_apply_kernel<Tin, Tout><<<1, SCAN_THREADS, 0, s>>>(in, out, n, nullptr);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        return SDOT_OK;
    }
    Tout* sums = reinterpret_cast<Tout*>(temp);
    char* next = temp + ((nb * sizeof(Tout) + 255) / 256) * 256;
    scan_sums_kernel<Tin, Tout><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, n, sums);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    int rc = scan_impl<Tout, Tout>(sums, sums, nb, next, s);
    if (rc) return rc;
    scan_apply_kernel<Tin, Tout><<<(unsigned)nb, SCAN_THREADS, 0, s>>>(in, out, n, sums);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    return SDOT_OK;
}

int scan_exclusive_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, void* temp,
                              cudaStream_t s) {
    return scan_impl<int32_t, int64_t>(in, out, n, (char*)temp, s);
}
int scan_exclusive_i32(const int32_t* in, int32_t* out, int64_t n, void* temp,
                       cudaStream_t s) {
    return scan_impl<int32_t, int32_t>(in, out, n, (char*)temp, s);
}

// ---------------------------------------------------------------------------
// grid build
// ---------------------------------------------------------------------------
struct GridParams {
    int G[3];
    double h[3];
    double L[3];
};

__device__ __forceinline__ int cell_coord(double x, double h, int G) {
    int c = (int)floor(x / h);
    return c < 0 ? 0 : (c >= G ? G - 1 : c);
}

__global__ void keys_kernel(const double* __restrict__ pos, int64_t N, GridParams gp,
                            int32_t* __restrict__ key, int32_t* __restrict__ count,
                            int* __restrict__ bad) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
    bool ok = isfinite(x) && isfinite(y) && isfinite(z) && x >= 0.0 && y >= 0.0 &&
              z >= 0.0 && x < gp.L[0] && y < gp.L[1] && z < gp.L[2];
    if (!ok) {
        atomicOr(bad, 1);
        x = y = z = 0.0;
    }
    int cx = cell_coord(x, gp.h[0], gp.G[0]);
    int cy = cell_coord(y, gp.h[1], gp.G[1]);
    int cz = cell_coord(z, gp.h[2], gp.G[2]);
    int32_t k = (cz * gp.G[1] + cy) * gp.G[0] + cx;
    key[i] = k;
    atomicAdd(&count[k], 1);
}

__global__ void scatter_kernel(const int32_t* __restrict__ key, int64_t N,
                               const int32_t* __restrict__ start, int32_t* __restrict__ fill,
                               int32_t* __restrict__ perm) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    int32_t k = key[i];
    int32_t slot = start[k] + atomicAdd(&fill[k], 1);
    perm[slot] = (int32_t)i;
}

// insertion sort of each cell's seeds by caller index (cells hold few seeds)
__global__ void sort_cells_kernel(const int32_t* __restrict__ start, int64_t ncell,
                                  int32_t* __restrict__ perm) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    int32_t b = start[c], e = start[c + 1];
    for (int32_t t = b + 1; t < e; t++) {
        int32_t v = perm[t];
        int32_t u = t - 1;
        while (u >= b && perm[u] > v) {
            perm[u + 1] = perm[u];
            u--;
        }
        perm[u + 1] = v;
    }
}

__global__ void finalize_sort_kernel(const double* __restrict__ pos_user, int64_t N,
                                     const int32_t* __restrict__ perm,
                                     int32_t* __restrict__ iperm, Pos4* __restrict__ pos) {
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    int32_t i = perm[s];
    iperm[i] = (int32_t)s;
    pos[s] = Pos4::make(pos_user[3 * (int64_t)i], pos_user[3 * (int64_t)i + 1],
                          pos_user[3 * (int64_t)i + 2], (double)i);
}

int build_grid(DeviceState& d, const double* pos_user_dev, double seeds_per_leaf, void* temp,
               cudaStream_t s, const char* who) {
    const int64_t N = d.N;
    double vol = d.L[0] * d.L[1] * d.L[2];
    double h = cbrt(seeds_per_leaf * vol / (double)N);
    GridParams gp;
    int64_t ncell = 1;
    for (int a = 0; a < 3; a++) {
        double g = floor(d.L[a] / h);
        if (g < 1) g = 1;
        if (g > 1024) g = 1024;
        gp.G[a] = (int)g;
        gp.h[a] = d.L[a] / g;
        gp.L[a] = d.L[a];
        d.grid.G[a] = gp.G[a];
        d.grid.h[a] = gp.h[a];
        ncell *= gp.G[a];
    }
    d.grid.ncell = ncell;
    // temp layout: key[N] | count[ncell] | fill[ncell] | bad | scan temp
    char* t = (char*)temp;
    int32_t* key = (int32_t*)t;
    t += ((N * 4 + 255) / 256) * 256;
    int32_t* count = (int32_t*)t;
    t += ((ncell * 4 + 255) / 256) * 256;
    int32_t* fill = (int32_t*)t;
    t += ((ncell * 4 + 255) / 256) * 256;
    int* bad = (int*)t;
    t += 256;
    SDOT_CUDA_TRY(cudaMemsetAsync(count, 0, ncell * 4, s));
    SDOT_CUDA_TRY(cudaMemsetAsync(fill, 0, ncell * 4, s));
    SDOT_CUDA_TRY(cudaMemsetAsync(bad, 0, 4, s));
    unsigned nb = (unsigned)((N + 255) / 256);
    keys_kernel<<<nb, 256, 0, s>>>(pos_user_dev, N, gp, key, count, bad);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    // cell_start = exclusive scan of counts, with cell_start[ncell] = N
    int rc = scan_exclusive_i32(count, d.grid.cell_start, ncell, t, s);
    if (rc) return rc;
    int32_t nN = (int32_t)N;
    SDOT_CUDA_TRY(cudaMemcpyAsync(d.grid.cell_start + ncell, &nN, 4, cudaMemcpyHostToDevice, s));
    scatter_kernel<<<nb, 256, 0, s>>>(key, N, d.grid.cell_start, fill, d.perm);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    sort_cells_kernel<<<(unsigned)((ncell + 255) / 256), 256, 0, s>>>(d.grid.cell_start, ncell,
                                                                     d.perm);
                                                                     note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    finalize_sort_kernel<<<nb, 256, 0, s>>>(pos_user_dev, N, d.perm, d.iperm, d.pos);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    int hbad = 0;
    SDOT_CUDA_TRY(cudaMemcpyAsync(&hbad, bad, 4, cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    if (hbad) {
        set_error(std::string(who) + ": a position is not finite or lies outside [0, box)");
        return SDOT_ERR_ARG;
    }
    return SDOT_OK;
}

// ---------------------------------------------------------------------------
// kNN
// ---------------------------------------------------------------------------
struct KnnParams {
    int G[3];
    double h[3];
    double L[3];
    double halfL[3];
    int64_t N;
    int k;
};

// minimum-image component, same rule as a plain statement of it:
// if dx > L/2 subtract L, else if dx < -L/2 add L
__device__ __forceinline__ double wrap_d(double dx, double L, double halfL) {
    if (dx > halfL) return __dsub_rn(dx, L);
    if (dx < -halfL) return __dadd_rn(dx, L);
    return dx;
}

__device__ __forceinline__ double dist2_exact(const Pos4& a, const Pos4& b,
                                              const KnnParams& p) {
    double dx = wrap_d(__dsub_rn(b.x, a.x), p.L[0], p.halfL[0]);
    double dy = wrap_d(__dsub_rn(b.y, a.y), p.L[1], p.halfL[1]);
    double dz = wrap_d(__dsub_rn(b.z, a.z), p.L[2], p.halfL[2]);
    return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

template <int K>
struct TopK {
    double d[K];
    int o[K];   // caller index (tie key)
    int s[K];   // sorted index
    __device__ void init() {
#pragma unroll
        for (int t = 0; t < K; t++) {
            d[t] = DBL_MAX;
            o[t] = INT_MAX;
            s[t] = -1;
        }
    }
    __device__ __forceinline__ static bool less(double d1, int o1, double d2, int o2) {
        return d1 < d2 || (d1 == d2 && o1 < o2);
    }
    __device__ __forceinline__ void insert(double cd, int co, int cs) {
        if (!less(cd, co, d[K - 1], o[K - 1])) return;
#pragma unroll
        for (int t = K - 1; t >= 0; t--) {
            if (less(cd, co, d[t], o[t])) {
                bool sh = (t > 0) && less(cd, co, d[t - 1], o[t - 1]);
                d[t] = sh ? d[t - 1] : cd;
                o[t] = sh ? o[t - 1] : co;
                s[t] = sh ? s[t - 1] : cs;
            }
        }
    }
};

// Exact search of query q: rings of grid cells with the FP64 key, from ring 0 until
// the k-th key is below the squared distance to the first unvisited ring (brute force
// over all seeds when the rings would wrap onto visited cells).
template <int K>
__device__ __noinline__ void knn_exact(const Pos4* __restrict__ pos,
                                       const int32_t* __restrict__ cell_start,
                                       const KnnParams& p, int64_t q, TopK<K>& top) {
    const Pos4 yi = pos[q];
    top.init();
    int c[3];
    double m = DBL_MAX;
    {
        const double xs[3] = {yi.x, yi.y, yi.z};
        for (int a = 0; a < 3; a++) {
            int cc = (int)floor(xs[a] / p.h[a]);
            cc = cc < 0 ? 0 : (cc >= p.G[a] ? p.G[a] - 1 : cc);
            c[a] = cc;
            const double f = xs[a] - cc * p.h[a];
            double ma = fmin(f, p.h[a] - f);
            if (ma < 0) ma = 0;
            m = fmin(m, ma);
        }
    }
    const int Gmin = min(p.G[0], min(p.G[1], p.G[2]));
    const int k = p.k;
    bool done = false;
    for (int r = 0; !done; r++) {
        if (2 * r + 1 > Gmin) {
            // the next ring would wrap onto visited cells: finish by brute force
            top.init();
            for (int64_t t = 0; t < p.N; t++) {
                if (t == q) continue;
                const Pos4 yj = pos[t];
                top.insert(dist2_exact(yi, yj, p), (int)yj.w, (int)t);
            }
            break;
        }
        for (int oz = -r; oz <= r; oz++) {
            const int cz = ((c[2] + oz) % p.G[2] + p.G[2]) % p.G[2];
            for (int oy = -r; oy <= r; oy++) {
                const int cy = ((c[1] + oy) % p.G[1] + p.G[1]) % p.G[1];
                const bool face = (oz == -r || oz == r || oy == -r || oy == r);
                const int step = (face || r == 0) ? 1 : 2 * r;
                for (int ox = -r; ox <= r; ox += step) {
                    const int cx = ((c[0] + ox) % p.G[0] + p.G[0]) % p.G[0];
                    const int64_t cell = ((int64_t)cz * p.G[1] + cy) * p.G[0] + cx;
                    const int32_t b = cell_start[cell], e = cell_start[cell + 1];
                    for (int32_t t = b; t < e; t++) {
                        if (t == q) continue;
                        const Pos4 yj = pos[t];
                        top.insert(dist2_exact(yi, yj, p), (int)yj.w, t);
                    }
                }
            }
        }
        // every unvisited seed lies at least r*h + m away
        double bound = DBL_MAX;
        for (int a = 0; a < 3; a++) bound = fmin(bound, r * p.h[a] + m);
        double kth = DBL_MAX;
#pragma unroll
        for (int t = 0; t < K; t++)
            if (t == k - 1) kth = top.d[t];
        if (kth < DBL_MAX && kth < bound * bound * (1.0 - 1e-12)) done = true;
    }
}

// Grid-local FP32 offsets of every seed (in units of the grid cell) and its grid cell
// (x | y << 10 | z << 20, in w's bits), for the FP32 pass of the search.
__global__ void knn_prep_kernel(const Pos4* __restrict__ pos, int64_t N, KnnParams p,
                                float4* __restrict__ off) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N) return;
    const Pos4 y = pos[t];
    const double xs[3] = {y.x, y.y, y.z};
    int c[3];
    float o[3];
    for (int a = 0; a < 3; a++) {
        int cc = (int)floor(xs[a] / p.h[a]);
        cc = cc < 0 ? 0 : (cc >= p.G[a] ? p.G[a] - 1 : cc);
        c[a] = cc;
        o[a] = (float)((xs[a] - cc * p.h[a]) / p.h[a]);
    }
    off[t] = make_float4(o[0], o[1], o[2], __int_as_float(c[0] | (c[1] << 10) | (c[2] << 20)));
}

// k nearest seeds of every query, one warp a query.
//
// An FP32 pass keeps the seeds that may be among the nearest: approximate squared distances
// (grid-cell difference plus FP32 offset difference, in grid-cell units, minimum image),
// whose error is below Delta = 1e-5 (F_k + 1) for distances of a few grid cells, so every
// seed of the exact top k has an approximate key <= tau = F_k + 2 Delta (F_k: the k-th
// approximate key so far). The block of 3^3 grid cells around the query, then the shells
// beyond it, until the unvisited seeds are beyond tau + Delta. A row of grid cells along x
// is one run of the sorted order (the two ends of a row inside a shell are two), so 32
// lanes test 32 seeds at a time; the ones within tau are appended to a buffer of the warp,
// which is cut back to tau when it fills up. The entries left get the exact FP64 key (no
// FMA, ties by caller index) and each counts the entries before it: its place.
// What does not fit (shells that would wrap, more near ties than the buffer holds, as on a
// lattice with a large k) goes to a queue for the exact search.
//
// A thread a query with a sorted list in registers was bound by its serial chain (168
// registers, 12 warps an SM): 912,673 seeds, k = 24: 10.8 -> 2.6 ms; 4913 seeds, where 39
// blocks were all there was: 250 -> 27 us.
constexpr int KNN_WARPS = 8;   // queries of a block
constexpr int KNN_BUF = 128;   // buffer entries, 4 a lane
constexpr int KNN_FINAL = 96;  // entries that are ranked exactly, 3 a lane

struct KnnBuf {
    float key[KNN_BUF];
    int32_t s[KNN_BUF];
    unsigned long long d[KNN_FINAL];  // exact keys, as ordered bits
    int32_t o[KNN_FINAL];             // caller index
};

// Cut the buffer of n entries back to those <= tau; returns their number and tau (FLT_MAX
// while there are fewer than k). The k-th smallest key by bisection on the keys' bits
// (ordered, as they are not negative); it ends as soon as a pivot leaves exactly k below.
__device__ __forceinline__ int knn_prune(KnnBuf& B, int n, int k, float& tau, int lane) {
    if (n < k) return n;
    uint32_t v[4];
    int32_t s[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int t = lane + 32 * e;
        v[e] = t < n ? __float_as_uint(B.key[t]) : 0xffffffffu;
        s[e] = t < n ? B.s[t] : -1;
    }
    uint32_t lo = __reduce_min_sync(0xffffffffu, min(min(v[0], v[1]), min(v[2], v[3])));
    uint32_t mx = 0;
#pragma unroll
    for (int e = 0; e < 4; e++)
        if (v[e] != 0xffffffffu) mx = max(mx, v[e]);
    uint32_t hi = __reduce_max_sync(0xffffffffu, mx);
    while (lo < hi) {  // at most 32 steps; count(<= hi) >= k throughout
        const uint32_t mid = lo + ((hi - lo) >> 1);
        int c = 0;
#pragma unroll
        for (int e = 0; e < 4; e++) c += v[e] <= mid ? 1 : 0;
        c = __reduce_add_sync(0xffffffffu, c);
        if (c >= k) hi = mid;
        else lo = mid + 1;
        if (c == k) break;
    }
    mx = 0;
#pragma unroll
    for (int e = 0; e < 4; e++)
        if (v[e] <= hi) mx = max(mx, v[e]);
    const float Fk = __uint_as_float(__reduce_max_sync(0xffffffffu, mx));
    tau = Fk + 2.f * (1e-5f * (Fk + 1.f));
    const uint32_t tb = __float_as_uint(tau);
    int m = 0;
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const uint32_t b = __ballot_sync(0xffffffffu, v[e] <= tb);
        if (v[e] <= tb) {
            const int at = m + __popc(b & ((1u << lane) - 1u));
            B.key[at] = __uint_as_float(v[e]);
            B.s[at] = s[e];
        }
        m += __popc(b);
    }
    __syncwarp();
    return m;
}

__global__ void __launch_bounds__(KNN_WARPS * 32)
    knn_kernel(const Pos4* __restrict__ pos, const float4* __restrict__ off,
               const int32_t* __restrict__ cell_start, KnnParams p, int32_t* __restrict__ knn,
               double* __restrict__ d2k, int* __restrict__ flags, int32_t* __restrict__ rest,
               int32_t* __restrict__ nrest) {
    __shared__ KnnBuf bufs[KNN_WARPS];
    const int lane = threadIdx.x & 31;
    KnnBuf& B = bufs[threadIdx.x >> 5];
    const int64_t q = (int64_t)blockIdx.x * KNN_WARPS + (threadIdx.x >> 5);
    if (q >= p.N) return;
    const int k = p.k;
    const float4 oi = off[q];
    const int lc = __float_as_int(oi.w);
    const int c[3] = {lc & 1023, (lc >> 10) & 1023, (lc >> 20) & 1023};
    const float G[3] = {(float)p.G[0], (float)p.G[1], (float)p.G[2]};
    // grid cells are near-cubic; distances in units of the x cell size
    const float sy = (float)(p.h[1] / p.h[0]), sz = (float)(p.h[2] / p.h[0]);
    const float m = fminf(fminf(fminf(oi.x, 1.f - oi.x), fminf(oi.y, 1.f - oi.y) * sy),
                          fminf(oi.z, 1.f - oi.z) * sz);
    const int Gmin = min(p.G[0], min(p.G[1], p.G[2]));
    float tau = FLT_MAX;
    int n = 0;
    bool ok = false, full = false;
    for (int r = 1; 2 * r + 1 <= Gmin && !full; r++) {
        const int w = 2 * r + 1, rows = w * w;
        for (int base = 0; base < rows && !full; base += 32) {
            // this lane's row of grid cells: one run, or two
            const int row = base + lane;
            int32_t s0 = 0, s1 = 0;
            int n0 = 0, n1 = 0;
            if (row < rows) {
                const int rz = row / w, ry = row - rz * w;
                int cy = c[1] + ry - r, cz = c[2] + rz - r;
                if (cy < 0) cy += p.G[1];
                else if (cy >= p.G[1]) cy -= p.G[1];
                if (cz < 0) cz += p.G[2];
                else if (cz >= p.G[2]) cz -= p.G[2];
                const int32_t* cs = cell_start + ((int64_t)cz * p.G[1] + cy) * p.G[0];
                int X0 = c[0] - r, X1 = c[0] + r;
                // r = 1 takes the whole block, later shells only their own cells
                const bool whole = r == 1 || ry == 0 || ry == w - 1 || rz == 0 || rz == w - 1;
                if (whole) {
                    if (X0 < 0) {
                        X0 += p.G[0];
                        X1 += p.G[0];
                    }
                    s0 = cs[X0];
                    n0 = cs[min(X1, p.G[0] - 1) + 1] - s0;
                    if (X1 >= p.G[0]) {
                        s1 = cs[0];
                        n1 = cs[X1 - p.G[0] + 1] - s1;
                    }
                } else {
                    if (X0 < 0) X0 += p.G[0];
                    if (X1 >= p.G[0]) X1 -= p.G[0];
                    s0 = cs[X0];
                    n0 = cs[X0 + 1] - s0;
                    s1 = cs[X1];
                    n1 = cs[X1 + 1] - s1;
                }
            }
            const int nn = n0 + n1;
            int incl = nn;
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            const int excl = incl - nn;
            const int32_t first = s0 - excl, jump = s1 - (s0 + n0);
            const int split = excl + n0;
            for (int b = 0; b < total; b += 32) {
                const int t = b + lane;
                // the lane owning flattened seed t: the first with incl > t
                int u = 0;
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int y = __shfl_sync(0xffffffffu, incl, u + step - 1);
                    if (y <= t) u += step;
                }
                int32_t s = t + __shfl_sync(0xffffffffu, first, u);
                const int sp = __shfl_sync(0xffffffffu, split, u);
                const int32_t jq = __shfl_sync(0xffffffffu, jump, u);
                if (t >= sp) s += jq;
                float d2 = FLT_MAX;
                if (t < total && s != (int32_t)q) {
                    const float4 oj = off[s];
                    const int lj = __float_as_int(oj.w);
                    const int cj[3] = {lj & 1023, (lj >> 10) & 1023, (lj >> 20) & 1023};
                    const float dd[3] = {oj.x - oi.x, oj.y - oi.y, oj.z - oi.z};
                    float dx[3];
#pragma unroll
                    for (int a = 0; a < 3; a++) {
                        int dc = cj[a] - c[a];
                        if (2 * dc > p.G[a]) dc -= p.G[a];
                        else if (2 * dc < -p.G[a]) dc += p.G[a];
                        dx[a] = (float)dc + dd[a];
                        if (dx[a] > 0.5f * G[a]) dx[a] -= G[a];
                        else if (dx[a] < -0.5f * G[a]) dx[a] += G[a];
                    }
                    dx[1] *= sy;
                    dx[2] *= sz;
                    d2 = dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2];
                }
                const bool keep = d2 <= tau && d2 < FLT_MAX;
                const uint32_t km = __ballot_sync(0xffffffffu, keep);
                if (!km) continue;
                if (keep) {
                    const int at = n + __popc(km & ((1u << lane) - 1u));
                    B.key[at] = d2;
                    B.s[at] = s;
                }
                n += __popc(km);
                __syncwarp();
                if (n > KNN_BUF - 32) {
                    n = knn_prune(B, n, k, tau, lane);
                    if (n > KNN_BUF - 32) {  // too many near ties
                        full = true;
                        break;
                    }
                }
            }
        }
        if (full) break;
        n = knn_prune(B, n, k, tau, lane);
        if (n < k) continue;
        // every unvisited seed lies at least r + m cell sizes away; tau's Delta is (tau -
        // F_k) / 2
        const float bound = (float)r * fminf(1.f, fminf(sy, sz)) + m;
        if (tau + 1e-5f * (tau + 1.f) < bound * bound * (1.f - 1e-6f)) {
            ok = true;
            break;
        }
    }
    if (!ok || n > KNN_FINAL) {
        if (lane == 0) rest[atomicAdd(nrest, 1)] = (int32_t)q;
        return;
    }
    // exact keys, then each entry's place among them
    const Pos4 yi = pos[q];
    for (int e = lane; e < n; e += 32) {
        const Pos4 yj = pos[B.s[e]];
        B.d[e] = (unsigned long long)__double_as_longlong(dist2_exact(yi, yj, p));
        B.o[e] = (int)yj.w;
    }
    __syncwarp();
    for (int e = lane; e < n; e += 32) {
        const unsigned long long d = B.d[e];
        const int o = B.o[e];
        int place = 0;
        for (int u = 0; u < n; u++) place += B.d[u] < d || (B.d[u] == d && B.o[u] < o) ? 1 : 0;
        if (place < k) knn[q * k + place] = B.s[e];
        if (place == k - 1) d2k[q] = __longlong_as_double((long long)d);
        if (place == 0 && d == 0ull) atomicOr(flags, 1);  // duplicate position
    }
}

// The queries knn_kernel left, one thread each, by the exact search; rest null: all of them, in
// the seeds' order (threads of a warp then find their near seeds at the same places of a
// brute force search: 37 ms for 20,000 seeds, in the order of a queue 62).
template <int K>
__global__ void __launch_bounds__(128)
    knn_rest_kernel(const Pos4* __restrict__ pos, const int32_t* __restrict__ cell_start,
                    KnnParams p, const int32_t* __restrict__ rest,
                    const int32_t* __restrict__ nrest, int32_t* __restrict__ knn,
                    double* __restrict__ d2k, int* __restrict__ flags) {
    const int k = p.k;
    const int64_t n = rest ? (int64_t)*nrest : p.N;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t q = rest ? (int64_t)rest[e] : e;
        TopK<K> top;
        knn_exact<K>(pos, cell_start, p, q, top);
#pragma unroll
        for (int t = 0; t < K; t++) {
            if (t < k) knn[q * k + t] = top.s[t];
            if (t == k - 1) d2k[q] = top.d[t];
        }
        if (top.d[0] == 0.0) atomicOr(flags, 1);  // duplicate position
        if (top.s[0] < 0) atomicOr(flags, 2);      // fewer than k other seeds
    }
}

int build_knn(DeviceState& d, cudaStream_t s, int* dup_flag_host) {
    NvtxRange nv("knn");
    KnnParams p;
    for (int a = 0; a < 3; a++) {
        p.G[a] = d.grid.G[a];
        p.h[a] = d.grid.h[a];
        p.L[a] = d.L[a];
        p.halfL[a] = 0.5 * d.L[a];
    }
    p.N = d.N;
    p.k = d.k;
    int* flags = (int*)(d.counters + 3);
    int32_t* nrest = d.counters + 4;
    SDOT_CUDA_TRY(cudaMemsetAsync(flags, 0, 8, s));
    // FP32 grid-local offsets and grid cells: posf serves as scratch here (the first
    // Laguerre evaluation rewrites it), queue holds the queries for the exact search. A box
    // under three grid cells thin has no 3^3 grid cells around a query: the exact search.
    const bool thin = p.G[0] < 3 || p.G[1] < 3 || p.G[2] < 3;
    if (!thin) {
        knn_prep_kernel<<<(unsigned)((d.N + 127) / 128), 128, 0, s>>>(d.pos, d.N, p, d.posf);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        knn_kernel<<<(unsigned)((d.N + KNN_WARPS - 1) / KNN_WARPS), KNN_WARPS * 32, 0, s>>>(
            d.pos, d.posf, d.grid.cell_start, p, d.knn, d.knn_d2k, flags, d.queue, nrest);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
    }
    const int64_t rb = (d.N + 127) / 128, most = 4 * (int64_t)num_sms();
    const unsigned nb = (unsigned)(rb < most ? rb : most);
#define SDOT_KNN_REST(KK)                                                                    \
    knn_rest_kernel<KK><<<nb, 128, 0, s>>>(d.pos, d.grid.cell_start, p, thin ? nullptr : d.queue, \
                                           nrest, d.knn, d.knn_d2k, flags)
    // (a list longer than k takes in and shifts what cannot be in the answer: 20,000 seeds of
    // a box two grid cells thin, k = 24, all by brute force: 37 ms with 24 entries, 85 with 32)
    if (d.k <= 8) SDOT_KNN_REST(8);
    else if (d.k <= 16) SDOT_KNN_REST(16);
    else if (d.k <= 24) SDOT_KNN_REST(24);
    else if (d.k <= 32) SDOT_KNN_REST(32);
    else SDOT_KNN_REST(64);
#undef SDOT_KNN_REST
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    int h = 0;
    SDOT_CUDA_TRY(cudaMemcpyAsync(&h, flags, 4, cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    *dup_flag_host = h;
    return SDOT_OK;
}

__global__ void knn_user_kernel(const int32_t* __restrict__ knn, const int32_t* __restrict__ perm,
                                int64_t N, int k, int32_t* __restrict__ out) {
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N * k) return;
    int64_t s = t / k;
    int r = (int)(t - s * k);
    out[(int64_t)perm[s] * k + r] = perm[knn[t]];
}

int knn_to_user(const DeviceState& d, int32_t* out, cudaStream_t s) {
    int64_t n = d.N * d.k;
    knn_user_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(d.knn, d.perm, d.N, d.k, out);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    return SDOT_OK;
}

}  // namespace sdot
