// Power spectrum of a periodic mesh: the estimator behind the fractional BAO signal
// d(k) = P_wig(k) / P_nw(k) - 1 of Sec. "BAO reconstruction" (Fig. 2), applied to the
// densities sdot_mesh deposits for a wiggle / no-wiggle pair.
//
// delta = rho / mean(rho) - 1 on an M^3 mesh of a cubic box of side L; delta_k is the
// discrete Fourier transform divided by M^3, P(k) = L^3 |delta_k|^2 at k = 2 pi n / L,
// and mode n != 0 goes into bin b = floor(|n| + 1/2) for 1 <= b <= nbins. Per bin: the
// mean P over the modes, their mean |k| and their count, every mode of the full
// transform counted once (the real-to-complex half holds each pair +-n once, except on
// the planes n_c = 0 and n_c = M/2, where both members are stored).
//
// The transform is cuFFT's double-precision real-to-complex 3D FFT (a plain library
// transform, loaded with dlopen on first use so that nothing else in the library depends
// on it). The binning is this file's: mean(rho) by a fixed-order reduction; per bin the
// largest |F_k|^2 (integer maximum on the bits), then the sums of |F_k|^2 / max as 64-bit
// fixed point (unit 2^-38 of the bin's maximum, rounded once for each group of modes
// (+-n_a, +-n_b, n_c)) and of |n| (unit 2^-28), so the result does not depend on the order
// of the atomic additions.
#include <dlfcn.h>
#include <float.h>
#include <limits.h>
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <string>
#include <vector>

#include <cufft.h>

#include "internal.cuh"

namespace sdot {

namespace {

struct CufftApi {
    cufftResult (*plan3d)(cufftHandle*, int, int, int, cufftType) = nullptr;
    cufftResult (*set_stream)(cufftHandle, cudaStream_t) = nullptr;
    cufftResult (*exec_d2z)(cufftHandle, cufftDoubleReal*, cufftDoubleComplex*) = nullptr;
    cufftResult (*destroy)(cufftHandle) = nullptr;
    bool ok = false;
};

const CufftApi& cufft_api() {
    static const CufftApi api = [] {
        CufftApi a;
        // by soname (already loaded, or on the loader's path), then in the toolkit
        std::vector<std::string> names = {"libcufft.so.12", "libcufft.so.13", "libcufft.so.11",
                                          "libcufft.so"};
        const char* home = getenv("CUDA_HOME");
        for (const std::string dir : {std::string(home ? home : "/usr/local/cuda") + "/lib64/",
                                      std::string("/usr/local/cuda/lib64/")})
            for (const char* n : {"libcufft.so.12", "libcufft.so.13", "libcufft.so"})
                names.push_back(dir + n);
        void* h = nullptr;
        for (const std::string& n : names)
            if ((h = dlopen(n.c_str(), RTLD_NOW | RTLD_LOCAL))) break;
        if (!h) return a;
        a.plan3d = reinterpret_cast<decltype(a.plan3d)>(dlsym(h, "cufftPlan3d"));
        a.set_stream = reinterpret_cast<decltype(a.set_stream)>(dlsym(h, "cufftSetStream"));
        a.exec_d2z = reinterpret_cast<decltype(a.exec_d2z)>(dlsym(h, "cufftExecD2Z"));
        a.destroy = reinterpret_cast<decltype(a.destroy)>(dlsym(h, "cufftDestroy"));
        a.ok = a.plan3d && a.set_stream && a.exec_d2z && a.destroy;
        return a;
    }();
    return api;
}

constexpr int SPEC_THREADS = 256;
// fixed-point units: a bin holds at most ~2^24 weighted modes (M <= 1024), so sums stay
// below 2^62: |F_k|^2 / bin max (<= 1) in 2^-38, |n| (<= 887) in 2^-28
constexpr double FIX_P = 274877906944.0;  // 2^38
constexpr double FIX_K = 268435456.0;     // 2^28

// The working copy of the mesh (the transform may overwrite its input) and, in the same
// read, the partial sums of its mean.
__global__ void copy_sum_kernel(const double* __restrict__ rho, int64_t n, double* __restrict__ in,
                                double* __restrict__ part) {
    __shared__ double sh[SPEC_THREADS / 32];
    double v = 0.0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (int64_t)gridDim.x * blockDim.x) {
        const double r = rho[t];
        if (in != rho) in[t] = r;
        v += r;
    }
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < SPEC_THREADS / 32; w++) s += sh[w];
        part[blockIdx.x] = s;
    }
}

// one warp: each lane's share of the partials in order, then the lanes in order
__global__ void mesh_sum_final(const double* __restrict__ part, int nb,
                               double* __restrict__ out) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 32) s += part[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) *out = s;
}

// Segmented sum (or maximum) towards the first lane of each run of equal keys (keys do
// not decrease over the lanes); same[e]: the lane 2^e further on has this lane's key.
template <typename T, bool MAX>
__device__ __forceinline__ T run_reduce(T v, const bool (&same)[5]) {
#pragma unroll
    for (int e = 0; e < 5; e++) {
        const T u = __shfl_down_sync(0xffffffffu, v, 1 << e);
        if (same[e]) v = MAX ? (u > v ? u : v) : v + u;
    }
    return v;
}

// The modes of the half space (layout M x M x (M/2 + 1), last index fastest), binned. A
// warp takes the rows (+-a, +-b) of the first two indices together, a lane one value of the
// third: up to four modes with one |n|, so one bin and one count. Along a row |n| does not
// decrease over the lanes, so equal bins are runs, which are summed by shuffles before one
// lane adds to the block's bins in shared memory; the block adds those to the global bins
// once. The bin and |n| come from the integer |n|^2 without FP64, which is issued at a
// sixteenth of FP32's rate: an FP32 root and its residual give |n| in 2^-28 to one unit, and
// the integer |n|^2 2^56 - K^2 says which way the nearest unit K lies (an FP64 root rounds 6 of
// the 786,432 integers up to the |n|^2 of M = 1024 the wrong way, the root and residual alone 116).
// SUM = false: the largest |F_k|^2 per bin (bits in b0). SUM = true: b0 the sum of |F_k|^2
// in units of the bin's maximum / 2^38, b1 that of |n| in 2^-28, b2 the mode count.
// M = 512 (67 M modes, 1.08 GB read twice): maximum 4.6 -> 0.25 ms, sums 4.8 -> 0.51 ms, where
// every mode took an FP64 root and up to three global atomics.
template <bool SUM>
__global__ void __launch_bounds__(SPEC_THREADS)
    spec_kernel(const cufftDoubleComplex* __restrict__ F, int M, int nbins,
                const unsigned long long* __restrict__ maxbits, unsigned long long* __restrict__ b0,
                unsigned long long* __restrict__ b1, unsigned long long* __restrict__ b2) {
    extern __shared__ unsigned long long spec_bins[];  // SUM: 3 nbins, else nbins
    const int nsh = (SUM ? 3 : 1) * nbins;
    for (int t = threadIdx.x; t < nsh; t += blockDim.x) spec_bins[t] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int Mh = M / 2 + 1;  // distinct |n_a|, |n_b|, and values of n_c
    const int nwarp = gridDim.x * (blockDim.x >> 5);
    for (int q = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < Mh * Mh; q += nwarp) {
        const int a = q / Mh, b = q - a * Mh;
        const int a2 = (a != 0 && 2 * a != M) ? M - a : -1, b2i = (b != 0 && 2 * b != M) ? M - b : -1;
        const cufftDoubleComplex* r0 = F + ((int64_t)a * M + b) * Mh;
        const cufftDoubleComplex* r1 = a2 >= 0 ? F + ((int64_t)a2 * M + b) * Mh : nullptr;
        const cufftDoubleComplex* r2 = b2i >= 0 ? F + ((int64_t)a * M + b2i) * Mh : nullptr;
        const cufftDoubleComplex* r3 =
            a2 >= 0 && b2i >= 0 ? F + ((int64_t)a2 * M + b2i) * Mh : nullptr;
        const int rows = (r1 ? 2 : 1) * (r2 ? 2 : 1);
        const int ab2 = a * a + b * b;
        for (int c0 = 0; c0 < Mh; c0 += 32) {
            const int c = c0 + lane;
            const int d2 = ab2 + c * c;
            // bin = floor(sqrt(d2) + 1/2): the root rounded, corrected by integers
            const float root = sqrtf((float)d2);
            int bin = (int)(root + 0.5f);
            while (bin > 0 && bin * (bin - 1) >= d2) bin--;
            while ((bin + 1) * bin < d2) bin++;
            if (c >= Mh || bin > nbins) bin = INT_MAX;
            const uint32_t live = __ballot_sync(0xffffffffu, bin != INT_MAX);
            if (!live) break;  // larger |n| only from here on
            double p = 0.0;
            unsigned long long top = 0;  // u >= 0: its bits order like its value, NaN above all
            if (bin != INT_MAX) {
                auto add = [&](const cufftDoubleComplex* r) {
                    if (!r) return;
                    const cufftDoubleComplex f = r[c];
                    const double u = f.x * f.x + f.y * f.y;
                    const unsigned long long ub = (unsigned long long)__double_as_longlong(u);
                    if (SUM) p += u;
                    else top = ub > top ? ub : top;
                };
                add(r0);
                add(r1);
                add(r2);
                add(r3);
            }
            double unit = FIX_P;  // of p / maximum
            if (SUM && p > DBL_MAX) {  // four finite squares, too large together: quarters
                auto quarter = [&](const cufftDoubleComplex* r) {
                    if (!r) return;
                    const cufftDoubleComplex f = r[c];
                    p += 0.25 * (f.x * f.x + f.y * f.y);
                };
                p = 0.0;
                unit = 4.0 * FIX_P;
                quarter(r0);
                quarter(r1);
                quarter(r2);
                quarter(r3);
            }
            bool same[5];
#pragma unroll
            for (int e = 0; e < 5; e++) {
                const int k = __shfl_down_sync(0xffffffffu, bin, 1 << e);
                same[e] = lane + (1 << e) < 32 && k == bin;
            }
            const int prev = __shfl_up_sync(0xffffffffu, bin, 1);
            const bool head = bin != INT_MAX && bin > 0 && (lane == 0 || prev != bin);
            if (!SUM) {
                const unsigned long long v = run_reduce<unsigned long long, true>(top, same);
                if (head) atomicMax(&spec_bins[bin - 1], v);
            } else {
                // modes stored for both members of a pair count once
                const unsigned w = (c == 0 || 2 * c == M) ? 1u : 2u;
                unsigned long long ps = 0, ks = 0;
                if (bin != INT_MAX && bin > 0) {
                    const double pm = __longlong_as_double((long long)maxbits[bin - 1]);
                    ps = pm > 0.0 ? (unsigned long long)llrint(p / pm * unit) * w : 0ull;
                    const float rest = fmaf(-root, root, (float)d2) / (2.f * root);
                    unsigned long long K = (unsigned long long)((long long)(root * (float)FIX_K) +
                                                                llrintf(rest * (float)FIX_K));
                    // (K - 1/2)^2 < |n|^2 2^56 < (K + 1/2)^2; |rest56| < 2^40, so 64 bits do
                    const long long rest56 =
                        (long long)(((unsigned long long)d2 << 56) - K * K);
                    K += rest56 > (long long)K ? 1 : 0;
                    K -= rest56 <= -(long long)K ? 1 : 0;
                    ks = K * (w * rows);
                }
                ps = run_reduce<unsigned long long, false>(ps, same);
                ks = run_reduce<unsigned long long, false>(ks, same);
                const unsigned cnt =
                    run_reduce<unsigned, false>(bin != INT_MAX ? w * rows : 0u, same);
                if (head) {
                    atomicAdd(&spec_bins[bin - 1], ps);
                    atomicAdd(&spec_bins[nbins + bin - 1], ks);
                    atomicAdd(&spec_bins[2 * nbins + bin - 1], (unsigned long long)cnt);
                }
            }
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nbins; t += blockDim.x) {
        if (!SUM) {
            if (spec_bins[t]) atomicMax(&b0[t], spec_bins[t]);
        } else if (spec_bins[2 * nbins + t]) {
            atomicAdd(&b0[t], spec_bins[t]);
            atomicAdd(&b1[t], spec_bins[nbins + t]);
            atomicAdd(&b2[t], spec_bins[2 * nbins + t]);
        }
    }
}

}  // namespace

}  // namespace sdot

using namespace sdot;

extern "C" int sdot_power_spectrum(const double* rho, int M, double L, int nbins, double* P,
                                   double* kmean, int64_t* nmodes, void* stream) {
    set_error("");
    if (!rho || !P || M < 2 || M > 1024 || !(L > 0.0) || !isfinite(L) || nbins < 1 ||
        nbins > 2 * M) {
        set_error("sdot_power_spectrum: need rho, P, 2 <= M <= 1024, a finite L > 0 and "
                  "1 <= nbins <= 2 M");
        return SDOT_ERR_ARG;
    }
    const CufftApi& fft = cufft_api();
    if (!fft.ok) {
        set_error("sdot_power_spectrum: libcufft could not be loaded");
        return SDOT_ERR_CUDA;
    }
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int64_t n = (int64_t)M * M * M;
    const int Mh = M / 2 + 1;
    const int64_t nmode = (int64_t)M * M * Mh;
    NvtxRange nv("power_spectrum");
    // device scratch: a copy of rho (an out-of-place real-to-complex transform may use its
    // input as work space), the transform, the reduction partials and the bins
    const int nb_sum = 4 * num_sms();
    double* in = nullptr;
    cufftDoubleComplex* F = nullptr;
    double* part = nullptr;
    unsigned long long* bins = nullptr;  // maxbits, psum, ksum, cnt: nbins each
    cufftHandle plan = 0;
    bool have_plan = false;
    int rc = SDOT_OK;
    auto fail = [&](int code, const std::string& msg) {
        set_error("sdot_power_spectrum: " + msg);
        rc = code;
    };
    do {
        if (cudaMalloc(&in, (size_t)n * 8) != cudaSuccess ||
            cudaMalloc(&F, (size_t)nmode * sizeof(cufftDoubleComplex)) != cudaSuccess ||
            cudaMalloc(&part, (size_t)(nb_sum + 1) * 8) != cudaSuccess ||
            cudaMalloc(&bins, (size_t)4 * nbins * 8) != cudaSuccess) {
            cudaGetLastError();
            fail(SDOT_ERR_OOM, "device allocation failed");
            break;
        }
        // rho on this device is copied by the kernel that sums it; other memory first
        cudaPointerAttributes at;
        int dev = -1;
        const bool here = cudaPointerGetAttributes(&at, rho) == cudaSuccess &&
                          cudaGetDevice(&dev) == cudaSuccess &&
                          at.type == cudaMemoryTypeDevice && at.device == dev;
        cudaGetLastError();
        if ((!here &&
             cudaMemcpyAsync(in, rho, (size_t)n * 8, cudaMemcpyDefault, s) != cudaSuccess) ||
            cudaMemsetAsync(bins, 0, (size_t)4 * nbins * 8, s) != cudaSuccess) {
            fail(SDOT_ERR_CUDA, "copy of rho failed");
            break;
        }
        copy_sum_kernel<<<nb_sum, SPEC_THREADS, 0, s>>>(here ? rho : in, n, in, part);
        note_launch();
        mesh_sum_final<<<1, 32, 0, s>>>(part, nb_sum, part + nb_sum);
        note_launch();
        if (fft.plan3d(&plan, M, M, M, CUFFT_D2Z) != CUFFT_SUCCESS) {
            fail(SDOT_ERR_CUDA, "cufftPlan3d failed");
            break;
        }
        have_plan = true;
        if (fft.set_stream(plan, s) != CUFFT_SUCCESS || fft.exec_d2z(plan, in, F) != CUFFT_SUCCESS) {
            fail(SDOT_ERR_CUDA, "cufftExecD2Z failed");
            break;
        }
        // 3 nbins 8-byte bins of shared memory a block: at most 48 KB (nbins <= 2 M = 2048)
        const unsigned grid = (unsigned)(8 * num_sms());
        const size_t sh = (size_t)nbins * 8;
        spec_kernel<false><<<grid, SPEC_THREADS, sh, s>>>(F, M, nbins, nullptr, bins, nullptr,
                                                          nullptr);
        note_launch();
        spec_kernel<true><<<grid, SPEC_THREADS, 3 * sh, s>>>(F, M, nbins, bins, bins + nbins,
                                                             bins + 2 * nbins, bins + 3 * nbins);
        note_launch();
        if (cudaGetLastError() != cudaSuccess) {
            fail(SDOT_ERR_CUDA, "kernel launch failed");
            break;
        }
        std::vector<unsigned long long> h((size_t)4 * nbins);
        double sum = 0.0;
        if (cudaMemcpyAsync(h.data(), bins, h.size() * 8, cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaMemcpyAsync(&sum, part + nb_sum, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            fail(SDOT_ERR_CUDA, "read-back failed");
            break;
        }
        const double mean = sum / (double)n;
        if (!(mean > 0.0) || !isfinite(mean)) {
            fail(SDOT_ERR_ARG, "the mean of rho must be positive and finite");
            break;
        }
        // P = L^3 |F_k|^2 / (M^3 mean)^2 with F the unnormalised transform of rho
        const double norm = L * L * L / ((double)n * (double)n * mean * mean);
        for (int b = 0; b < nbins; b++) {
            const double c = (double)h[3 * nbins + b];
            double pm;
            memcpy(&pm, &h[b], 8);
            P[b] = c > 0 ? norm * pm * ((double)h[nbins + b] / FIX_P) / c : 0.0;
            if (kmean) kmean[b] = c > 0 ? 2.0 * M_PI / L * ((double)h[2 * nbins + b] / FIX_K) / c : 0.0;
            if (nmodes) nmodes[b] = (int64_t)h[3 * nbins + b];
        }
    } while (false);
    if (have_plan) fft.destroy(plan);
    cudaFree(in);
    cudaFree(F);
    cudaFree(part);
    cudaFree(bins);
    return rc;
}
