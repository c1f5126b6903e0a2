// The cells a carried certificate certifies, in a pass of their own before the general
// first pass (FP32 cells of a context that holds a previous diagram).
//
// Near convergence 95 to 99% of the cells keep their topology and their certificate. For
// them an evaluation is: planes at the new psi, vertices, the checks, the integrals. The
// general pass (process_cell) does that too, and this kernel does the same arithmetic in
// the same order (the geometry is the same inline code, the lengths and plane offsets name
// their roundings; a test compares the two passes bit for bit); but a block there waits for
// its slowest cell, and a cell whose topology broke is clipped from the box meanwhile. Here
// every cell does the same short work, and whatever does not fit it (a broken topology, a
// certificate that no longer holds, more than MAXF facets, a cell far from its frame) goes
// to a queue that the general pass then takes, from scratch: nothing is written before a
// cell is through.
//
// What bounds it: GB300 issues an FP64 warp instruction every 16 cycles of an SM, and the
// general path used about 120 a cell (the plane offsets, warp sums of four FP64 totals, a
// last FP64 step done by every lane). Here:
//  - a plane's offset 1/2 |d|^2 - d.z + psi_i - psi_j is summed in pairs of FP32 (48 bits)
//    from the exact fixed-point d and rounded once to FP32, as the FP64 sum was;
//  - facets and the certificate's seeds are built in one round of lanes;
//  - the four FP64 totals are summed together, six additions a lane, and finished one
//    quantity a lane.
// A vertex is compared with the stored supports and ball directly, so no bounds of the
// polytope are reduced; the faces' cycles come from a table of the dual edges, one
// lookup a step, where searching a face's entries took as many as it has vertices.
// 2.1 M cells, 99% carried: 5.0 ms, where the general pass took 20 ms; the late Newton step
// of that 129^3 box 53.0 -> 23.2 ms, of a 256^3 box 411 -> 177 ms.
#include "cell.cuh"

namespace sdot {

constexpr int CARRY_WARPS = 8;   // warps of a block
constexpr int CARRY_BLOCKS = 4;  // blocks per SM the registers are sized for
constexpr int MAXF = 26;         // facets (with the 6 box planes, one face a lane)
constexpr int NPL2 = MAXF + CERT_NEAR;  // planes: facets, then certificate seeds

struct CarryCell {
    V4<float> pl[NPL2];
    float plen[NPL2];
    float vx[TOPO], vy[TOPO], vz[TOPO];
    uint32_t start[MAXF];             // per face: lowest vertex slot << 8 | next plane
    uint16_t edge[MAXF * MAXF];       // dual edge x -> y: vertex slot | third plane << 8
    float sup[28];                    // stored supports less the margin
};

// s + e = a + b exactly (Knuth's two-sum)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
    return s;
}

// The cell's own seed and frame, every lane the same.
struct CarrySeed {
    int c[3];
    uint32_t io[3];
    float phi, plo;
    float zh[3], zl[3];  // frame origin as an FP32 pair (exact)
};

// plane_fix's offset, in FP64: the few planes whose offset the pair sum cannot round
static __device__ __noinline__ float plane_offset64(const ClipParams& cp, CarrySeed si, int32_t j) {
    SeedRef r;
    Frame f;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        r.c[a] = si.c[a];
        r.io[a] = si.io[a];
        f.z[a] = si.zh[a];
        f.zd[a] = (double)si.zh[a] + (double)si.zl[a];
    }
    r.phi = si.phi;
    r.plo = si.plo;
    float nx, ny, nz, w;
    plane_fix(cp, r, f, j, nx, ny, nz, w);
    return w;
}

// plane_fix in pairs of FP32, to the same bits: the normal's operations are the same; the
// offset's error before its one rounding is below 2^-43 of its terms, and where that could
// change the rounding (about one plane in 10^5) the FP64 sum decides. Returns false for a
// seed more than 256 grid cells away, whose difference does not fit the pair exactly.
__device__ __forceinline__ bool plane_pair(const ClipParams& cp, const CarrySeed& si, int32_t j,
                                           V4<float>& pn) {
    const int lc = cp.leafc[j];
    const uint4 oq = cp.ioff[j];
    const float pj = cp.posf[j].w, plj = cp.pslo[j];
    const int cj[3] = {lc & 1023, (lc >> 10) & 1023, (lc >> 20) & 1023};
    const uint32_t oj[3] = {oq.x, oq.y, oq.z};
    float d[3], th = 0.f, tl = 0.f, mag = fabsf(si.phi) + fabsf(pj);
    bool near = true;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        int dc = cj[a] - si.c[a];
        if (2 * dc > cp.G[a]) dc -= cp.G[a];
        else if (2 * dc < -cp.G[a]) dc += cp.G[a];
        long long di = ((long long)dc << 32) + (long long)oj[a] - (long long)si.io[a];
        const long long per = (long long)cp.G[a] << 32;
        if (2 * di > per) di -= per;
        else if (2 * di < -per) di += per;
        const int hi = (int)(di >> 16);
        near = near && abs(hi) <= (1 << 24);
        const float hf = (float)hi, lf = (float)(int)(di & 0xffff);
        const float h1 = cp.hfix[a], h16 = __fmul_rn(h1, 65536.f);
        d[a] = __fmul_rn(__fmaf_rn(hf, 65536.f, lf), h1);
        // d as a pair: two exact products
        const float p = __fmul_rn(hf, h16), q = __fmul_rn(lf, h1);
        float pq;
        const float dh = two_sum(p, q, pq);
        const float dl = __fadd_rn(pq, __fadd_rn(__fmaf_rn(hf, h16, -p), __fmaf_rn(lf, h1, -q)));
        // u = d / 2 - z
        float ue;
        const float uh = two_sum(__fmul_rn(0.5f, dh), -si.zh[a], ue);
        const float ul = __fadd_rn(ue, __fmaf_rn(0.5f, dl, -si.zl[a]));
        // t += d u
        const float m = __fmul_rn(dh, uh);
        const float me = __fmaf_rn(dl, uh, __fmaf_rn(dh, ul, __fmaf_rn(dh, uh, -m)));
        mag += fabsf(m) + 0.5f * dh * dh;
        float se;
        th = two_sum(th, m, se);
        tl = __fadd_rn(tl, __fadd_rn(se, me));
    }
    float pe, se;
    const float ph = two_sum(si.phi, -pj, pe);
    th = two_sum(th, ph, se);
    tl = __fadd_rn(tl, __fadd_rn(__fadd_rn(se, pe), __fsub_rn(si.plo, plj)));
    pn.x = d[0];
    pn.y = d[1];
    pn.z = d[2];
    const float err = 1.2e-13f * mag;
    pn.w = __fadd_rn(th, __fadd_rn(tl, err));
    if (pn.w != __fadd_rn(th, __fsub_rn(tl, err))) pn.w = plane_offset64(cp, si, j);
    return near;
}

__device__ __forceinline__ float redux_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
__device__ __forceinline__ float redux_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Sums of four quantities over the warp: lane l ends with the sum of quantity l >> 3.
template <typename T>
__device__ __forceinline__ T warp_sum4(T v0, T v1, T v2, T v3, int lane) {
    const bool hi = lane & 16;
    T a = hi ? v2 : v0, b = hi ? v3 : v1;
    a += __shfl_xor_sync(FULLMASK, hi ? v0 : v2, 16);
    b += __shfl_xor_sync(FULLMASK, hi ? v1 : v3, 16);
    const bool up = lane & 8;
    T s = up ? b : a;
    s += __shfl_xor_sync(FULLMASK, up ? a : b, 8);
    s += __shfl_xor_sync(FULLMASK, s, 4);
    s += __shfl_xor_sync(FULLMASK, s, 2);
    s += __shfl_xor_sync(FULLMASK, s, 1);
    return s;
}

// One cell; false: it goes to the general pass (nothing was written).
__device__ __forceinline__ bool carry_cell(CarryCell& S, const ClipParams& cp, int64_t i,
                                           float cons, const float* snap, float halfLmin,
                                           float psimax_glob, int lane) {
    const int nc = cp.cert_n[i], nf = cp.fcnt[i], nt = cp.topo_n[i];
    if (nc > CERT_NEAR || nf < 4 || nf > MAXF || nt < 4 || nt > TOPO) return false;
    const float* cf = cp.cert_f + i * CERT_F;
    const float Mn = __fsub_rd(cf[4], cons), Wn = __fsub_rd(cf[5], cons);
    if (!(cons >= 0.f && Wn >= 0.f)) return false;
    // the cell's seed and frame (load_cell's)
    CarrySeed si;
    {
        float z[3];
#pragma unroll
        for (int a = 0; a < 3; a++) z[a] = cp.anchor[3 * i + a];
        if (!(isfinite(z[0]) && isfinite(z[1]) && isfinite(z[2]))) z[0] = z[1] = z[2] = 0.f;
        const int lc = cp.leafc[i];
        const uint4 q = cp.ioff[i];
        si.io[0] = q.x;
        si.io[1] = q.y;
        si.io[2] = q.z;
        si.phi = cp.posf[i].w;
        si.plo = cp.pslo[i];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            si.c[a] = (lc >> (10 * a)) & 1023;
            const float za = fminf(fmaxf(z[a], -cp.halfLt[a]), cp.halfLt[a]);
            // a multiple of ht / 4096, which the pair holds exactly
            const float r = rintf(za * snap[a]), q1 = cp.ht[a] * (1.f / 4096.f);
            si.zh[a] = __fmul_rn(r, q1);
            si.zl[a] = __fmaf_rn(r, q1, -si.zh[a]);
        }
    }
    // planes: lane k < nf the facets, then the certificate's seeds
    const int np = nf + nc;
    bool ok = true;
    for (int k = lane; k < np; k += 32) {
        const int32_t j = k < nf ? cp.fcol[i * FCAP + k] : cp.cert_j[i * CERT_NEAR + k - nf];
        V4<float> pn;
        pn.x = pn.y = pn.z = pn.w = 0.f;
        if (j >= 0 && j < cp.N && j != (int32_t)i) ok = plane_pair(cp, si, j, pn) && ok;
        else ok = false;
        S.pl[k] = pn;
        S.plen[k] = length3(pn.x, pn.y, pn.z);
    }
    if (lane < 27)
        S.sup[lane] = lane == 13 ? INFINITY
                                 : __fsub_rn(__half2float(__ushort_as_half(
                                                 cp.cert_s[i * CERT_S + lane])),
                                             1e-5f);
    if (lane < nf) S.start[lane] = 0xffffffffu;
    for (int q = lane; q < nf * MAXF / 2; q += 32) reinterpret_cast<uint32_t*>(S.edge)[q] = ~0u;
    __syncwarp();
    // vertices, one or two a lane: the point of three planes, well conditioned, inside
    // every other facet and every seed of the certificate (the exact tests of topo_init and
    // cert_check), inside the stored ball and below the stored supports
    bool ill = false;
    float r0 = 0.f;
    float mn[3] = {1e30f, 1e30f, 1e30f}, mx[3] = {-1e30f, -1e30f, -1e30f};
    const float z0 = si.zh[0], z1 = si.zh[1], z2 = si.zh[2];
    {
        const float c0 = cf[0], c1 = cf[1], c2 = cf[2];
        const float Rt = (cf[3] - 1.1e-5f) * (1.f - 2e-6f), R2 = Rt > 0.f ? Rt * Rt : -1.f;
        for (int s = lane; s < nt; s += 32) {
            const uint32_t t = cp.topo[i * TOPO + s];
            const uint32_t a = (t & 0xff) - 6, b = ((t >> 8) & 0xff) - 6, c = ((t >> 16) & 0xff) - 6;
            if (a >= (uint32_t)nf || b >= (uint32_t)nf || c >= (uint32_t)nf) {  // box planes too
                ok = false;
                continue;
            }
            const V4<float> A = S.pl[a], Bq = S.pl[b], Cq = S.pl[c];
            bool well;
            const V3<float> v =
                vertex_of3(A, Bq, Cq, S.plen[a], S.plen[b], S.plen[c], 1e-3f, well);
            ill |= nearly_parallel(A, Bq) || nearly_parallel(Bq, Cq) || nearly_parallel(Cq, A);
            if (!well || !(isfinite(v.x) && isfinite(v.y) && isfinite(v.z))) ok = false;
            S.vx[s] = v.x;
            S.vy[s] = v.y;
            S.vz[s] = v.z;
            mn[0] = fminf(mn[0], v.x);
            mn[1] = fminf(mn[1], v.y);
            mn[2] = fminf(mn[2], v.z);
            mx[0] = fmaxf(mx[0], v.x);
            mx[1] = fmaxf(mx[1], v.y);
            mx[2] = fmaxf(mx[2], v.z);
            // the dual edges and, per face, the lowest vertex
            S.edge[a * MAXF + b] = (uint16_t)(s | (c << 8));
            S.edge[b * MAXF + c] = (uint16_t)(s | (a << 8));
            S.edge[c * MAXF + a] = (uint16_t)(s | (b << 8));
            atomicMin(&S.start[a], ((uint32_t)s << 8) | c);
            atomicMin(&S.start[b], ((uint32_t)s << 8) | a);
            atomicMin(&S.start[c], ((uint32_t)s << 8) | b);
            const float x = v.x + z0, y = v.y + z1, z = v.z + z2;
            const float m2 = fmaf(x, x, fmaf(y, y, z * z));
            r0 = fmaxf(r0, m2);
            if (!(0.5f * m2 * 1.0001f + 1e-6f <= Mn)) ok = false;
            const float dx = x - c0, dy = y - c1, dz = z - c2;
            if (!(dx * dx + dy * dy + dz * dz <= R2)) ok = false;
            // direction (ux, uy, uz) at (ux + 1) + 3 (uy + 1) + 9 (uz + 1)
#pragma unroll
            for (int k = 14; k < 27; k++) {
                const int ux = k % 3 - 1, uy = (k / 3) % 3 - 1, uz = k / 9 - 1;
                const float h = fmaf((float)ux, x, fmaf((float)uy, y, (float)uz * z));
                if (!(h <= S.sup[k] && -h <= S.sup[26 - k])) ok = false;
            }
#pragma unroll 2
            for (int q = 0; q < np; q++) {
                float sd;
                if (beyond(v, S.pl[q], S.plen[q], sd) && q != (int)a && q != (int)b && q != (int)c)
                    ok = false;
            }
        }
    }
    if (!__all_sync(FULLMASK, ok)) return false;
    // the cell must stay inside the minimum-image range (cell_too_large)
    {
        const float R0 = sqrtf(redux_max(r0));
        const float dpsi = fmaxf(psimax_glob - si.phi, 0.f);
        if (R0 + sqrtf(R0 * R0 + 2.f * dpsi) > halfLmin * 0.9999f) return false;
    }
    float o[3];
#pragma unroll
    for (int a = 0; a < 3; a++) o[a] = 0.5f * (redux_min(mn[a]) + redux_max(mx[a]));
    ill = __any_sync(FULLMASK, ill);
    __syncwarp();
    // one face a lane: the fan of its lowest vertex, along the cycle of the dual edges.
    // Facet f is on lane 6 + f, where integrate has it (its slot, after the 6 box planes), so
    // that the sums over the lanes below are integrate's in its order.
    const int f = lane - 6;
    const bool face = f >= 0 && f < nf;
    float fv6 = 0.f, fmx = 0.f, fmy = 0.f, fmz = 0.f, Sx = 0.f, Sy = 0.f, Sz = 0.f;
    int steps = 0;
    float coef = -1.f;
    float A = 0.f;
    if (face) {
        const uint32_t st = S.start[f];
        if (st == 0xffffffffu) {
            ok = false;
        } else {
            const int s0 = (int)(st >> 8);
            uint32_t y = st & 0xff;
            V3<float> v0;
            v0.x = S.vx[s0] - o[0];
            v0.y = S.vy[s0] - o[1];
            v0.z = S.vz[s0] - o[2];
            V3<float> vp = v0;
            for (steps = 1; steps <= nt; steps++) {
                const uint32_t e = S.edge[f * MAXF + y];
                if (e == 0xffffu) {
                    ok = false;
                    break;
                }
                const int s = (int)(e & 0xff);
                if (s == s0) break;
                y = e >> 8;
                V3<float> vc;
                vc.x = S.vx[s] - o[0];
                vc.y = S.vy[s] - o[1];
                vc.z = S.vz[s] - o[2];
                if (steps >= 2)
                    fan_triangle(v0, vp, vc, Sx, Sy, Sz, fv6, fmx, fmy, fmz);
                vp = vc;
            }
            const float ax2 = 0.5f * Sx, ay2 = 0.5f * Sy, az2 = 0.5f * Sz;
            A = length3(ax2, ay2, az2);
            Sx = ax2;
            Sy = ay2;
            Sz = az2;
            coef = A / S.plen[f];
            if (steps < 3 || !(A > 0.f)) ok = false;  // fewer facets than the topology has
        }
    }
    // every vertex on each of its three faces exactly once
    if (__reduce_add_sync(FULLMASK, steps) != 3 * nt) ok = false;
    if (!__all_sync(FULLMASK, ok)) return false;
    const float cs = warp_sum4(Sx, Sy, Sz, A, lane);
    const float sx = __shfl_sync(FULLMASK, cs, 0), sy = __shfl_sync(FULLMASK, cs, 8),
                sz = __shfl_sync(FULLMASK, cs, 16), sabs = __shfl_sync(FULLMASK, cs, 24);
    const bool bad = ill || !(length3(sx, sy, sz) <= 1e-4f * sabs);
    // totals, one quantity a lane: volume, then the moment about o carried to the seed
    const int quant = lane >> 3, ax = quant > 0 ? quant - 1 : 0;
    const double tot = warp_sum4((double)fv6, (double)fmx, (double)fmy, (double)fmz, lane);
    const double vol = __shfl_sync(FULLMASK, tot, 0) * (1.0 / 6.0);
    const float zh = ax == 0 ? si.zh[0] : (ax == 1 ? si.zh[1] : si.zh[2]);
    const float zl = ax == 0 ? si.zl[0] : (ax == 1 ? si.zl[1] : si.zl[2]);
    const float oa = ax == 0 ? o[0] : (ax == 1 ? o[1] : o[2]);
    const double off = ((double)zh + (double)zl) + (double)oa;
    const double mom = fma(24.0 * off, vol, tot) * (1.0 / 24.0);
    const float fv = (float)vol;
    if (!(fv > 0.f && isfinite(fv))) return false;
    const float cen = (float)mom / fv;
    // a cell this far from its frame is clipped again by the general pass
    {
        const float zf = zh;
        const float dc = quant > 0 ? cen - zf : 0.f;
        const float d0 = __shfl_sync(FULLMASK, dc, 8), d1 = __shfl_sync(FULLMASK, dc, 16),
                    d2 = __shfl_sync(FULLMASK, dc, 24);
        float dz2 = 0.f;
        dz2 += d0 * d0;
        dz2 += d1 * d1;
        dz2 += d2 * d2;
        if (dz2 > REFRAME_DIST * REFRAME_DIST) return false;
    }
    // outputs (the facet list, the topology and their counts stay as they are)
    if (face) cp.fval[i * FCAP + f] = (double)coef * cp.a;
    if ((lane & 7) == 0) {
        const double a3 = cp.a * cp.a * cp.a;
        if (quant == 0) {
            cp.vol[i] = vol * a3;
            float* c = cp.cert_f + i * CERT_F;
            c[4] = Mn;
            c[5] = Wn;
            cp.status[i] = (uint8_t)(bad ? CS_INCONSISTENT : CS_OK);
            if (bad) cp.q64_out[atomicAdd(cp.q64_cnt, 1)] = (int32_t)i;
        } else {
            cp.m1[3 * i + ax] = mom * (a3 * cp.a);
            cp.anchor[3 * i + ax] = cen;
        }
    }
    return true;
}

// cells of the context to queue (count cnt): those the general pass has to take
__global__ void __launch_bounds__(CARRY_WARPS * 32, CARRY_BLOCKS)
    carry_kernel(const __grid_constant__ ClipParams cp, int32_t* __restrict__ queue,
                 int32_t* __restrict__ cnt, int32_t* __restrict__ work) {
    __shared__ CarryCell cells[CARRY_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float cons = __fadd_ru(__fsub_ru(ord2f(cp.cert_dpsi[0]), ord2f(cp.cert_dpsi[1])), 1e-6f);
    if (!(cons <= CERT_ETA)) {  // no certificate outlives this change of psi
        const int64_t step = (int64_t)gridDim.x * blockDim.x;
        const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        for (int64_t t = t0; t < cp.N; t += step) queue[t] = (int32_t)t;
        if (t0 == 0) *cnt = (int32_t)cp.N;
        return;
    }
    const float psimax_glob = top_psimax(cp, lane);
    const float halfLmin = 0.5f * fminf(cp.Lt[0], fminf(cp.Lt[1], cp.Lt[2]));
    const float snap[3] = {4096.f / cp.ht[0], 4096.f / cp.ht[1], 4096.f / cp.ht[2]};
    int carried = 0;
    while (true) {
        int64_t i = 0;
        if (lane == 0) i = atomicAdd(work, 1);
        i = __shfl_sync(FULLMASK, i, 0);
        if (i >= cp.N) break;
        if (carry_cell(cells[warp], cp, i, cons, snap, halfLmin, psimax_glob, lane)) carried++;
        else if (lane == 0) queue[atomicAdd(cnt, 1)] = (int32_t)i;
        __syncwarp();
    }
    if (lane == 0 && carried) atomicAdd(cp.cert_carried, carried);
}

int launch_carry(const ClipParams& cp, int32_t* queue, int32_t* cnt, int32_t* work, cudaStream_t s) {
    const int64_t need = (cp.N + CARRY_WARPS - 1) / CARRY_WARPS;
    const int64_t most = (int64_t)CARRY_BLOCKS * num_sms();
    carry_kernel<<<(unsigned)(need < most ? need : most), CARRY_WARPS * 32, 0, s>>>(cp, queue, cnt,
                                                                                  work);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    return SDOT_OK;
}

}  // namespace sdot
