// After the solve: the Kantorovich potential at tau_I on a mesh and the mass density of
// the cells moved to an intermediate time (Sec. "Monge-Ampere-Kantorovich
// Reconstruction", the Legendre transform of psi and the last paragraph; Fig. 1).
//
//  - phi_I(q) = min_i [1/2 |q - x_i|^2 - psi_i], attained in the Laguerre cell i(q) that
//    contains q: every cell claims the mesh points inside it (planes tested with a small
//    tolerance, so a point on a facet is claimed by both cells), the smallest value of
//    its own 1/2 |q - x_i|^2 - psi_i wins (integer atomic minimum on the value's ordered
//    bits), then the claimants holding exactly that value take the owner by an integer
//    minimum on their (caller) index. The value is computed in the order
//    ((dx^2 + dy^2) + dz^2) / 2 - psi_i with correctly rounded operations.
//  - The Zel'dovich map q -> q + lambda (x_i - q) (lambda = D(tau)/D(tau_F)) shrinks cell
//    i about x_i by 1 - lambda and carries its mass nu_i uniformly. The mass of voxel v
//    is sum_i nu_i |V_i cap h_i^-1(v)| / |V_i| with h_i that homothety: each cell is
//    clipped by the six planes of every pulled-back voxel its moved bounding box meets.
//    The masses are summed in 64-bit fixed point (unit: 2^-62 of the box's mass, so no
//    voxel can overflow), so the sum does not depend on the order of the atomic
//    additions.
//
// One warp per cell. The cell is rebuilt in FP64 (seed frame) from its stored topology, or
// from the facets of the context's last evaluation, which are its complete neighbour set.
//
// What bounds it is the chain of one warp's instructions, 7 warps an SM (12 cycles an
// instruction, 3 of them fetching it; the FP64 pipe, a warp instruction every 16 cycles of an
// SM, is 53% busy), so:
//  - a cell is cut into z slabs, those into y slabs, and a y slab by the x planes from the
//    top down in place, each piece the difference of two volumes: about 13 clips and 11
//    volumes for a cell that meets 2.2 voxels an axis, where every voxel's six planes cut a
//    copy of the whole cell (64 clips);
//  - a volume is a sum over the vertices and their three faces, with no chain along a face,
//    of three FP64 operations each (mesh_volume);
//  - a mesh point is tested against the planes in FP32, in FP64 only where that is too
//    close to say;
//  - the owner needs no second pass unless some point was claimed twice.
// 110,592 cells, 96^3 points and voxels: 49.4 ms with the six planes of every voxel, 11.4 now.
// Error of the density against exact clipping, 12^3 cells: the unit of |box| / 2^62 in which
// masses are added, 7e-16 rms on 16^3 voxels, as with the six planes.
#include <math.h>

#include <string>

#include "cell.cuh"

namespace sdot {

struct MeshParams {
    int M;                           // mesh points (voxels) per axis
    int pass;                        // 0: deposit, phi minimum, owner; 1: owner only
    double s;                        // 1 - lambda
    double h[3], inv_h[3];           // voxel size, its inverse
    double inv_unit;                 // 1 / fixed-point unit of the voxel masses
    const double* nu;                // masses (sorted order)
    const double* centre;            // 3 M: voxel centres (m + 1/2) L / M per axis
    unsigned long long* mass_fx;     // M^3 voxel masses (fixed point), or null
    unsigned long long* phi_ord;     // M^3 ordered bits of phi, or null
    int32_t* owner;                  // M^3 owner (caller index), or null
    int32_t* flags;                  // [0] cells that could not be rebuilt
    int32_t* twice;                  // set when a point is claimed by two cells
    int32_t* work;                   // work counter
    int32_t* rest;                   // cells for the large polytopes
    int32_t* nrest;                  // their number
};

__device__ __forceinline__ unsigned long long d2ord(double f) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(f);
    return (u & 0x8000000000000000ull) ? ~u : (u | 0x8000000000000000ull);
}
__device__ __forceinline__ double ord2d(unsigned long long u) {
    return __longlong_as_double(
        (long long)((u & 0x8000000000000000ull) ? (u & 0x7fffffffffffffffull) : ~u));
}
// (a cell lies within a box of its seed, so voxel indices are between -M and 2 M)
__device__ __forceinline__ int wrap_index(int v, int M) {
    const int r = v % M;
    return r < 0 ? r + M : r;
}
// minimum-image component, the rule of the oracle: if dx > L/2 subtract L, else if
// dx < -L/2 add L
__device__ __forceinline__ double wrap_rn(double dx, double L) {
    if (dx > __dmul_rn(0.5, L)) return __dsub_rn(dx, L);
    if (dx < -__dmul_rn(0.5, L)) return __dadd_rn(dx, L);
    return dx;
}

// Polytopes of a cell with at most MESH_MAXF facets: with the six voxel planes it has at most
// 32 faces, so 60 vertices, and no clip can overflow. Other cells go to the large ones.
using MeshCap = Cap<64, 128, 8>;
constexpr int MESH_MAXF = 26;

// a plane's axis and side
__device__ __forceinline__ int32_t mesh_tag(int a, bool up) { return a | (up ? 0 : 4); }

// volume of polytope slot about its frame origin (units of a^3). Every lane gets the value.
// Faces are scaled to n_a = +-1 along their axis a, which pj holds (mesh_tag): 6 V is the sum
// over the faces of +-w times twice the face's area seen along a, a sum of cross products of
// consecutive vertices in two coordinates (three FP64 operations a vertex and face).
// NaN when the faces' cycles do not close: every entry of a face has to follow exactly one
// other (rounding in near-degenerate clips can leave a vertex list that is no polytope).
template <class C>
__device__ __noinline__ double mesh_volume(int slot, int lane) {
    Poly<double, C>& P = poly_at<double, C>(slot);
    const int nt = P.nt, np = P.np;
    for (int f = lane; f < np; f += 32) P.fend[f] = 0u;
    __syncwarp();
    for (int s = lane; s < nt; s += 32) {
        const uint32_t t = P.tri[s];
        atomicAdd(&P.fend[t & 0xff], 1u);
        atomicAdd(&P.fend[(t >> 8) & 0xff], 1u);
        atomicAdd(&P.fend[(t >> 16) & 0xff], 1u);
    }
    __syncwarp();
    {
        uint32_t carry = 0;
        for (int f0 = 0; f0 < np; f0 += 32) {
            const int f = f0 + lane;
            const uint32_t c = f < np ? P.fend[f] : 0u;
            uint32_t incl = c;
            for (int q = 1; q < 32; q <<= 1) {
                const uint32_t y = __shfl_up_sync(FULLMASK, incl, q);
                if (lane >= q) incl += y;
            }
            if (f < np) P.fend[f] = carry + incl - c;  // start, advanced by the fill
            carry += __shfl_sync(FULLMASK, incl, 31);
        }
    }
    __syncwarp();
    for (int s = lane; s < nt; s += 32) {
        const uint32_t t = P.tri[s];
        const uint32_t a = t & 0xff, b = (t >> 8) & 0xff, c = (t >> 16) & 0xff;
        const uint32_t sv = (uint32_t)s << 16;
        P.fent[atomicAdd(&P.fend[a], 1u)] = b | (c << 8) | sv;
        P.fent[atomicAdd(&P.fend[b], 1u)] = c | (a << 8) | sv;
        P.fent[atomicAdd(&P.fend[c], 1u)] = a | (b << 8) | sv;
    }
    __syncwarp();
    double v6 = 0.0;
    bool ok = true;
    unsigned taken = 0;  // sum of the entries that follow one
    for (int s0 = 0; s0 < nt; s0 += 32) {
        const int s = s0 + lane;
        const bool act = s < nt;
        const uint32_t t = act ? P.tri[s] : 0u;
#pragma unroll 1
        for (int e = 0; e < 3; e++) {
            const uint32_t f = (t >> (8 * e)) & 0xff, y = (t >> (8 * ((e + 2) % 3))) & 0xff;
            // the next vertex of face f after s: its entry's first plane is y
            int q = f > 0 ? (int)P.fend[f - 1] : 0;
            const int end = act ? (int)P.fend[f] : 0;
            while (q < end && (P.fent[q] & 0xff) != y) q++;
            __syncwarp();  // the lanes part in the search; the FP64 work is for all of them
            const bool some = q < end;
            ok = ok && (some || !act);
            taken += some ? q : 0;
            const int tag = P.pj[f], a = tag & 3;
            const int v = act ? s : 0, w = some ? (int)(P.fent[q] >> 16) : 0;
            const double* u1 = a == 0 ? P.vy : (a == 1 ? P.vz : P.vx);
            const double* u2 = a == 0 ? P.vz : (a == 1 ? P.vx : P.vy);
            const double d = u1[v] * u2[w] - u2[v] * u1[w], h = P.pl[f].w;
            if (some) v6 = fma(tag & 4 ? -h : h, d, v6);
        }
    }
    v6 = warp_sum(v6);
    const unsigned n3 = 3u * (unsigned)nt;
    ok = __reduce_add_sync(FULLMASK, taken) == n3 * (n3 - 1) / 2 && ok;
    return __all_sync(FULLMASK, ok) ? v6 * (1.0 / 6.0) : NAN;
}

// bounds of the vertices along an axis, in FP32, a little outside
template <class C>
__device__ __forceinline__ void mesh_extent(int slot, int a, int lane, float& lo, float& hi) {
    const Poly<double, C>& P = poly_at<double, C>(slot);
    const double* x = a == 0 ? P.vx : (a == 1 ? P.vy : P.vz);
    uint32_t l = 0xffffffffu, h = 0u;
    for (int s = lane; s < P.nt; s += 32) {
        const uint32_t u = f2ord((float)x[s]);
        l = min(l, u);
        h = max(h, u);
    }
    lo = ord2f(__reduce_min_sync(FULLMASK, l));
    hi = ord2f(__reduce_max_sync(FULLMASK, h));
    const float m = 1e-6f * (fabsf(lo) + fabsf(hi)) + 1e-9f;
    lo -= m;
    hi += m;
}

// clip polytope slot by x_a <= b (up) or x_a >= b; false when nothing is left or, with bad
// set, when the clip failed. A plane within rounding of a facet, edge or cluster of vertices
// can be refused (CLIP_TWICE): it is then moved aside by SHIFT, twice that, and so on (units
// of a; the tolerance of beyond is 1e-13 of the terms) until it clears them.
constexpr double SHIFT = 4e-13;
template <class C>
__device__ __forceinline__ bool mesh_cut(int slot, int a, double b, bool up, int lane, bool& bad,
                                         bool* cut = nullptr) {
    V4<double> pn;
    const double sg = up ? 1.0 : -1.0;
    pn.x = a == 0 ? sg : 0.0;
    pn.y = a == 1 ? sg : 0.0;
    pn.z = a == 2 ? sg : 0.0;
    pn.w = sg * b;
    int r = poly_clip_once<double, C>(slot, pn, 1.0, mesh_tag(a, up), lane);
    for (int k = 0; r == CLIP_TWICE && k < 14; k++) {
        pn.w = sg * (b + (k & 1 ? -SHIFT : SHIFT) * (double)(1 << (k >> 1)));
        r = poly_clip_once<double, C>(slot, pn, 1.0, mesh_tag(a, up), lane);
    }
    if (r == CLIP_TWICE) r = CLIP_CAP;
    if (cut) *cut = r != CLIP_NONE;
    if ((r & CLIP_BAD) || r == CLIP_CAP) bad = true;
    return r != CLIP_EMPTY && r != CLIP_CAP;
}

template <class C>
__global__ void __launch_bounds__(32)
    mesh_kernel(const __grid_constant__ ClipParams cp, const __grid_constant__ MeshParams mp) {
    constexpr bool BIG = C::MP > MeshCap::MP;
    __shared__ float4 plf[C::MP];  // the cell's planes in FP32
    const int lane = threadIdx.x & 31;
    constexpr int ps = 0, zs = 1, ys = 2;  // the cell, a z slab, a y slab of that
    Poly<double, C>& P = poly_at<double, C>(ps);
    const int M = mp.M;
    const int64_t nwork = BIG ? (int64_t)*mp.nrest : cp.N;
    while (true) {
        int64_t i = 0;
        if (lane == 0) i = atomicAdd(mp.work, 1);
        i = __shfl_sync(FULLMASK, i, 0);
        if (i >= nwork) break;
        if (BIG) i = mp.rest[i];
        const int nf = min(cp.fcnt[i], FCAP), ntopo = cp.topo_n[i];
        bool built = BIG || nf <= MESH_MAXF;
        if (built) {
            load_cell<double, C>(ps, cp, i, lane);
            if (!(ntopo > 0 && topo_init<double, C>(ps, cp, nf, ntopo, lane))) {
                poly_init<double, C>(ps, cp, lane);
                built = clip_list<double, C>(ps, cp, cp.fcol + i * FCAP, nf, lane) == CLIP_NONE;
            }
        }
        if (!built) {
            if (lane == 0) {
                if (BIG) atomicAdd(mp.flags, 1);
                else mp.rest[atomicAdd(mp.nrest, 1)] = (int32_t)i;
            }
            continue;
        }
        const CellCtx& cc = P.cc;
        const double y[3] = {cc.yi.x, cc.yi.y, cc.yi.z};
        const double psii = cc.psii;
        const int32_t caller = (int32_t)cc.yi.w;
        // bounds of the cell (seed frame, units of a)
        float lo[3], hi[3];
#pragma unroll
        for (int a = 0; a < 3; a++) mesh_extent<C>(ps, a, lane, lo[a], hi[a]);
        // --- point location: the mesh points inside the cell --------------------------
        if (mp.phi_ord) {
            const int np = P.np;
            __syncwarp();
            for (int k = lane; k < np; k += 32)
                plf[k] = make_float4((float)P.pl[k].x, (float)P.pl[k].y, (float)P.pl[k].z,
                                     (float)P.pl[k].w);
            __syncwarp();
            long long m0[3];
            int cnt[3];
            float p0[3], hs[3];
            bool any = true;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                m0[a] = (long long)ceil((y[a] + cp.a * (double)lo[a]) / mp.h[a] - 0.5);
                const long long m1 =
                    (long long)floor((y[a] + cp.a * (double)hi[a]) / mp.h[a] - 0.5);
                cnt[a] = (int)(m1 - m0[a] + 1);
                any = any && m1 >= m0[a];
                p0[a] = (float)((((double)m0[a] + 0.5) * mp.h[a] - y[a]) * cp.inv_a);
                hs[a] = (float)(mp.h[a] * cp.inv_a);
            }
            // the largest coordinate that enters, whose rounding the FP32 test allows for
            float ext = 0.f;
#pragma unroll
            for (int a = 0; a < 3; a++) ext = fmaxf(ext, fmaxf(fabsf(lo[a]), fabsf(hi[a])) + hs[a]);
            const long long npts = any ? (long long)cnt[0] * cnt[1] * cnt[2] : 0;
            for (long long t = lane; t < npts; t += 32) {
                const int tz = (int)(t / (cnt[0] * cnt[1]));
                const int tr = (int)(t - (long long)tz * cnt[0] * cnt[1]);
                const int ty = tr / cnt[0], tx = tr - ty * cnt[0];
                // FP32: outside, inside, or too close to some plane to say
                const float fx = p0[0] + (float)tx * hs[0], fy = p0[1] + (float)ty * hs[1],
                            fz = p0[2] + (float)tz * hs[2];
                bool in = true, close = false;
                for (int k = 0; k < np; k++) {
                    const float4 pl = plf[k];
                    const float sd = pl.x * fx + pl.y * fy + pl.z * fz - pl.w;
                    const float tol =
                        4e-6f * (fabsf(pl.w) + (fabsf(pl.x) + fabsf(pl.y) + fabsf(pl.z)) * ext);
                    if (sd > tol) {
                        in = false;
                        break;
                    }
                    close |= sd > -tol;
                }
                if (!in) continue;
                int w[3];
                double p[3];
                const int tt[3] = {tx, ty, tz};
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    w[a] = wrap_index((int)m0[a] + tt[a], M);
                    p[a] = wrap_rn(__dsub_rn(mp.centre[a * M + w[a]], y[a]), cp.L[a]);
                }
                if (close) {
                    // inside every plane of the cell (units of a), with a tolerance of the
                    // terms involved
                    const double pa[3] = {p[0] * cp.inv_a, p[1] * cp.inv_a, p[2] * cp.inv_a};
                    for (int k = 0; k < np && in; k++) {
                        const V4<double> pl = P.pl[k];
                        const double sd = pa[0] * pl.x + pa[1] * pl.y + pa[2] * pl.z - pl.w;
                        const double sc =
                            fabs(pl.w) +
                            P.plen[k] * (fabs(pa[0]) + fabs(pa[1]) + fabs(pa[2]));
                        if (sd > 1e-12 * sc) in = false;
                    }
                    if (!in) continue;
                }
                double s2 = 0.0;
#pragma unroll
                for (int a = 0; a < 3; a++) s2 = __dadd_rn(s2, __dmul_rn(p[a], p[a]));
                const double f = __dsub_rn(__dmul_rn(0.5, s2), psii);
                const int64_t m = ((int64_t)w[2] * M + w[1]) * M + w[0];
                if (mp.pass == 0) {
                    atomicMin(&mp.phi_ord[m], d2ord(f));
                    if (mp.owner && atomicMin(&mp.owner[m], caller) != INT32_MAX) *mp.twice = 1;
                } else if (mp.phi_ord[m] == d2ord(f)) {
                    atomicMin(&mp.owner[m], caller);
                }
            }
        }
        if (mp.pass != 0 || !mp.mass_fx) continue;
        // --- deposit: the cell in the slabs of every pulled-back voxel it meets ---------
        // the frame moves to the centre of the bounds, so that the volumes' terms are of
        // the cell's own size
        double c[3];
#pragma unroll
        for (int a = 0; a < 3; a++) c[a] = 0.5 * ((double)lo[a] + (double)hi[a]);
        __syncwarp();
        for (int s = lane; s < P.nt; s += 32) {
            P.vx[s] -= c[0];
            P.vy[s] -= c[1];
            P.vz[s] -= c[2];
        }
        // and the planes are scaled to a largest component of 1 (mesh_volume)
        for (int k = lane; k < P.np; k += 32) {
            V4<double> n = P.pl[k];
            // (the high words decide: the others stay below 1 + 1e-6)
            const int hx = __double2hiint(n.x) & INT32_MAX, hy = __double2hiint(n.y) & INT32_MAX,
                      hz = __double2hiint(n.z) & INT32_MAX;
            const int a = hx >= hy && hx >= hz ? 0 : (hy >= hz ? 1 : 2);
            const double sc = 1.0 / fabs(a == 0 ? n.x : (a == 1 ? n.y : n.z));
            n.w = (n.w - (n.x * c[0] + n.y * c[1] + n.z * c[2])) * sc;
            n.x = a == 0 ? copysign(1.0, n.x) : n.x * sc;
            n.y = a == 1 ? copysign(1.0, n.y) : n.y * sc;
            n.z = a == 2 ? copysign(1.0, n.z) : n.z * sc;
            P.pl[k] = n;
            P.plen[k] *= sc;
            P.pj[k] = mesh_tag(a, (a == 0 ? n.x : (a == 1 ? n.y : n.z)) > 0.0);
        }
        __syncwarp();
        const double volP = mesh_volume<C>(ps, lane);
        if (!(volP > 0.0)) {
            if (lane == 0) atomicAdd(mp.flags, 1);
            continue;
        }
        // voxel edge v along axis a, pulled back to the cell's frame. The difference v h - y
        // comes first: scaled apart, the two lose what they cancel (N^(1/3) units in the
        // last place of a, and the masses on the plane's two sides with it)
        const double ks = 1.0 / (mp.s * cp.a);
        auto edge = [&](int a, int v) { return fma((double)v, mp.h[a], -y[a]) * ks - c[a]; };
        auto range = [&](int slot, int a, int& va, int& vb) {
            float l, h;
            mesh_extent<C>(slot, a, lane, l, h);
            const double sa = mp.s * cp.a;
            // (l and h lie outside by far more than the rounding of the product)
            va = (int)floor(fma((double)l + c[a], sa, y[a]) * mp.inv_h[a]);
            vb = (int)floor(fma((double)h + c[a], sa, y[a]) * mp.inv_h[a]);
        };
        const double unit = mp.nu[i] / volP * mp.inv_unit;  // fixed-point mass per volume
        bool bad = false;
        int z0, z1;
        range(ps, 2, z0, z1);
        // (a cell in one slab is cut in place)
        const int zq = z0 < z1 ? zs : ps;
        for (int vz = z0; vz <= z1; vz++) {
            if (z0 < z1) poly_copy<double, C>(zs, ps, lane);
            if (vz > z0 && !mesh_cut<C>(zs, 2, edge(2, vz), false, lane, bad)) continue;
            if (vz < z1 && !mesh_cut<C>(zs, 2, edge(2, vz + 1), true, lane, bad))
                continue;
            int y0, y1;
            range(zq, 1, y0, y1);
            const int yq = y0 < y1 ? ys : zq;
            for (int vy = y0; vy <= y1; vy++) {
                if (y0 < y1) poly_copy<double, C>(ys, zq, lane);
                if (vy > y0 && !mesh_cut<C>(ys, 1, edge(1, vy), false, lane, bad))
                    continue;
                if (vy < y1 &&
                    !mesh_cut<C>(ys, 1, edge(1, vy + 1), true, lane, bad))
                    continue;
                int x0, x1;
                range(yq, 0, x0, x1);
                const int64_t row = ((int64_t)wrap_index(vz, M) * M + wrap_index(vy, M)) * M;
                // volume below the next plane (of the whole cell, where nothing was cut yet)
                double left = z0 == z1 && y0 == y1 ? volP : mesh_volume<C>(yq, lane);
                for (int vx = x1; vx >= x0; vx--) {
                    double below = 0.0;
                    if (vx > x0) {
                        bool cut;
                        const bool some = mesh_cut<C>(yq, 0, edge(0, vx), true,
                                                      lane, bad, &cut);
                        below = !some ? 0.0 : (cut ? mesh_volume<C>(yq, lane) : left);
                    }
                    if (isnan(left) || isnan(below)) {  // a piece whose faces do not close
                        bad = true;
                        break;
                    }
                    const double mass = (left - below) * unit;
                    if (lane == 0 && mass > 0.0)
                        atomicAdd(&mp.mass_fx[row + wrap_index(vx, M)],
                                  (unsigned long long)llrint(mass));
                    left = below;
                    if (!(left > 0.0)) break;
                }
                __syncwarp();
            }
        }
        if (bad && lane == 0) atomicAdd(mp.flags, 1);
    }
}

__global__ void mesh_centre_kernel(int M, double Lx, double Ly, double Lz,
                                   double* __restrict__ centre) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * M) return;
    const int a = t / M;
    const double L = a == 0 ? Lx : (a == 1 ? Ly : Lz);
    centre[t] = __ddiv_rn(__dmul_rn((double)(t - a * M) + 0.5, L), (double)M);
}

__global__ void mesh_init_kernel(int64_t n, unsigned long long* mass_fx,
                                 unsigned long long* phi_ord, int32_t* owner) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (mass_fx) mass_fx[t] = 0ull;
    if (phi_ord) phi_ord[t] = 0xffffffffffffffffull;
    if (owner) owner[t] = INT32_MAX;
}

__global__ void mesh_out_kernel(int64_t n, const unsigned long long* __restrict__ mass_fx,
                                double unit_per_vox, const unsigned long long* __restrict__ phi_ord,
                                double* __restrict__ rho, double* __restrict__ phi,
                                int32_t* __restrict__ missing) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    if (rho) rho[t] = (double)mass_fx[t] * unit_per_vox;
    if (phi_ord) {
        const unsigned long long u = phi_ord[t];
        if (u == 0xffffffffffffffffull) atomicAdd(missing, 1);  // no cell claimed the point
        if (phi) phi[t] = ord2d(u);
    }
}

// ClipParams for rebuilding the cells of context d from its facets (FP64, seed frame)
ClipParams mesh_clip_params(DeviceState& d);

int mesh_eval(DeviceState& d, int M, double lambda, double* rho_dev, double* phi_dev,
              int32_t* owner_dev, void* scratch, cudaStream_t s) {
    NvtxRange nv("mesh");
    const int64_t n = (int64_t)M * M * M;
    unsigned long long* mass_fx = rho_dev ? (unsigned long long*)scratch : nullptr;
    unsigned long long* phi_ord =
        (phi_dev || owner_dev) ? (unsigned long long*)scratch + (rho_dev ? n : 0) : nullptr;
    // [26] rebuild failures, [27] unclaimed points, [28] work counter; of the counters an
    // evaluation uses: [4] work counter of the large polytopes, [5] their cells, [6] claimed
    // twice
    SDOT_CUDA_TRY(cudaMemsetAsync(d.counters + 26, 0, 3 * sizeof(int32_t), s));
    SDOT_CUDA_TRY(cudaMemsetAsync(d.counters + 4, 0, 3 * sizeof(int32_t), s));
    const unsigned nb = (unsigned)((n + 255) / 256);
    mesh_init_kernel<<<nb, 256, 0, s>>>(n, mass_fx, phi_ord, owner_dev);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    mesh_centre_kernel<<<(unsigned)((3 * M + 255) / 256), 256, 0, s>>>(M, d.L[0], d.L[1], d.L[2],
                                                                      d.partials);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    MeshParams mp;
    mp.M = M;
    mp.s = 1.0 - lambda;
    for (int a = 0; a < 3; a++) {
        mp.h[a] = d.L[a] / M;
        mp.inv_h[a] = M / d.L[a];
    }
    const double mass_unit = d.L[0] * d.L[1] * d.L[2] / 4611686018427387904.0;  // |box| / 2^62
    mp.inv_unit = 1.0 / mass_unit;
    mp.nu = d.nu;
    mp.centre = d.partials;
    mp.mass_fx = mass_fx;
    mp.phi_ord = phi_ord;
    mp.owner = owner_dev;
    mp.flags = d.counters + 26;
    mp.twice = d.counters + 6;
    mp.rest = d.queue;
    mp.nrest = d.counters + 5;
    ClipParams cp = mesh_clip_params(d);
    // three polytopes a warp, one warp a block
    const size_t smem = 3 * sizeof(Poly<double, MeshCap>), smem_big = 3 * sizeof(Poly<double, CapL>);
    static const cudaError_t attr = [=] {
        const cudaError_t e = cudaFuncSetAttribute(
            mesh_kernel<MeshCap>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return e != cudaSuccess
                   ? e
                   : cudaFuncSetAttribute(mesh_kernel<CapL>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)smem_big);
    }();
    SDOT_CUDA_TRY(attr);
    auto cells = [&](int pass) -> int {
        mp.pass = pass;
        mp.work = d.counters + 28;
        mesh_kernel<MeshCap><<<8 * num_sms(), 32, smem, s>>>(cp, mp);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        mp.work = d.counters + 4;
        mesh_kernel<CapL><<<4 * num_sms(), 32, smem_big, s>>>(cp, mp);
        note_launch();
        SDOT_CUDA_TRY(cudaGetLastError());
        return SDOT_OK;
    };
    int rc = cells(0);
    if (rc) return rc;
    if (owner_dev) {
        int32_t twice = 0;
        SDOT_CUDA_TRY(cudaMemcpyAsync(&twice, mp.twice, 4, cudaMemcpyDeviceToHost, s));
        SDOT_CUDA_TRY(cudaStreamSynchronize(s));
        if (twice) {  // points on facets: the owners again, among the cells of the minimum
            SDOT_CUDA_TRY(cudaMemsetAsync(d.counters + 28, 0, sizeof(int32_t), s));
            SDOT_CUDA_TRY(cudaMemsetAsync(d.counters + 4, 0, 2 * sizeof(int32_t), s));
            mesh_init_kernel<<<nb, 256, 0, s>>>(n, nullptr, nullptr, owner_dev);
            note_launch();
            SDOT_CUDA_TRY(cudaGetLastError());
            if ((rc = cells(1))) return rc;
        }
    }
    const double vox = mp.h[0] * mp.h[1] * mp.h[2];
    mesh_out_kernel<<<nb, 256, 0, s>>>(n, mass_fx, mass_unit / vox, phi_ord, rho_dev,
                                       phi_dev, d.counters + 27);
    note_launch();
    SDOT_CUDA_TRY(cudaGetLastError());
    int32_t h[2];
    SDOT_CUDA_TRY(cudaMemcpyAsync(h, d.counters + 26, 8, cudaMemcpyDeviceToHost, s));
    SDOT_CUDA_TRY(cudaStreamSynchronize(s));
    if (h[0] > 0) {
        set_error("sdot_mesh: " + std::to_string(h[0]) +
                  " cell(s) could not be rebuilt from their facets or clipped by a voxel");
        return SDOT_ERR_CAPACITY;
    }
    if (h[1] > 0) {
        set_error("sdot_mesh: " + std::to_string(h[1]) + " mesh point(s) claimed by no cell");
        return SDOT_ERR_CUDA;
    }
    return SDOT_OK;
}

}  // namespace sdot
