"""The work a user of the library has it do, as cases that can be timed and compared.

A case is a dict of plain values; ``kind`` names the call, ``n`` the lattice side of the
box (N = n^3 seeds, more with clumps). Every box is a Zel'dovich-displaced lattice like
those of ``ics.py`` (made on the device, from the seed alone):

  knn_static  kNN lists without allocation: the smallest call, launches and latency
  first       create (grid hash, kNN lists) and the first diagram at psi = 0, destroy
  step        the evaluations of one Newton step on a live context: a line-search trial
              (volumes) and the accepted weights (volumes, centroids, Hessian)
  solve       a whole reconstruction: create, damped Newton, displacement, destroy
  mesh        phi_I, owners and the moved-cell density on a mesh
  spectrum    the power spectrum of a density mesh
  serve       a batch of host jobs through the reconstruction server
"""
import itertools
import math

import numpy as np
import torch

from paper_2110_08868_gb300 import binding as B
from paper_2110_08868_gb300 import ics

DEV = "cuda"


def listed():
    return [
        # a caller inside another framework's memory pool asks for neighbour lists
        dict(name="knn_static_17", kind="knn_static", n=17, k=24, rms=0.3),
        # a new snapshot arrives: hash it, build its lists, look at its Voronoi diagram
        dict(name="first_mixed_97", kind="first", n=97, k=24, prec="mixed", spectrum="bbks",
             rms=1.5),
        # late Newton steps: psi hardly moves between evaluations (an ordinary box, and
        # one the size of the bench's)
        dict(name="step_mixed_129", kind="step", n=129, prec="mixed", rms=0.3, step=2e-5,
             scale=1.0, clumps=0),
        dict(name="step_mixed_256", kind="step", n=256, prec="mixed", rms=0.3, step=2e-5,
             scale=1.0, clumps=0),
        # FP64 evaluations, with psi steps that outrun the carried certificates
        dict(name="step_fp64_45", kind="step", n=45, prec="fp64", rms=0.3, step=1e-3,
             scale=1.0, clumps=0),
        # early Newton: large psi steps, cells far from balance, every cell walks
        dict(name="step_mixed_far_100", kind="step", n=100, prec="mixed", rms=0.3, step=0.02,
             scale=0.5, clumps=0),
        # clumped seeds at solved weights: cells with many close, nearly parallel bisectors
        dict(name="step_mixed_clumps_33", kind="step", n=33, prec="mixed", rms=0.3, step=2e-5,
             scale=1.0, clumps=4),
        # whole reconstructions: a small FP64 box, and a mixed one with clumps
        dict(name="solve_fp64_16", kind="solve", n=16, prec="fp64", rms=0.3, tol=1e-10, clumps=0),
        dict(name="solve_mixed_clumps_35", kind="solve", n=35, prec="mixed", rms=0.3, tol=1e-9,
             clumps=5),
        # after the solve: potential, owners and density of the moved cells on a mesh
        dict(name="mesh_48_m96", kind="mesh", n=48, M=96, lam=0.5, rms=0.3),
        # the BAO estimator on a reconstructed density
        dict(name="spectrum_512", kind="spectrum", M=512),
        # many small boxes at once
        dict(name="serve_6", kind="serve", jobs=6, lo=18, hi=36, tol=1e-9),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["knn_static", "first", "step", "step", "step", "solve", "mesh",
                       "spectrum", "serve"])
    rms = round(rng.uniform(0.1, 0.4), 3)
    prec = rng.choice(["mixed", "fp64"])
    if kind == "knn_static":
        return dict(kind=kind, n=_logint(rng, 8, 31), k=rng.randint(4, 32), rms=rms)
    if kind == "first":
        return dict(kind=kind, n=_logint(rng, 12, 110), k=rng.choice([8, 16, 24, 24, 32]),
                    prec=prec, spectrum=rng.choice(["kinv", "bbks"]), rms=rms)
    if kind == "step":
        clumps = rng.choice([0, 0, 0, 2])
        step = float("%.2e" % math.exp(rng.uniform(math.log(1e-5), math.log(2e-2))))
        top = 36 if clumps else 70 if prec == "fp64" else 100 if step > 5e-4 else 160
        return dict(kind=kind, n=_logint(rng, 12, top), prec=prec, rms=rms, step=step,
                    scale=1.0 if clumps else rng.choice([0.3, 0.7, 1.0, 1.0]), clumps=clumps)
    if kind == "solve":
        return dict(kind=kind, n=_logint(rng, 12, 40), prec=prec, rms=rms, tol=1e-9,
                    clumps=rng.choice([0, 1, 2]))
    if kind == "mesh":
        return dict(kind=kind, n=_logint(rng, 12, 56), M=_logint(rng, 16, 112),
                    lam=round(rng.uniform(0.0, 0.9), 3), rms=rms)
    if kind == "spectrum":
        return dict(kind=kind, M=_logint(rng, 16, 512))
    lo = rng.randint(12, 24)
    return dict(kind=kind, jobs=rng.randint(2, 8), lo=lo, hi=lo + rng.randint(2, 12), tol=1e-9)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _box(n, L, spectrum, rms, seed):
    """A Zel'dovich box (the recipe of ics.zeldovich_box) on the device: positions (N, 3)
    and the potential psi = |s|^2 / 2 + phi(q) whose Laguerre cells lie around the lattice
    points q (s = grad phi: the weights of the continuous problem's solution)."""
    g = _gen(seed)
    a = L / n
    dk = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=DEV, dtype=torch.float64))
    k1 = torch.fft.fftfreq(n, d=1.0 / n, device=DEV, dtype=torch.float64) * (2 * math.pi / L)
    k3 = torch.fft.rfftfreq(n, d=1.0 / n, device=DEV, dtype=torch.float64) * (2 * math.pi / L)
    kz, ky, kx = k1[:, None, None], k1[None, :, None], k3[None, None, :]
    k2 = kx * kx + ky * ky + kz * kz
    kk = k2.sqrt()
    keep = (kk > 0) & (kk < math.pi * n / L)
    kk = torch.where(keep, kk, 1.0)
    if spectrum == "kinv":
        P = 1.0 / kk
    else:  # the BBKS form of ics.spectrum_bbks_wiggle
        q = kk / 0.21
        x = 2.34 * q
        t = torch.log1p(x) / x * (1 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3
                                  + (6.71 * q) ** 4) ** -0.25
        P = kk * t * t * (1.0 + 0.1 * torch.sin(105.0 * kk) / (105.0 * kk))
    phik = torch.where(keep, dk * P.sqrt() / kk ** 2, torch.zeros((), dtype=dk.dtype, device=DEV))
    del dk, P, kk, k2, keep
    s = torch.empty((n ** 3, 3), dtype=torch.float64, device=DEV)
    for c, kc in enumerate((kx, ky, kz)):
        s[:, c] = torch.fft.irfftn(1j * kc * phik, s=(n, n, n)).reshape(-1)
    phi = torch.fft.irfftn(phik, s=(n, n, n)).reshape(-1)
    f = rms * a / (s * s).sum(1).mean().sqrt()
    s *= f
    phi *= f
    c = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) * a
    z, y, x = torch.meshgrid(c, c, c, indexing="ij")
    pos = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1) + s
    pos = torch.remainder(pos, L)
    pos[pos >= L] = 0.0
    psi = 0.5 * (s * s).sum(1) + phi
    return pos.contiguous(), (psi - psi.mean()).contiguous()


def _clumped(n, L, rms, clumps, seed):
    """Positions with clumps of width 0.05 a (ics.add_clumps; the bench's box has about 420
    seeds a clump)."""
    y, _ = _box(n, L, "kinv", rms, seed)
    if not clumps:
        return y
    z = ics.add_clumps(y.cpu().numpy(), L, n, clumps, clumps * _clump_seeds(n), 0.05,
                       int(seed) + 100)
    return torch.from_numpy(np.ascontiguousarray(z)).to(DEV)


def _size(case):
    L = 1000.0 if case.get("spectrum") == "bbks" else 1.0
    return case["n"], L, L / case["n"]


def _clump_seeds(n):
    return min(420, n ** 3 // 40)


def _seeds(case):
    """The number of seeds of a case's box."""
    n = case["n"]
    return n ** 3 + case.get("clumps", 0) * _clump_seeds(n)


def _weights(case, seed):
    """Positions and the two weights of a step case: the accepted ones and a trial that
    differs by white noise of case["step"] a^2."""
    n, L, a = _size(case)
    if case["clumps"]:
        y = _clumped(n, L, case["rms"], case["clumps"], seed)
        with B.Solver(y, [L] * 3, precision="mixed") as s:
            s.solve(1e-4)
            psi = torch.from_numpy(s.psi()).to(DEV)
    else:
        y, psi = _box(n, L, "kinv", case["rms"], seed)
        psi = psi * case["scale"]
    noise = torch.randn(psi.shape, generator=_gen(seed + 7), device=DEV, dtype=torch.float64)
    return y, psi, psi + case["step"] * a * a * noise


def _job_sides(case):
    return np.rint(np.geomspace(case["lo"], case["hi"], case["jobs"])).astype(int)[::-1]


def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device=DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "knn_static":
        n, L, _ = _size(case)
        st["pos"], _ = _box(n, L, "kinv", case["rms"], seed)
        st["L"] = L
        st["nbr"] = _empty(n ** 3, case["k"], dtype=torch.int32)
    elif kind == "first":
        n, L, _ = _size(case)
        st["pos"], _ = _box(n, L, case["spectrum"], case["rms"], seed)
        st["L"] = L
        st["opt"] = B.sdot_default_options(precision=case["prec"], k=case["k"])
    elif kind == "step":
        # a context in the middle of its solve: it has been evaluated at both weights
        n, L, _ = _size(case)
        y, psi, trial = _weights(case, seed)
        st["solver"] = B.Solver(y, [L] * 3, precision=case["prec"])
        st["psi"], st["trial"] = psi, trial
        # the caller's buffers for the Hessian (16.5 entries a row, with room)
        st["col"] = torch.zeros(20 * len(y) + 1024, dtype=torch.int32, device=DEV)
        st["val"] = torch.zeros(20 * len(y) + 1024, dtype=torch.float64, device=DEV)
        _evaluate(st["solver"].ctx, trial, _empty(len(y)))
        _evaluate(st["solver"].ctx, psi, _empty(len(y)))
    elif kind == "solve":
        n, L, _ = _size(case)
        st["pos"] = _clumped(n, L, case["rms"], case["clumps"], seed)
        st["L"] = L
        st["opt"] = B.sdot_default_options(precision=case["prec"])
    elif kind == "mesh":
        n, L, _ = _size(case)
        y, psi = _box(n, L, "kinv", case["rms"], seed)
        st["solver"] = B.Solver(y, [L] * 3)
        _evaluate(st["solver"].ctx, psi, _empty(len(y)))
        m = case["M"] ** 3
        st["out"] = (_empty(m), _empty(m), _empty(m, dtype=torch.int32))
    elif kind == "spectrum":
        M = case["M"]
        st["rho"] = _density(M, seed)
    else:
        st["boxes"] = [_box(int(n), 1.0, "kinv", 0.3, 1000 * seed + j)[0].cpu().numpy()
                       for j, n in enumerate(_job_sides(case))]
        st["server"] = B.Server(hbm_budget=16 << 30, max_active=8)
    return st


def _density(M, seed):
    g = torch.randn((M, M, M), generator=_gen(seed), device=DEV, dtype=torch.float64)
    return torch.exp(0.4 * g)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _evaluate(ctx, psi, vol, cen=None, hess=None):
    """sdot_laguerre as a line search calls it: weights that empty a cell are an answer."""
    rc = B.sdot_laguerre(ctx, psi, vol, cen, hess)
    if rc != B.SDOT_ERR_EMPTY_CELL:
        B.check(rc)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "knn_static":
        B.check(B.sdot_knn_static(st["pos"], [st["L"]] * 3, case["k"], st["nbr"]))
        return st["nbr"]
    if kind == "first":
        N = st["pos"].shape[0]
        rc, ctx = B.sdot_create(st["pos"], None, [st["L"]] * 3, st["opt"])
        B.check(rc)
        try:
            nbr, vol, cen = _empty(N, case["k"], dtype=torch.int32), _empty(N), _empty(N, 3)
            B.check(B.sdot_knn(ctx, nbr))
            B.check(B.sdot_laguerre(ctx, None, vol, cen, None))
        finally:
            B.sdot_destroy(ctx)
        return dict(nbr=nbr, vol=vol, cen=cen)
    if kind == "step":
        ctx, N = st["solver"].ctx, st["solver"].N
        vol_t, vol, cen, h = _empty(N), _empty(N), _empty(N, 3), B.sdot_csr()
        _evaluate(ctx, st["trial"], vol_t)
        _evaluate(ctx, st["psi"], vol, cen, h)
        rp, col, val = _empty(N + 1, dtype=torch.int64), st["col"], st["val"]
        if h.nnz > col.shape[0]:
            raise ValueError("the Hessian does not fit the buffers")
        B.check(B.sdot_csr_copy(h, rp, col, val))
        return dict(vol_t=vol_t, vol=vol, cen=cen, row_ptr=rp, col=col, val=val)
    if kind == "solve":
        N = st["pos"].shape[0]
        rc, ctx = B.sdot_create(st["pos"], None, [st["L"]] * 3, st["opt"])
        B.check(rc)
        try:
            psi, disp = _empty(N), _empty(N, 3)
            B.check(B.sdot_solve(ctx, case["tol"]))
            B.check(B.sdot_get_psi(ctx, psi))
            B.check(B.sdot_displacement(ctx, disp))
        finally:
            B.sdot_destroy(ctx)
        return dict(psi=psi, disp=disp)
    if kind == "mesh":
        rho, phi, own = st["out"]
        B.check(B.sdot_mesh(st["solver"].ctx, case["lam"], case["M"], rho, phi, own))
        return dict(rho=rho, phi=phi, owner=own)
    if kind == "spectrum":
        P, k, n = B.sdot_power_spectrum(st["rho"], 1000.0)
        return dict(P=P, k=k, n=n)
    srv = st["server"]
    ids = [srv.submit(y, [1.0] * 3, case["tol"]) for y in st["boxes"]]
    out = []
    for j in ids:
        srv.wait(j)
        r = srv.result(j)
        out.append(dict(disp=r["disp"], psi=r["psi"]))
    return out


# ---------------------------------------------------------------------------
# the least a pass has to do
# ---------------------------------------------------------------------------
FACETS = 15.5        # mean facets of a cell
CELL_FLOP = 6000.0   # one cell: 24 plane tests x 20 vertices x 6, 60 vertices x 10, 48 fans x 45
SOLVE_EVALS = 8      # evaluations of a quadratically converging damped Newton solve
SOLVE_CG = 200       # its CG iterations


def _solve_work(N):
    it = N * (8 * FACETS + 40.0)  # a CG iteration: matrix once, vectors once
    return dict(bytes=56.0 * N + SOLVE_CG * it,
                flops=N * (SOLVE_EVALS * CELL_FLOP + SOLVE_CG * (2 * FACETS + 14)))


def work(case):
    kind = case["kind"]
    if kind == "spectrum":
        M = case["M"]
        return dict(bytes=8.0 * M ** 3, flops=2.5 * M ** 3 * math.log2(M ** 3))
    if kind == "serve":
        w = [_solve_work(float(n) ** 3) for n in _job_sides(case)]
        return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))
    N = float(_seeds(case))
    if kind == "knn_static":
        return dict(bytes=N * (24 + 4 * case["k"]), flops=N * 27 * 2 * 8.0)
    if kind == "first":
        return dict(bytes=N * (24 + 4 * case["k"] + 32), flops=N * (27 * 2 * 8.0 + CELL_FLOP))
    if kind == "step":
        csr = 8 + 12 * (FACETS + 1)
        return dict(bytes=N * (24 + 2 * 16 + 24 + csr), flops=2 * N * CELL_FLOP)
    if kind == "solve":
        return _solve_work(N)
    return dict(bytes=N * 40 + 20.0 * case["M"] ** 3,
                flops=N * CELL_FLOP + 8.0 * case["M"] ** 3 * 6 * 10)


# ---------------------------------------------------------------------------
# the same in 64 bits, by enumeration
# ---------------------------------------------------------------------------
def _wrap(d, L):
    return d - L * torch.round(d / L)


def _cells64(y, psi, L, near=192, K=36, vmax=96):
    """Laguerre cells by enumeration in units of the spacing: per cell the K planes that
    bound it (the nearest ones to a point inside, then those that cut its vertices), every
    triple's point that no plane cuts off, and the tetrahedra (centre, face centre, edge).
    Six planes 6 spacings away keep every step's polytope bounded; no cell may reach them.
    Returns volumes, first moments about the seed, and the facets (i, j, area / |d|), or
    None when no such planes are found."""
    N = y.shape[0]
    a = L / N ** (1.0 / 3.0)
    y, psi, Lu = y / a, psi / (a * a), L / a
    near = min(near, N - 1)
    far = torch.cat([torch.eye(3, dtype=torch.float64, device=DEV)] * 2)
    far[3:] *= -1
    trip = torch.tensor(list(itertools.combinations(range(K), 3)), device=DEV)
    vol, mom, fac = _empty(N), _empty(N, 3), []
    size = max(64, min(512, int(2e8 / N)))
    for b in range(0, N, size):
        i = torch.arange(b, min(N, b + size), device=DEV)
        dd = sum(_wrap(y[None, :, c] - y[i, None, c], Lu) ** 2 for c in range(3))
        dd[torch.arange(len(i), device=DEV), i] = math.inf
        j = torch.topk(dd, near, dim=1, largest=False).indices
        del dd
        d = _wrap(y[j] - y[i][:, None], Lu)                      # (b, near, 3)
        ln = d.norm(dim=2)
        w = 0.5 * ln * ln + psi[i][:, None] - psi[j]
        d = torch.cat([d, far[None].expand(len(i), -1, -1)], 1)
        w = torch.cat([w, torch.full((len(i), 6), min(6.0, 0.5 * Lu), device=DEV,
                                     dtype=torch.float64)], 1)
        ln = d.norm(dim=2)
        # a point inside the cell (0.1 from its planes, if there is one), then the planes
        # nearest to it
        x = torch.zeros((len(i), 3, 1), dtype=torch.float64, device=DEV)
        for _ in range(60):
            over, t = ((torch.bmm(d, x)[..., 0] - w) / ln + 0.1).max(1)
            n1 = torch.gather(d / ln[..., None], 1, t[:, None, None].expand(-1, 1, 3))
            x = x - (over.clamp(min=0)[:, None, None] * n1).transpose(1, 2)
        score = (torch.bmm(d, x)[..., 0] - w) / ln
        score[:, near:] = 1e9
        # the vertices; the cells that some plane still cuts go round again
        n, act = len(i), torch.arange(len(i), device=DEV)
        sel = torch.zeros((n, K), dtype=torch.int64, device=DEV)
        tv = torch.zeros((n, vmax, 3), dtype=torch.int64, device=DEV)
        vv, vok = _empty(n, vmax, 3), torch.zeros((n, vmax), dtype=torch.bool, device=DEV)
        for _ in range(40):
            da, wa, sa = d[act], w[act], torch.topk(score, K, dim=1).indices
            n3 = torch.gather(da, 1, sa[..., None].expand(-1, -1, 3))
            wk = torch.gather(wa, 1, sa)
            p, q, r = (n3[:, trip[:, t]] for t in range(3))
            qr, rp, pq = (torch.linalg.cross(u, v, dim=2) for u, v in ((q, r), (r, p), (p, q)))
            det = (p * qr).sum(2, keepdim=True)
            v = sum(wk[:, trip[:, t], None] * c for t, c in enumerate((qr, rp, pq))) / det
            del p, q, r, qr, rp, pq
            ok = torch.isfinite(v).all(2) & (v.abs().amax(2) <= Lu)
            sd = torch.bmm(torch.nan_to_num(v, posinf=0.0, neginf=0.0), n3.transpose(1, 2))
            ok &= (sd - wk[:, None]).amax(2) <= 1e-11
            if int(ok.sum(1).max()) > vmax or int(ok.sum(1).min()) < 4:
                return None
            vi = torch.topk(ok.to(torch.int8), vmax, dim=1).indices
            ok = torch.gather(ok, 1, vi)
            v = torch.gather(v, 1, vi[..., None].expand(-1, -1, 3))
            v = torch.where(ok[..., None], v, torch.zeros((), dtype=v.dtype, device=DEV))
            sel[act], tv[act], vv[act], vok[act] = sa, trip[vi], v, ok
            viol = torch.bmm(v, da.transpose(1, 2)) - wa[:, None]
            viol = torch.where(ok[..., None], viol, -math.inf).amax(1)
            cut = viol.amax(1) > 1e-11
            if not bool(cut.any()):
                break
            score = (score + 0.3 * (viol > 1e-11))[cut]  # a plane that cut is kept longer
            act = act[cut]
        else:
            return None
        cen = vv.sum(1) / vok.sum(1)[:, None]
        # per face: membership, centre; edges: vertex pairs sharing two planes
        mem = torch.zeros((len(i), vmax, K), device=DEV, dtype=torch.float64)
        mem.scatter_(2, tv, 1.0)
        mem *= vok[..., None]
        fc = torch.bmm(mem.transpose(1, 2), vv) / mem.sum(1).clamp(min=1)[..., None]
        shared = torch.bmm(mem, mem.transpose(1, 2))
        e = torch.triu(shared == 2, 1).nonzero()                  # (E, 3): cell, u, v
        both = mem[e[:, 0], e[:, 1]] * mem[e[:, 0], e[:, 2]]      # (E, K), two ones
        f = both.nonzero()                                        # (2E, 2): edge, face
        c0, u, vtx = e[f[:, 0], 0], e[f[:, 0], 1], e[f[:, 0], 2]
        o, p, q, r = cen[c0], fc[c0, f[:, 1]], vv[c0, u], vv[c0, vtx]
        s = torch.linalg.cross(q - p, r - p, dim=1)
        t6 = ((p - o) * s).sum(1).abs()
        bv = torch.zeros(len(i), dtype=torch.float64, device=DEV).index_add_(0, c0, t6) / 6
        bm = torch.zeros((len(i), 3), dtype=torch.float64, device=DEV).index_add_(
            0, c0, t6[:, None] * (o + p + q + r)) / 24
        vol[i], mom[i] = bv, bm
        area = torch.zeros((len(i), K), dtype=torch.float64, device=DEV)
        area.view(-1).index_add_(0, c0 * K + f[:, 1], 0.5 * s.norm(dim=1))
        ci, k = (area > 0).nonzero().unbind(1)
        js = sel[ci, k]
        if bool((js >= near).any()):
            return None
        fac.append((i[ci], j[ci, js], area[ci, k] / ln[ci, js]))
    fi, fj, fv = (torch.cat(x) for x in zip(*fac))
    return vol * a ** 3, mom * a ** 4, (fi, fj, fv * a)


def _hessian64(N, fac):
    """CSR of L: the facets both cells see, the mean of their values, diagonal first."""
    fi, fj, fv = fac
    key, o = torch.sort(fi * N + fj)
    v = fv[o]
    at = torch.searchsorted(key, fj[o] * N + fi[o]).clamp(max=len(key) - 1)
    both = key[at] == fj[o] * N + fi[o]
    i, j, v = fi[o][both], fj[o][both], 0.5 * (v + v[at])[both]
    diag = torch.zeros(N, dtype=torch.float64, device=DEV).index_add_(0, i, v)
    ids = torch.arange(N, device=DEV)
    rows = torch.cat([ids, i])
    order = torch.argsort(rows * (N + 1) + torch.cat([torch.zeros_like(ids), j + 1]))
    col = torch.zeros(20 * N + 1024, dtype=torch.int32, device=DEV)
    val = torch.zeros(20 * N + 1024, dtype=torch.float64, device=DEV)
    col[:len(rows)] = torch.cat([ids, j])[order].to(torch.int32)
    val[:len(rows)] = torch.cat([diag, -v])[order]
    rp = torch.zeros(N + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=N), 0)
    return rp, col, val


def _centroid(y, vol, mom, L):
    return torch.remainder(y + mom / vol[:, None], L)


def exact(case, seed):
    kind = case["kind"]
    if kind == "spectrum":
        return _spectrum64(_density(case["M"], seed), 1000.0)
    if kind == "mesh":
        n, L, _ = _size(case)
        y, psi = _box(n, L, "kinv", case["rms"], seed)
        return dict(rho=None, phi=_phi64(y, psi, L, case["M"]), owner=None)
    if kind == "first" and case["n"] <= 48:
        n, L, _ = _size(case)
        y, psi = _box(n, L, case["spectrum"], case["rms"], seed)
        c = _cells64(y, torch.zeros_like(psi), L)
        return None if c is None else dict(nbr=None, vol=c[0], cen=_centroid(y, c[0], c[1], L))
    if kind == "step" and case["n"] <= 45 and not case["clumps"]:
        n, L, _ = _size(case)
        y, psi, trial = _weights(case, seed)
        t, c = _cells64(y, trial, L), _cells64(y, psi, L)
        if t is None or c is None:
            return None
        rp, col, val = _hessian64(len(y), c[2])
        if case["prec"] != "fp64":  # FP32 sees a facet of no area or not: no fixed layout
            rp = col = val = None
        return dict(vol_t=t[0], vol=c[0], cen=_centroid(y, c[0], c[1], L), row_ptr=rp, col=col,
                    val=val)
    if kind == "solve" and case["n"] <= 16 and not case["clumps"]:
        n, L, _ = _size(case)
        y, psi = _box(n, L, "kinv", case["rms"], seed)
        return _solve64(y, psi, L)
    return None


def _solve64(y, psi, L):
    """Newton from the continuous problem's weights, dense linear algebra."""
    N = y.shape[0]
    nu = L ** 3 / N
    for _ in range(12):
        c = _cells64(y, psi, L)
        if c is None or not float(c[0].min()) > 0:
            return None
        g = nu - c[0]
        if float(g.abs().max()) <= 1e-13 * nu:
            break
        fi, fj, fv = c[2]
        H = torch.zeros((N, N), dtype=torch.float64, device=DEV)
        H.view(-1).index_add_(0, fi * N + fj, -fv)
        H = 0.5 * (H + H.T)
        H.diagonal().sub_(H.sum(1))
        H += H.diagonal().mean() / N  # the constants are the kernel
        psi = psi + torch.linalg.solve(H, g - g.mean())
        psi = psi - psi.mean()
    else:
        if not float(g.abs().max()) <= 1e-11 * nu:
            return None
    return dict(psi=psi, disp=-c[1] / c[0][:, None])


def _phi64(y, psi, L, M):
    h = L / M
    c = (torch.arange(M, device=DEV, dtype=torch.float64) + 0.5) * h
    x2 = [_wrap(c[:, None] - y[None, :, k], L) ** 2 for k in range(3)]  # (M, N) per axis
    out = _empty(M, M, M)
    for z in range(M):
        for y0 in range(M):
            r = 0.5 * (x2[2][z] + x2[1][y0]) - psi
            near = torch.topk(r, min(4096, len(r)), largest=False)
            v = near.values[None] + 0.5 * x2[0][:, near.indices]
            out[z, y0] = v.amin(1)
            if len(r) > 4096 and bool((out[z, y0] > near.values[-1]).any()):
                out[z, y0] = (r[None] + 0.5 * x2[0]).amin(1)
    return out.reshape(-1)


def _spectrum64(rho, L):
    M = rho.shape[0]
    F = torch.fft.fftn(rho / rho.mean() - 1.0) / M ** 3
    f = torch.fft.fftfreq(M, d=1.0 / M, device=DEV, dtype=torch.float64)
    nn = (f[:, None, None] ** 2 + f[None, :, None] ** 2 + f[None, None, :] ** 2).sqrt()
    b = torch.floor(nn + 0.5).long().reshape(-1)
    nb = M // 2
    b = torch.where(b <= nb, b, 0)
    cnt = torch.bincount(b, minlength=nb + 1)[1:]
    P = torch.bincount(b, weights=(F.real ** 2 + F.imag ** 2).reshape(-1), minlength=nb + 1)[1:]
    k = torch.bincount(b, weights=nn.reshape(-1), minlength=nb + 1)[1:]
    out = (L ** 3 * P / cnt, 2 * math.pi / L * k / cnt, cnt)
    return dict(zip("Pkn", (x.cpu().numpy() for x in out)))
