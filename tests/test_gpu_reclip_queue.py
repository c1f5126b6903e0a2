"""The FP64 re-clip's work lists hold every cell once: a box in which every cell fails the
FP32 check (each seed has a close twin, so every cell sees nearly parallel bisectors) and one
of them, a hub with more facets than the small polytope takes, overflows its first FP64
re-clip. The list of the re-clip is then full to its last entry when the hub is listed again.
The context's memory comes from an allocator that puts a guard behind every block; the guards
must be untouched, and the cells those of the FP64 path.
"""
import numpy as np
import pytest

from paper_2110_08868_gb300 import ics

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2110_08868_gb300 import binding as B  # noqa: E402

GUARD = 4096


def twin_box(n=6, n_sphere=48, seed=3):
    """A jittered n^3 lattice of twins (two seeds 0.004 a apart), the site at the centre
    replaced by a hub with twins on a sphere of radius 0.4 a around it."""
    a = 1.0 / n
    rng = np.random.default_rng(seed)
    q = ics.lattice(n, 1.0) + rng.uniform(-0.1, 0.1, (n ** 3, 3)) * a
    c = np.array([0.5, 0.5, 0.5])
    d = q - c
    q = q[np.linalg.norm(d - np.round(d), axis=1) > 0.6 * a]
    k = np.arange(n_sphere) + 0.5
    th = np.arccos(1 - 2 * k / n_sphere)
    ph = np.pi * (1 + 5 ** 0.5) * k
    sph = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    one = np.concatenate([q, c + 0.4 * a * sph])
    u = rng.standard_normal(one.shape)
    u *= 0.004 * a / np.linalg.norm(u, axis=1)[:, None]
    return np.ascontiguousarray(np.mod(np.concatenate([c[None], one, one + u]), 1.0))


def test_reclip_lists_hold_every_cell():
    y = twin_box()
    N = len(y)
    blocks = {}

    def alloc(n):
        t = torch.full((n + GUARD + 256,), 0xA5, dtype=torch.uint8, device="cuda")
        p = (t.data_ptr() + 255) // 256 * 256
        blocks[p] = (t, p - t.data_ptr() + n)
        return p

    def free(p):
        t, end = blocks.pop(p)
        torch.cuda.synchronize()
        assert bool((t[end:end + GUARD - 256] == 0xA5).all()), "a block was overrun"

    B.check(B.sdot_set_allocator(alloc, free))
    try:
        with B.Solver(y, [1.0] * 3, precision="mixed") as s:
            g = s.laguerre(None, allow_empty=True)
            st = s.status()
            info = B.sdot_eval_info()
            B.check(B.sdot_last_eval(s.ctx, info))
            torch.cuda.synchronize()
            for t, end in blocks.values():
                assert bool((t[end:end + GUARD - 256] == 0xA5).all()), "a block was overrun"
    finally:
        B.check(B.sdot_set_allocator())
    over = int(np.count_nonzero(st & (32 | 64)))
    print(f"N {N}, re-clipped {info.reclipped_fp64}, over the small polytope {over}")
    assert over >= 1 and info.reclipped_fp64 + over > N, "the lists were not filled"
    assert not (st & 2).any()
    with B.Solver(y, [1.0] * 3, precision="fp64") as s:
        r = s.laguerre(None, allow_empty=True)
    np.testing.assert_allclose(g["vol"], r["vol"], rtol=0, atol=1e-10 / N)
