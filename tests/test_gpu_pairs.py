"""The float32 coupling kernel's pair lists against the float64 path, where its
loops change: no support at all, supports below and above one and two warps'
rows, pairs that end inside a warp, supports next to clamped vertices, several
rounds of every loop (3- and 4-rings), and caller-supplied supports.

Tolerance: the products are float32 sums of at most a few thousand terms over
local systems whose condition is below 1e3 here, so one sweep's updates agree
to 1e-4 of the largest, as between the mixed path and the oracle elsewhere.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


def _scene(size, seed=5):
    sc = meshgen.stretch_box(*size, E=1e5, nu=0.3, factor=1.05, jitter_amount=0.05, seed=seed)
    x0 = sc.x0 + meshgen.normal(seed + 1, np.arange(3 * sc.n)).reshape(-1, 3) * 0.02 * sc.cell * (sc.pinned == 0)[:, None]
    return sc, x0


def _agree(m, x0, threads, updates=("cc", "jgs2")):
    m.set_launch_shape(couple_threads=threads)
    for update in updates:
        step = []
        for precision in ("fp64", "mixed"):
            x = cc.to_soa(x0)
            m.sweep(x, update=update, precision=precision)
            step.append(cc.from_soa(x) - x0)
        assert np.abs(step[1] - step[0]).max() <= 1e-4 * np.abs(step[0]).max()


@pytest.mark.parametrize("threads", [32, 64, 128, 256])
@pytest.mark.parametrize("size,k", [((2, 1, 1), 1), ((2, 3, 1), 2), ((4, 3, 3), 1), ((5, 4, 6), 2), ((6, 5, 7), 3),
                                    ((7, 6, 8), 4)])
def test_pair_lists_agree_with_float64(size, k, threads):
    sc, x0 = _scene(size)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(k)
    _agree(m, x0, threads)
    m.close()


def test_supports_given_by_the_caller():
    """Empty, single and far-away supports: entries of every other vertex are dropped."""
    sc, x0 = _scene((4, 4, 4))
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(2)
    ptr, idx, U = m.export("sup_ptr"), m.export("sup_idx"), m.export("U").reshape(-1, 3, 3)
    keep = np.ones(idx.size, dtype=bool)
    for v in range(sc.n):
        s, e = ptr[v], ptr[v + 1]
        if v % 3 == 0:
            keep[s:e] = False
        elif v % 3 == 1:
            keep[s + 1:e:2] = False
    new_ptr = np.concatenate([[0], np.cumsum([keep[ptr[v]:ptr[v + 1]].sum() for v in range(sc.n)])])
    m.set_subspace(new_ptr, idx[keep], U[keep])
    _agree(m, x0, 64)
    m.close()
