"""Block rows formed from the positions against the per-tet store and gather,
where the row kernel's loops change: edges of few, of exactly eight and of
more than eight tets, rows of more than 24 tets and more than 16 neighbours,
rows of more than eight upper blocks, a last warp with fewer than four rows,
and a 1-ring too large for it (both settings then run the gather).

Tolerances: both builds evaluate the same sums in another order, so one sweep's
updates agree to rounding times the local systems' condition (below 1e4 here):
1e-10 of the largest update in float64, 1e-4 in mixed precision (float32
blocks), as between the mixed path and the oracle elsewhere.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


def _spindle(count):
    """`count` tets around one edge (two free axis vertices, ids first), every
    other ring vertex pinned (fewer would leave a patch free to turn)."""
    th = 2.0 * np.pi * np.arange(count) / count
    ring = np.stack([np.cos(th), np.sin(th), 0.1 * np.cos(3 * th)], axis=1)
    X = np.concatenate([[[0.0, 0.0, -0.7], [0.05, 0.02, 0.8]], ring])
    tets = np.array([[0, 1, 2 + i, 2 + (i + 1) % count] for i in range(count)], dtype=np.int32)
    pinned = np.zeros(count + 2, dtype=np.uint8)
    pinned[2::2] = 1
    rng = np.random.default_rng(count)
    x0 = X + rng.uniform(-0.02, 0.02, X.shape) * (pinned == 0)[:, None]
    return X, tets, pinned, x0


def _steps(X, tets, pinned, x0, precision, update, h=0.0):
    out = []
    for rows in (0, 1):
        m = cc.Mesh(X, tets, pinned, E=1e5, nu=0.3, h=h)
        m.color()
        m.build_subspace(1)
        m.set_sweep_variant(rows_from_positions=rows)
        x = cc.to_soa(x0)
        xt = cc.to_soa(x0 + 1e-3) if h else None
        _, g, _ = m.energy_grad(x, xt, precision=precision)
        m.sweep(x, xt, update=update, precision=precision)
        out.append((cc.from_soa(g), cc.from_soa(x) - x0))
        m.close()
    return out


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("count", [3, 8, 9, 17, 41, 90, 300])
def test_rows_of_any_valence_agree_with_the_gather(count, precision, tol):
    X, tets, pinned, x0 = _spindle(count)
    for update in ("cc", "cd"):
        (g0, d0), (g1, d1) = _steps(X, tets, pinned, x0, precision, update)
        assert np.abs(g1 - g0).max() <= 1e-10 * np.abs(g0).max()
        assert np.abs(d1 - d0).max() <= tol * np.abs(d0).max()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("size,unit,h", [((1, 1, 1), 1.0, 0.0), ((2, 3, 1), 1e-6, 0.0), ((3, 2, 4), 1e4, 0.01)])
def test_boxes_in_any_unit_of_length_agree_with_the_gather(size, unit, h, precision, tol):
    sc = meshgen.stretch_box(*size, E=1e5, nu=0.3, factor=1.1, jitter_amount=0.05, seed=2)
    x0 = sc.x0 + meshgen.normal(3, np.arange(3 * sc.n)).reshape(-1, 3) * 0.03 * sc.cell * (sc.pinned == 0)[:, None]
    pinned = sc.pinned.copy()
    if size == (1, 1, 1):
        pinned[np.argmax(pinned)] = 0  # a cube's eight corners are all clamped: one goes free
    (g0, d0), (g1, d1) = _steps(unit * sc.X, sc.tets, pinned, unit * x0, precision, "cc", h)
    assert np.abs(g1 - g0).max() <= 1e-10 * np.abs(g0).max()
    assert np.abs(d1 - d0).max() <= tol * np.abs(d0).max()
