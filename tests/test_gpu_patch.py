"""Patch solves (float32 factor, float64 refinement) where their loops change:
every patch size from one to 64 vertices (the 16-unknown tiles' edges, one to
twelve block columns), and a patch with more blocks than the kernel lists.

Tolerance: both sides solve the same float64 system to rounding times its
condition (below 1e5 here), 1e-10 of the largest basis entry, as elsewhere.
"""
import numpy as np
import pytest

import meshgen
from oracle import fem, subspace, topology

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


def _bases(m):
    return m.export("sup_ptr"), m.export("sup_idx"), m.export("U").reshape(-1, 3, 3)


def test_every_patch_size_matches_the_oracle():
    sc = meshgen.stretch_box(8, 6, 6, E=1e5, nu=0.3, factor=1.2, jitter_amount=0.05, seed=8)
    x = sc.x0 + meshgen.normal(9, np.arange(3 * sc.n)).reshape(-1, 3) * 0.02 * sc.cell * (sc.pinned == 0)[:, None]
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(2)
    ptr, idx, _ = _bases(m)
    size = np.diff(ptr)
    free = np.flatnonzero(size)
    sup = [idx[ptr[v]:ptr[v + 1]] for v in range(sc.n)]
    for q, v in enumerate(free[np.argsort(-size[free], kind="stable")][:64]):  # sizes 64, 63, .., 1, nearest first
        near = np.argsort(np.linalg.norm(sc.X[sup[v]] - sc.X[v], axis=1), kind="stable")[:64 - q]
        sup[v] = np.sort(sup[v][near])
    assert set(range(1, 65)) <= {s.size for s in sup}
    m.set_subspace(np.concatenate([[0], np.cumsum([s.size for s in sup])]), np.concatenate(sup),
                   np.zeros((sum(s.size for s in sup), 3, 3)))
    assert m.build_subspace_at(cc.to_soa(x)) == 0
    assert m.info().patch_float64 == 0
    pb = fem.problem_from_scene(sc)
    want, kept = subspace.rebuild_bases_at(pb, sup, [np.zeros((s.size, 3, 3)) for s in sup], x)
    ptr, _, U = _bases(m)
    assert kept == 0
    for v in free:
        np.testing.assert_allclose(U[ptr[v]:ptr[v + 1]], want[v], rtol=0, atol=1e-10 * max(1.0, np.abs(want[v]).max()))
    m.close()


def test_a_patch_of_more_blocks_than_the_list_matches_the_oracle():
    """Two skew polylines of 29 vertices, joined: every vertex of one meets every vertex of the other."""
    count = 29
    t = np.linspace(-1.0, 1.0, count)
    X = np.concatenate([np.stack([t, 0 * t, 0 * t - 0.5], axis=1), np.stack([0 * t, t, 0 * t + 0.5], axis=1)])
    tets = np.array([[a, a + 1, count + b, count + b + 1] for a in range(count - 1) for b in range(count - 1)],
                    dtype=np.int32)
    pinned = np.zeros(2 * count, dtype=np.uint8)
    pinned[[0, count - 1, count, 2 * count - 1]] = 1
    m = cc.Mesh(X, tets, pinned, E=1e5, nu=0.3)
    m.color()
    m.build_subspace(2)
    ptr, idx, U = _bases(m)
    vol = np.linalg.det((X[tets[:, 1:]] - X[tets[:, :1]]))
    tets[vol < 0] = tets[vol < 0][:, [0, 2, 1, 3]]
    pb = fem.Problem(X, tets, pinned, fem.Model("snh", 1e5, 0.3))
    topo = topology.Topology(pb.n, pb.tets, pb.free)
    sup, want = subspace.build_local_bases(pb, topo, 2)
    assert max(s.size for s in sup) == 2 * count - 5
    for v in np.flatnonzero(pb.free):
        np.testing.assert_array_equal(idx[ptr[v]:ptr[v + 1]], sup[v])
        np.testing.assert_allclose(U[ptr[v]:ptr[v + 1]], want[v], rtol=0, atol=1e-10 * max(1.0, np.abs(want[v]).max()))
    m.close()
