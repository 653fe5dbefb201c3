"""The slot-map coupling kernels (k_couple, k_couple_warp) against the oracle on
the meshes that run them: every launch shape in the mixed path of a dynamic mesh,
and both precisions of a static mesh with supports of 1 021 vertices, one more
than the pair lists' fields hold (1 020 still takes the lists).

Tolerances as for the other sweeps against the oracle: the largest update to 1e-9
in float64 and to 1e-4 in mixed precision.
"""
import functools

import numpy as np
import pytest

import meshgen
from oracle import fem, solvers, subspace, topology

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu

SHAPES = [(32, 0)] + [(t, r) for t in (64, 128, 256) for r in (1, 2, 4, 8)]


def _oracle(sc):
    pb = fem.problem_from_scene(sc)
    return pb, topology.Topology(pb.n, pb.tets, pb.free)


def _noisy(sc, amount):
    return sc.x0 + meshgen.normal(6, np.arange(3 * sc.n)).reshape(-1, 3) * amount * sc.cell * (sc.pinned == 0)[:, None]


def _split(m, n):
    ptr, idx, U = m.export("sup_ptr"), m.export("sup_idx"), m.export("U").reshape(-1, 3, 3)
    return [idx[ptr[v]:ptr[v + 1]] for v in range(n)], [U[ptr[v]:ptr[v + 1]] for v in range(n)]


def _agree(got, want, x0, tol):
    assert np.abs((got - x0) - (want - x0)).max() <= tol * np.abs(want - x0).max()


def _beam(k):
    sc = meshgen.cantilever(4, 5, 7, cell=1 / 16, E=1e6, nu=0.4)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(k)
    return sc, m


@functools.lru_cache(maxsize=None)
def _beam_oracle(k, update):
    sc, m = _beam(k)
    pb, topo = _oracle(sc)
    sup, U = _split(m, sc.n)
    m.close()
    x0 = _noisy(sc, 0.05)
    return x0, solvers.sweep(pb, topo, sup, U, x0, x0 + 1e-3, update, "colored")


@pytest.mark.parametrize("threads,lanes", SHAPES)
@pytest.mark.parametrize("k,update,fused", [(2, "cc", 0), (2, "cc", 1), (3, "cc", 0), (2, "jgs2", 0)])
def test_every_launch_shape_of_a_dynamic_mixed_sweep(k, update, fused, threads, lanes):
    x0, want = _beam_oracle(k, update)
    sc, m = _beam(k)
    assert sc.h > 0
    m.set_launch_shape(couple_threads=threads, couple_row_lanes=lanes)
    m.set_sweep_variant(fused_condense=fused)
    x = cc.to_soa(x0)
    m.sweep(x, cc.to_soa(x0 + 1e-3), update=update, precision="mixed")
    m.close()
    _agree(cc.from_soa(x), want, x0, 1e-4)


@functools.lru_cache(maxsize=None)
def _wide(count):
    """A body whose 1-ring supports are widened to the `count` nearest free
    vertices at two vertices, and one sweep of the oracle on it."""
    sc = meshgen.stretch_box(11, 11, 11, E=1e5, nu=0.3, factor=1.1, jitter_amount=0.05, seed=4)
    pb, topo = _oracle(sc)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(1)
    sup, U = _split(m, sc.n)
    m.close()
    H = pb.hessian(pb.X)
    free = np.flatnonzero(pb.free)
    for target in (sc.X.mean(axis=0), sc.X[free[3]]):
        i = free[np.argmin(np.linalg.norm(sc.X[free] - target, axis=1))]
        others = free[free != i]
        near = np.argsort(np.linalg.norm(sc.X[others] - sc.X[i], axis=1), kind="stable")[:count]
        sup[i] = np.sort(others[near]).astype(np.int32)
        U[i] = subspace.local_basis(H, int(i), sup[i])
    x0 = _noisy(sc, 0.02)
    return sc, sup, U, x0, solvers.sweep(pb, topo, sup, U, x0, None, "cc", "colored")


@pytest.mark.parametrize("threads,lanes", [(32, 0), (64, 4), (64, 8), (128, 1), (256, 2)])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("count", [1020, 1021])
def test_supports_at_the_limit_of_the_pair_lists(count, precision, threads, lanes):
    sc, sup, U, x0, want = _wide(count)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(1)
    m.set_subspace(np.concatenate([[0], np.cumsum([len(s) for s in sup])]), np.concatenate(sup), np.concatenate(U))
    m.set_launch_shape(couple_threads=threads, couple_row_lanes=lanes)
    x = cc.to_soa(x0)
    if precision == "fp64" and threads == 32:  # a warp's share of an SM never held this many float64 rows
        with pytest.raises(cc.CCError) as e:
            m.sweep(x, precision=precision)
        assert e.value.status == cc.ERR_INVALID_ARG
    else:
        m.sweep(x, precision=precision)
        _agree(cc.from_soa(x), want, x0, 1e-9 if precision == "fp64" else 1e-4)
    m.close()
