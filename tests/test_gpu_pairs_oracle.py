"""The pair-list coupling kernels of both precisions against the oracle, which
reads the exported supports and bases but no list: the bodies of test_gpu_pairs
(no support at all, supports around one and two warps' rows, pairs that end inside
a warp, supports next to clamped vertices, several rounds of every loop, supports
given by the caller) and every thread count.  And the one-warp launch of large
colours, two shares a warp, against two warps: the same bits.

Tolerances as for the other sweeps against the oracle: the largest update to 1e-9
in float64 and to 1e-4 in mixed precision.
"""
import numpy as np
import pytest

import meshgen
from oracle import fem, solvers, topology

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402
from test_gpu_pairs import _scene  # noqa: E402

pytestmark = pytest.mark.gpu


def _check(sc, x0, m):
    pb = fem.problem_from_scene(sc)
    topo = topology.Topology(pb.n, pb.tets, pb.free)
    ptr, idx, U = m.export("sup_ptr"), m.export("sup_idx"), m.export("U").reshape(-1, 3, 3)
    sup, bases = [idx[ptr[v]:ptr[v + 1]] for v in range(sc.n)], [U[ptr[v]:ptr[v + 1]] for v in range(sc.n)]
    for update in ("cc", "jgs2"):
        want = solvers.sweep(pb, topo, sup, bases, x0, None, update, "colored") - x0
        for precision, tol in (("fp64", 1e-9), ("mixed", 1e-4)):
            for threads in (32, 64, 128, 256):
                m.set_launch_shape(couple_threads=threads)
                x = cc.to_soa(x0)
                m.sweep(x, update=update, precision=precision)
                assert np.abs(cc.from_soa(x) - x0 - want).max() <= tol * np.abs(want).max(), (update, precision, threads)


@pytest.mark.parametrize("size,k", [((2, 1, 1), 1), ((2, 3, 1), 2), ((4, 3, 3), 1), ((5, 4, 6), 2), ((6, 5, 7), 3),
                                    ((7, 6, 8), 4)])
def test_pair_lists_agree_with_the_oracle(size, k):
    sc, x0 = _scene(size)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(k)
    _check(sc, x0, m)
    m.close()


def test_supports_given_by_the_caller_agree_with_the_oracle():
    """Empty supports, every other vertex of the 2-ring, and one far-away vertex."""
    sc, x0 = _scene((4, 4, 4))
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(2)
    ptr, idx, U = m.export("sup_ptr"), m.export("sup_idx"), m.export("U").reshape(-1, 3, 3)
    free = np.flatnonzero(sc.pinned == 0)
    sup, bases = [], []
    for v in range(sc.n):
        S, B = idx[ptr[v]:ptr[v + 1]], U[ptr[v]:ptr[v + 1]]
        if v % 3 == 0:
            S, B = S[:0], B[:0]
        elif v % 3 == 1:
            S, B = S[::2], B[::2]
        elif len(S):
            far = free[-1] if v < free[-1] // 2 else free[0]
            if far != v and far not in S:
                at = np.searchsorted(S, far)
                S, B = np.insert(S, at, far), np.insert(B, at, 0.05 * np.eye(3), axis=0)
        sup.append(S)
        bases.append(B)
    m.set_subspace(np.concatenate([[0], np.cumsum([len(s) for s in sup])]), np.concatenate(sup), np.concatenate(bases))
    _check(sc, x0, m)
    m.close()


@pytest.mark.parametrize("update", ["cc", "jgs2"])
@pytest.mark.parametrize("k", [2, 3])
def test_one_warp_with_two_shares_gives_the_bits_of_two_warps(k, update):
    sc, x0 = _scene((18, 17, 16))
    assert int((sc.pinned == 0).sum()) > 152 * 32  # one Jacobi list above the line
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(k)
    got = []
    for fused in (0, 1):  # the fused launch always takes two warps
        m.set_sweep_variant(fused_condense=fused)
        x = cc.to_soa(x0)
        m.sweep(x, update=update, schedule="jacobi", precision="mixed")
        got.append(cc.from_soa(x))
    m.close()
    np.testing.assert_array_equal(got[0], got[1])
