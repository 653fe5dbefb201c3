"""cc_autotune changes what it says and nothing else: the row build of the tuned
precision, never a dynamic mesh's mixed one unless the caller has switched it.

Bits are compared at equal launch shapes.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


def _beam():
    sc = meshgen.stretch_box(6, 5, 12, E=1e5, nu=0.3, factor=1.05, jitter_amount=0.05, seed=8)
    m = cc.Mesh(sc.X, sc.tets, sc.pinned, E=1e5, nu=0.3, h=1e-2)
    m.color()
    m.build_subspace(2)
    return sc, m


def _mixed_sweep(m, sc):
    x = cc.to_soa(sc.x0)
    m.sweep(x, x + 1e-3, precision="mixed")
    return cc.from_soa(x)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_a_dynamic_mesh_keeps_its_mixed_rows(precision):
    sc, m = _beam()
    x = cc.to_soa(sc.x0)
    tune = m.autotune(x, x + 1e-3, precision=precision, sweeps=2)
    got = _mixed_sweep(m, sc)
    m.close()
    _, m = _beam()
    m.set_launch_shape(tune["couple_threads"], tune["gather_warps"], tune["couple_row_lanes"])
    m.set_sweep_variant(fused_condense=int(tune["fused_condense"]))
    np.testing.assert_array_equal(got, _mixed_sweep(m, sc))
    m.close()
    if precision == "mixed":
        assert not tune["rows_from_positions"] and tune["variant_ms"][2:] == [0.0, 0.0]


def test_a_switched_dynamic_mesh_is_tuned_over_both_row_builds():
    sc, m = _beam()
    m.set_sweep_variant(rows_from_positions=1)
    x = cc.to_soa(sc.x0)
    assert all(t > 0 for t in m.autotune(x, x + 1e-3, precision="mixed", sweeps=2)["variant_ms"])
    m.close()
