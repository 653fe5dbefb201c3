"""cc_autotune and cc_set_sweep_variant change what they say and nothing else:
the row build of the tuned precision, never a dynamic mesh's mixed one unless the
caller has switched it; no memory kept that the choice does not read; a variant
without memory is left out, and a call that fails leaves the mesh as it was.

Bits are compared at equal launch shapes.  Sizes: the mixed store takes 416 bytes
a tet; cudaMalloc gives 2 MiB pieces, 48 MiB for all of a call's other buffers.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu

MIB = 1 << 20


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


def test_row_lanes_are_not_chosen_for_kernels_without_them():
    sc = meshgen.stretch_box(5, 4, 6, E=1e5, nu=0.3, factor=1.05, jitter_amount=0.05, seed=8)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(2)
    m.set_launch_shape(couple_row_lanes=2)
    for precision in ("mixed", "fp64"):
        tune = m.autotune(cc.to_soa(sc.x0), precision=precision, sweeps=2)
        assert tune["couple_row_lanes"] == 2 and len(set(tune["row_lanes_ms"])) == 1
    m.close()


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def body():
    """A quasistatic body with its mixed state, and one sweep's positions."""
    for side in (4, 48):  # every kernel has been loaded once
        sc = meshgen.stretch_box(side, side, side, E=1e5, nu=0.3, factor=1.02, jitter_amount=0.0)
        m = cc.Mesh.from_scene(sc)
        m.color()
        m.build_subspace(2)
        if side == 4:
            m.autotune(cc.to_soa(sc.x0), precision="mixed", sweeps=1)
            m.close()
    x = cc.to_soa(sc.x0)
    m.sweep(x, precision="mixed")
    yield sc, m, cc.from_soa(x)
    m.close()


def _sweep(body):
    x = cc.to_soa(body[0].x0)
    body[1].sweep(x, precision="mixed")
    return cc.from_soa(x)


def test_a_switch_without_memory_changes_nothing(body):
    sc, m, want = body
    assert 416 * sc.T > 64 * MIB + 48 * MIB
    hold = torch.empty(_free() - 64 * MIB, dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(cc.CCError) as e:
            m.set_sweep_variant(rows_from_positions=0)
        assert e.value.status == cc.ERR_OOM
    finally:
        del hold
        torch.cuda.empty_cache()
    hold = torch.empty(_free() - 64 * MIB, dtype=torch.uint8, device="cuda")
    try:
        got = _sweep(body)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want - sc.x0).max()
    m.build_subspace(2)
    np.testing.assert_array_equal(_sweep(body), want)


def test_tuning_gives_back_the_store_and_works_without_memory_for_it(body):
    sc, m, want = body
    m.build_subspace(2)
    _sweep(body)
    before = _free()
    tune = m.autotune(cc.to_soa(sc.x0), precision="mixed", sweeps=1)
    assert tune["rows_from_positions"] and all(t > 0 for t in tune["variant_ms"])
    assert before - _free() <= 48 * MIB
    hold = torch.empty(_free() - 64 * MIB, dtype=torch.uint8, device="cuda")
    try:
        tune = m.autotune(cc.to_soa(sc.x0), precision="mixed", sweeps=1)
        got = _sweep(body)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert tune["variant_ms"][:2] == [0.0, 0.0] and tune["rows_from_positions"]
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want - sc.x0).max()
