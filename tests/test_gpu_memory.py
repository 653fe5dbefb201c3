"""Device memory of the coupling kernels' lists: only those that a mesh's sweeps
read are made, and a mesh that fits without pair lists is built and swept even
where they do not fit, before its solver state exists or after.

Sizes: a list of 2-rings takes 8 bytes per support entry and 4 per pair (at least
200 pairs a free vertex on these bodies), a slot map at most 8 codes per row.
cudaMalloc gives 2 MiB pieces, 48 MiB for all of a call's buffers.  Results of the
two kernels agree to 1e-4 of the largest update, as in the other tests.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu

SIDE = 48
MIB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def body():
    sc = meshgen.stretch_box(SIDE, SIDE, SIDE, E=1e5, nu=0.3, factor=1.02, jitter_amount=0.0)
    for h in (0.0, 1e-2):  # every kernel below has been loaded once
        small = meshgen.stretch_box(3, 4, 3, E=1e5, nu=0.3, factor=1.02, jitter_amount=0.0)
        m = cc.Mesh.from_scene(small) if h == 0 else cc.Mesh(small.X, small.tets, small.pinned, E=1e5, nu=0.3, h=h)
        m.color()
        m.build_subspace(2)
        for precision in ("mixed", "fp64"):
            m.energy_grad(cc.to_soa(small.x0), cc.to_soa(small.x0) if h else None, precision=precision)
            m.sweep(cc.to_soa(small.x0), cc.to_soa(small.x0) if h else None, precision=precision)
        m.close()
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(2)
    x = cc.to_soa(sc.x0)
    m.sweep(x, precision="mixed")
    total, free_rows = int(m.export("sup_ptr")[-1]), int((sc.pinned == 0).sum())
    want = cc.from_soa(x) - sc.x0
    m.close()
    sizes = {"bases": 112 * total, "slots": 8 * (total + free_rows), "pairs": 8 * total + 800 * free_rows}
    assert sizes["pairs"] > sizes["slots"] + 48 * MIB
    return sc, sizes, want


def _mesh(sc, h=0.0, states=("mixed", "fp64")):
    m = cc.Mesh.from_scene(sc) if h == 0 else cc.Mesh(sc.X, sc.tets, sc.pinned, E=1e5, nu=0.3, h=h)
    m.color()
    x = cc.to_soa(sc.x0)
    for precision in states:  # allocates that path's solver state
        m.energy_grad(x, x if h else None, precision=precision, want_grad=False)
    return m, x


def _leave(size):
    """Holds all but `size` bytes of the device."""
    torch.cuda.empty_cache()
    return torch.empty(_free() - int(size), dtype=torch.uint8, device="cuda")


def test_a_dynamic_mesh_makes_no_pair_lists_before_a_float64_sweep(body):
    sc, sizes, _ = body
    m, x = _mesh(sc, h=1e-2)
    before = _free()
    m.build_subspace(2)
    m.sweep(x, x.clone(), precision="mixed")
    assert before - _free() <= sizes["bases"] + sizes["slots"] + 48 * MIB
    m.sweep(x, x.clone(), precision="fp64")
    assert before - _free() >= sizes["bases"] + sizes["pairs"]
    m.close()


def test_bases_come_before_the_pair_lists(body):
    sc, sizes, want = body
    m, x = _mesh(sc)
    hold = _leave(sizes["bases"] + sizes["slots"] + 48 * MIB)
    try:
        m.build_subspace(2)
        m.sweep(x, precision="mixed")
        got = cc.from_soa(x) - sc.x0
    finally:
        del hold
        torch.cuda.empty_cache()
    m.close()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()


def test_solver_state_takes_the_place_of_the_pair_lists(body):
    sc, sizes, want = body
    m, x = _mesh(sc, states=())
    m.build_subspace(2)
    hold = _leave(64 * MIB)  # the mixed state takes 83 MiB
    try:
        m.sweep(x, precision="mixed")
        got = cc.from_soa(x) - sc.x0
    finally:
        del hold
        torch.cuda.empty_cache()
    m.close()
    assert np.abs(got - want).max() <= 1e-4 * np.abs(want).max()


def test_a_call_after_one_that_ran_out_of_memory_works(body):
    sc, sizes, want = body
    m, x = _mesh(sc)
    hold = _leave(sizes["bases"] / 2)
    try:
        with pytest.raises(cc.CCError) as e:
            m.build_subspace(2)
        assert e.value.status == cc.ERR_OOM
    finally:
        del hold
        torch.cuda.empty_cache()
    with pytest.raises(cc.CCError):  # no subspace, so no sweep that reads one
        m.sweep(x, precision="mixed")
    m.build_subspace(2)
    m.sweep(x, precision="mixed")
    m.close()
    assert np.abs(cc.from_soa(x) - sc.x0 - want).max() <= 1e-4 * np.abs(want).max()
