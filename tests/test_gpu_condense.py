"""The condensation with four lanes per vertex against the one with a lane per
vertex (run by the fused coupling kernel): colours that end inside a warp of
eight vertices, empty supports, local systems that fall back, and a colour on
either side of the line between the two.  Same roundings, so the same bits.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("size,schedule", [((2, 1, 1), "jacobi"), ((2, 3, 1), "jacobi"), ((4, 5, 3), "colored"),
                                           ((17, 16, 16), "jacobi"), ((18, 17, 16), "jacobi")])
def test_four_lanes_give_the_bits_of_one(size, schedule, precision):
    sc = meshgen.stretch_box(*size, E=1e5, nu=0.3, factor=1.2, jitter_amount=0.05, seed=3)
    m = cc.Mesh.from_scene(sc)
    m.color()
    m.build_subspace(1)
    wild = meshgen.normal(7, np.arange(3 * sc.n)).reshape(-1, 3) * sc.cell * (sc.pinned == 0)[:, None]
    for update in ("cc", "jgs2"):
        for amount in (0.02, 0.5):  # the second turns tets over: indefinite local systems
            got = []
            for fused in (0, 1):
                m.set_sweep_variant(fused_condense=fused)
                x = cc.to_soa(sc.x0 + amount * wild)
                try:
                    st = m.sweep(x, update=update, schedule=schedule, precision=precision)
                    got.append((cc.from_soa(x), st.fallback_empty, st.fallback_reduced, st.fallback_schur))
                except cc.CCError:  # a singular vertex: both report it
                    got.append((cc.from_soa(x), "error"))
            np.testing.assert_array_equal(got[0][0], got[1][0])
            assert got[0][1:] == got[1][1:]
    m.close()
