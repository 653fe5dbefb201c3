"""Which row build a float64 sweep takes by default: from the positions, but the
store and gather for a mesh with one vertex of many tets, whose shared memory
would leave every row too few warps.  The default's sweep has the bits of the
build that the switch names, and the gather's per-tet pass is launched or not.
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402
from test_gpu_rows import _spindle  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,rows", [(24, 1), (48, 1), (60, 0), (120, 0), (300, 0)])
def test_float64_rows_by_default(count, rows):
    sc = meshgen.stretch_box(3, 4, 3, E=1e5, nu=0.3, factor=1.1, jitter_amount=0.05, seed=4)
    X, tets, pinned, x0 = _spindle(count)
    X, tets = np.concatenate([sc.X, X]), np.concatenate([sc.tets, tets + sc.n])
    pinned, x0 = np.concatenate([sc.pinned, pinned]), np.concatenate([sc.x0, x0])
    out = []
    for switch in (-1, rows):
        m = cc.Mesh(X, tets, pinned, E=1e5, nu=0.3)
        m.color()
        m.build_subspace(1)
        m.set_sweep_variant(rows_from_positions=switch)
        x = cc.to_soa(x0)
        m.profile_enable(True)
        m.sweep(x, precision="fp64")
        out.append((cc.from_soa(x), m.profile_read()[cc.PROFILE_CLASSES[0]]["launches"]))
        m.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1] and (out[0][1] > 0) == (rows == 0)
