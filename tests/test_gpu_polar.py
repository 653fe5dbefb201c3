"""Fixed Corotational energy and gradient in float64 where the polar rotation's
float32 start is easy, coarse or fails: unit, stretched, flattened and
needle-like deformations (singular values down to 1e-4 and 1e-7), each turned by
a large rotation.

Tolerance: F and R carry float64 rounding (a few 1e-16) times the inverse of the
smallest sum of two singular values, and F - R, 0.02 to 0.1 at the first state,
cancels one to two digits: 1e-12 over that sum (1 at most), relative to the
largest gradient entry and to the energy.
"""
import numpy as np
import pytest

import meshgen
from oracle import fem

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stretch", [(1, 1, 1), (3, 0.5, 1), (1, 1, 1e-3), (1, 1e-4, 1e-4), (1e3, 1e2, 1e3),
                                     (1, 1e-7, 1e-7)])
def test_energy_and_gradient_match_the_oracle(stretch):
    sc = meshgen.stretch_box(4, 3, 5, E=1e5, nu=0.3, jitter_amount=0.05, seed=6)
    noise = meshgen.normal(7, np.arange(3 * sc.n)).reshape(-1, 3) * 0.02 * sc.cell
    c, s = np.cos(2.0), np.sin(2.0)
    A = np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]]) @ np.diag(stretch) @ np.array([[1, 0, 0], [0, c, s], [0, -s, c]])
    x = (sc.X + noise) @ A.T
    pb = fem.problem_from_scene(sc, "fcr")
    m = cc.Mesh.from_scene(sc, model="fcr")
    m.color()
    e, g, _ = m.energy_grad(cc.to_soa(x), precision="fp64")
    m.close()
    want_e, want_g = pb.energy(x), pb.gradient(x) * pb.free[:, None]
    low = sorted(stretch)
    tol = 1e-12 / min(1.0, low[0] + low[1])
    assert abs(e - want_e) <= tol * abs(want_e)
    assert np.abs(cc.from_soa(g) - want_g).max() <= tol * np.abs(want_g).max()
