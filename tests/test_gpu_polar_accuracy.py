"""The polar rotation of Fixed Corotational's float64 gradient, tet by tet, is no
further from the exact one than the float64 Newton iteration's: compact, flat
(one small singular value) and needle-like (two) deformations.

Every tet is a body of its own with the unit corner at rest, mu = 1 and lam = 0,
so its gradient is V P = (F - R) / 3 with F read from the positions without
rounding, and R = F - 3 g to three roundings of entries of about 1.

Tolerance: the root mean square over 4 096 tets of R's error (Frobenius, against
the same iteration in extended precision) is at most 1.25 times the float64
iteration's on the same F, for another order of the sums, and 3e-16 for the nine
entries' roundings outside it.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu

TETS = 4096


def _inverse_transpose(Y):
    r0, r1, r2 = Y[:, 0], Y[:, 1], Y[:, 2]
    C = np.stack([np.cross(r1, r2), np.cross(r2, r0), np.cross(r0, r1)], axis=1)
    return C / np.sum(r0 * C[:, 0], axis=1)[:, None, None]


def _newton(F):
    """Y <- (g Y + (g Y)^-T) / 2 with Higham's scaling, in F's precision."""
    Y = F.copy()
    for _ in range(40):
        T = _inverse_transpose(Y)
        g = np.sqrt(np.sqrt(np.sum(T * T, axis=(1, 2)) / np.sum(Y * Y, axis=(1, 2))))[:, None, None]
        Y = (g * Y + T / g) / 2
    return Y


def _rotations(rng):
    q = rng.standard_normal((TETS, 4))
    w, x, y, z = (q / np.linalg.norm(q, axis=1)[:, None]).T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], axis=1).reshape(-1, 3, 3)


@pytest.mark.parametrize("second,third", [(0.8, 0.8), (1, 1e-2), (1, 1e-4), (0.2, 0.2), (0.1, 0.1), (1e-2, 1e-2),
                                          (1e-3, 1e-3)])
def test_rotation_is_as_accurate_as_the_float64_iteration(second, third):
    rng = np.random.default_rng(11)
    s = np.array([1.0, second, third]) * np.exp(0.3 * (rng.random((TETS, 3)) - 0.5) * [0, 1, 1])
    F = np.einsum("tik,tk,tjk->tij", _rotations(rng), s, _rotations(rng))
    corner = np.concatenate([np.zeros((1, 3)), np.eye(3)])
    x = np.zeros((TETS, 4, 3))
    x[:, 1:] = F.transpose(0, 2, 1)
    tets = np.arange(4 * TETS, dtype=np.int32).reshape(-1, 4)
    m = cc.Mesh(np.tile(corner, (TETS, 1)), tets, np.zeros(4 * TETS, dtype=np.uint8), E=2.0, nu=0.0, model="fcr")
    m.color()
    _, g, _ = m.energy_grad(cc.to_soa(x.reshape(-1, 3)), precision="fp64")
    m.close()
    R = F - 3 * cc.from_soa(g).reshape(-1, 4, 3)[:, 1:].transpose(0, 2, 1)
    want = _newton(F.astype(np.longdouble))

    def rms(A):
        return float(np.sqrt(np.mean(np.sum((A - want) ** 2, axis=(1, 2)))))

    assert rms(R) <= 1.25 * rms(_newton(F)) + 3e-16
