"""GPU setup (entries) against 64-bit quadrature where its rules change: the
distance at which an offset moves from a block to a thread, every order of the
tent rule, wavenumbers on both sides of the short phase series, axes of one
voxel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import greens  # noqa: E402

pytestmark = pytest.mark.gpu


def _entries(kappa, D):
    """Offset D: the oracle next to the origin; from |D|_inf = 2 on the
    closed-form dyadic kernel by Gauss-Legendre on the 8 unit cells (the
    oracle's second differences of plane integrals cancel by |D|^2 there)."""
    if max(D) < 2:
        return greens.toeplitz_entries(kappa, [D])[0]
    x, w = np.polynomial.legendre.leggauss(18 if max(D) < 6 else 10)
    x, w = 0.5 * (x + 1), 0.5 * w
    t, wt = np.concatenate([x - 1, x]), np.concatenate([w * x, w * (1 - x)])
    v = [d + a for d, a in zip(D, np.meshgrid(t, t, t, indexing="ij"))]
    r2 = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
    r = np.sqrt(r2)
    e = wt[:, None, None] * wt[:, None] * wt * np.exp(-1j * kappa * r) / (4 * np.pi * r * r2)
    a, b = e * (r2 * kappa ** 2 - 1 - 1j * kappa * r), e * (3 - r2 * kappa ** 2 + 3j * kappa * r) / r2
    pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
    return np.array([np.sum(b * v[p] * v[q] + (a if p == q else 0)) for p, q in pairs])


@pytest.mark.parametrize("grid", [(1, 1, 1), (2, 1, 3), (10, 1, 1), (11, 2, 1), (1, 31, 2), (3, 12, 15), (40, 1, 10)])
@pytest.mark.parametrize("kappa", [0.0, 0.144, 0.145, 1.0])
def test_entries_across_the_rules(grid, kappa):
    """Each offset's entries relative to its largest component.  Rounding of the
    rule's nodes moves the reference's and this rule's sums by about 5e-16 each
    and the device adds a few units in the last place per point: 2e-14 bounds
    both with a margin of ten."""
    from paper_1803_06237_gb300 import vie
    plan = vie.vie_plan_create(grid, max(kappa, 0.1), 1.0 if kappa else 0.0, 1.0)
    assert plan.info()["kappa"] == pytest.approx(kappa)
    T = vie.vie_get_toeplitz(plan)
    kappa = plan.info()["kappa"]
    ref = np.empty_like(T)
    for z, y, x in np.ndindex(*T.shape[1:]):
        ref[:, z, y, x] = _entries(kappa, (x, y, z))
    err = np.abs(T - ref).max(axis=0) / np.abs(ref).max(axis=0)
    assert err.max() < 2e-14, (err.max(), np.unravel_index(err.argmax(), err.shape))
