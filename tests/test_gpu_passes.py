"""Operator passes with run-time radices against the oracle's FFT operator:
lengths of one, two and three stages, radices of both register classes, ragged
numbers of lines, planes of both classes of pass B and planes too large to
stage their spectrum.  Tolerances are those of the operator's other parity
tests (complex128 1e-12, complex64 2e-6 relative L2); the entries come from
the device table (checked on their own), so that grids of any length are
quick."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import jm, operator as op  # noqa: E402
from paper_1803_06237_gb300 import workloads  # noqa: E402

pytestmark = pytest.mark.gpu

# grid -> circulant: 1; 4 x 5 x 4; 16 (one radix); 25 x 25; 4096 (16^3); 675 x 64 x 25; 128 x 72 x 30;
# Mz = 32 (large class); My = 128 and 150 (radices 8 and 10 fused); a plane of 72 KB
GRIDS = [(1, 1, 1), (2, 3, 2), (8, 2, 1), (313, 4, 3), (2040, 2, 2), (333, 31, 13), (64, 35, 15), (17, 7, 16),
         (5, 64, 7), (9, 75, 6), (40, 12, 12), (600, 23, 4)]


@pytest.mark.parametrize("grid", GRIDS)
@pytest.mark.parametrize("dtype,tol", [(np.complex64, 2e-6), (np.complex128, 1e-12)])
def test_operator_and_source(grid, dtype, tol):
    from paper_1803_06237_gb300 import vie
    plan = vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085)
    eps = workloads.random_permittivity(grid, seed=3)
    vie.vie_set_permittivity(plan, eps)
    x = workloads.random_currents(grid, seed=4).astype(dtype)
    xd = torch.from_numpy(x.ravel()).cuda()
    y, b = torch.empty_like(xd), torch.empty_like(xd)
    vie.vie_matvec(plan, xd, y)
    vie.vie_rhs_from_source(plan, xd, b)
    M = op.contrast_M(op.chi_from_permittivity(eps, 2.085))
    Gh = op.green_spectrum(vie.vie_get_toeplitz(plan), grid, tuple(2 * v for v in grid))
    for got, ref in ((y, op.matvec(Gh, grid, M, x)), (b, op.rhs_from_source(Gh, grid, M, x))):
        got = got.cpu().numpy().astype(np.complex128)
        assert np.linalg.norm(got - ref.ravel()) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("grid", [(3, 2, 2), (20, 13, 9), (31, 30, 12), (9, 40, 5)])
@pytest.mark.parametrize("dtype,tol", [(np.complex64, 2e-6), (np.complex128, 1e-12)])
def test_jm_operator(grid, dtype, tol):
    from oracle import greens
    from paper_1803_06237_gb300 import vie
    plan = vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085)
    eps = workloads.random_permittivity(grid, seed=5)
    mu = workloads.random_permittivity(grid, seed=6)
    vie.vie_set_permittivity(plan, eps)
    vie.vie_set_permeability(plan, mu)
    nx, ny, nz = grid
    u = np.concatenate([workloads.random_currents(grid, seed=7), workloads.random_currents(grid, seed=8)]).astype(dtype)
    ud = torch.from_numpy(u.ravel()).cuda()
    y = torch.empty_like(ud)
    vie.vie_jm_matvec(plan, ud, y)
    size = tuple(2 * v for v in grid)
    kappa = plan.info()["kappa"]
    Gh = op.green_spectrum(vie.vie_get_toeplitz(plan), grid, size)
    Ch = jm.curl_spectrum(greens.curl_octant_table(kappa, grid), grid, size)
    ref = jm.matvec(Gh, Ch, grid, op.contrast_M(op.chi_from_permittivity(eps, 2.085)), jm.mu_contrast(mu), u, kappa)
    got = y.cpu().numpy().astype(np.complex128)
    assert np.linalg.norm(got - ref.ravel()) <= tol * np.linalg.norm(ref)


# planes too large for one CTA: every z length of the split pass B (5, 8, 9,
# 12, 15, 15, 18, 20, 24, 24, 25, 27, 30, 32), with and without a middle kx, ky
# that is its own image, last tiles of one to sixteen cells
SPLIT = [(2, 961, 3), (3, 601, 4), (4, 545, 5), (2, 405, 6), (3, 325, 7), (4, 338, 8), (2, 270, 9), (3, 243, 10),
         (4, 203, 11), (6, 211, 12), (2, 200, 13), (3, 182, 14), (4, 163, 15), (5, 152, 16)]


# planes that fit one block in complex64 but have no split into its radices; x
# and y lines of 324 = 9 6 6 and 400 = 10 10 4
SPLIT_SMALL = [(5, 150, 6), (4, 95, 12), (3, 170, 7), (6, 81, 15), (2, 101, 11), (162, 4, 3), (200, 162, 8),
               (3, 200, 7)]


@pytest.mark.parametrize("grid", SPLIT + SPLIT_SMALL)
@pytest.mark.parametrize("dtype,tol", [(np.complex64, 2e-6), (np.complex128, 1e-12)])
def test_operator_on_large_planes(grid, dtype, tol):
    test_operator_and_source(grid, dtype, tol)


# the cross-section with compiled strides (23 x 11 in 45 x 24), both operators
def test_compiled_cross_section():
    for dtype, tol in ((np.complex64, 2e-6), (np.complex128, 1e-12)):
        test_operator_and_source((13, 23, 11), dtype, tol)
        test_jm_operator((13, 23, 11), dtype, tol)


# the planes whose radices are compiled in (45 x 24 and 48 x 24) with every cross-section that meets in them
@pytest.mark.parametrize("grid", [(13, 21, 11), (12, 21, 12), (7, 22, 11), (16, 22, 12), (9, 23, 12), (13, 24, 11),
                                  (20, 24, 12)])
def test_compiled_planes(grid):
    from paper_1803_06237_gb300 import vie
    assert vie.vie_plan_create(grid, 0.02, 4.05, 2.085).info()["m"][1:] == (48 if grid[1] == 24 else 45, 24)
    test_operator_and_source(grid, np.complex64, 2e-6)
    test_jm_operator(grid, np.complex64, 2e-6)
