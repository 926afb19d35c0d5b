"""The network's complex64 output v + y s over the range of scales: at every
scale of v the FP32 result is the complex128 one rounded once (half a unit in
the last place, plus the 2^-29 of the 64-bit sum's own rounding)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-118, -101, -99, -40, 0, 60, 99, 101, 110])
def test_output_is_rounded_once_at_every_scale(exponent):
    grid = (24, 9, 5)
    plan = vie.vie_plan_create(grid, 0.02, 4.05, 2.085)
    vie.vie_set_permittivity(plan, workloads.random_permittivity(grid, seed=61))
    params = np.random.default_rng(62).standard_normal(vie.vie_net_param_count()).astype(np.float32) * 0.05
    net = vie.vie_net_create(params)
    v = (workloads.random_currents(grid, seed=63) * 2.0 ** exponent).astype(np.complex64).ravel()
    v32 = torch.from_numpy(v).cuda()
    v64 = torch.from_numpy(v.astype(np.complex128)).cuda()
    z32, z64 = torch.empty_like(v32), torch.empty_like(v64)
    vie.vie_net_apply(net, plan, v32, z32)
    vie.vie_net_apply(net, plan, v64, z64)
    torch.cuda.synchronize()
    got, ref = (torch.view_as_real(z).cpu().numpy().astype(np.float64) for z in (z32, z64))
    assert not np.array_equal(got, torch.view_as_real(v64).cpu().numpy())
    ulp = np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64)
    assert (np.abs(got - ref) <= 0.5000001 * ulp).all()
