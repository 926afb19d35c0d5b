"""Training's workspace on a grid whose weight-gradient operands do not fit the
bound on them together: the layers take turns, the memory held is that of the
activations and the bound, and the gradients are those of the FP32 kernels to
the rounding of the BF16 tensors (the bounds of the network's other tests)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu

LAYERS = [(8, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 32), (32, 6)]
BOUND = 1 << 30             # bytes of the operands past which layers take turns


# 2.1 GB of operands held at once, the largest layer's 0.6 GB; one layer alone past the bound
@pytest.mark.parametrize("grid", [(960, 160, 12), (1472, 200, 13)])
def test_operands_are_bounded(grid):
    nx, ny, nz = grid
    V = nx * ny * nz
    plan = vie.vie_plan_create(grid, 0.02, 4.05, 2.085)
    vie.vie_set_permittivity(plan, workloads.random_permittivity(grid, seed=41))
    g = torch.Generator(device="cuda").manual_seed(42)
    r, e = (torch.view_as_complex(torch.randn(3 * V, 2, generator=g, device="cuda")) for _ in range(2))
    params = np.random.default_rng(43).standard_normal(vie.vie_net_param_count()).astype(np.float32) * 0.03
    net = vie.vie_net_create(params)
    vie.vie_net_set_training(net, vie.VIE_TRAIN_TENSOR_BF16)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    vie.vie_net_zero_grad(net)
    loss = vie.vie_net_accumulate(net, plan, r, e)
    used = before - torch.cuda.mem_get_info()[0]
    # activations and their gradients: 32 channels of 2 bytes per level, by the tensors held; the network's
    # output in FP32; 64 MB for the partial sums and allocation granularity
    levels = [V]
    dims = (nx, ny)
    for _ in range(3):
        dims = tuple((d + 1) // 2 for d in dims)
        levels.append(dims[0] * dims[1] * nz)
    tensors = [2 + 3 + 4, 3 + 3 + 2, 3 + 3 + 2, 3 + 1]       # h, da, a; decin, u, ddecin; pre-activation gradients
    acts = sum(64 * t * v for t, v in zip(tensors, levels)) + 64 * V + 64 * V
    row = (nx + 63) // 64 * 64 * ny * nz
    assert used <= acts + max(BOUND, 2 * 160 * row) + (64 << 20), (used, acts)
    got = vie.vie_net_get_grads(net).astype(np.float64)
    vie.vie_net_set_training(net, vie.VIE_TRAIN_FP32)
    vie.vie_net_zero_grad(net)
    ref_loss = vie.vie_net_accumulate(net, plan, r, e)
    ref = vie.vie_net_get_grads(net).astype(np.float64)
    assert abs(loss - ref_loss) <= 1e-2 * ref_loss
    at = 0
    for ci, co in LAYERS:
        for size in (co * ci * 27, co):
            a, b = got[at:at + size], ref[at:at + size]
            at += size
            assert np.linalg.norm(a - b) <= 2e-2 * np.linalg.norm(b), (ci, co, size)
