"""Two host threads applying operators of different sizes on their own streams:
the same kernels, launched with different amounts of shared memory.  Every call
is accepted and the last result has the bits of the one computed alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie, workloads  # noqa: E402

pytestmark = pytest.mark.gpu


# planes of two sizes past 48 KB; x lines of 900 and 2000 values
@pytest.mark.parametrize("grids", [((30, 30, 13), (30, 34, 14)), ((900, 23, 11), (2000, 23, 11))])
def test_two_threads_two_sizes(grids):
    def problem(grid):
        plan = vie.vie_plan_create(grid, 0.02, 2 * np.pi / 1.55, 2.085)
        vie.vie_set_permittivity(plan, workloads.random_permittivity(grid, seed=31))
        x = torch.from_numpy(workloads.random_currents(grid, seed=32).astype(np.complex64).ravel()).cuda()
        return plan, x, vie.vie_matvec(plan, x, torch.empty_like(x)).clone()

    problems = [problem(g) for g in grids]
    torch.cuda.synchronize()
    refused = []

    def work(plan, x, y, stream):
        for _ in range(15000):
            try:
                vie.vie_matvec(plan, x, y, stream=stream)
            except vie.VieError as e:
                refused.append(str(e))
        stream.synchronize()

    outs = [torch.empty_like(x) for _, x, _ in problems]
    threads = [threading.Thread(target=work, args=(plan, x, y, torch.cuda.Stream()))
               for (plan, x, _), y in zip(problems, outs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not refused, (len(refused), refused[0])
    for (_, _, alone), y in zip(problems, outs):
        assert torch.equal(y, alone)
