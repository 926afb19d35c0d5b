"""The grid barriers' waits are bounded, and one block's time-out releases the
others: with a block missing, one block waits 50 ms and sets the abort word, the
rest, whose own limit is a second, leave by it.  The context stays usable."""
import time

import pytest

torch = pytest.importorskip("torch")

from paper_1803_06237_gb300 import vie  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("absent", [0, 3, 151])
def test_time_out_of_one_block_releases_the_others(absent):
    vie.load()
    assert vie.vie_probe_grid_barrier(-1, 50.0) is False
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    assert vie.vie_probe_grid_barrier(absent, 50.0) is True
    # two probes of 50 ms; either barrier's own limit alone is about a second
    assert time.perf_counter() - t0 < 0.6
    assert vie.vie_probe_grid_barrier(-1, 50.0) is False
    x = torch.ones(8, device="cuda")
    assert float(x.sum().item()) == 8.0
