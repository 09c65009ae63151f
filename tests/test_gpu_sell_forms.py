"""The two forms of the SELL gather (see sell_ahead): the one that reads ahead,
for small batches, and the plain loop once the device's threads are busy."""
import numpy as np
import pytest

from tests.test_gpu_edges import B, dev, torch, workload  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [21000, 23000, 40000])   # 2.16, 2.36 and 4.1 rounds
def test_forms_agree(torch, B, C):  # noqa: F811
    """A row is the same chain of additions either way: the same bits."""
    d, k, y = workload(32, 180, 33)
    net = B.Network(d, 0)
    net.set_format("sell", "none", 32, 1)

    def f(cells):
        ld = B.pad_ld(len(cells))
        out = torch.full((d.n_s, ld), -7.0, dtype=torch.float64, device="cuda")
        net.rhs_eval(dev(torch, k[:, cells], ld), dev(torch, y[:, cells], ld), out, len(cells))
        net.sync()
        return out.cpu().numpy()[:, : len(cells)]

    assert np.array_equal(f(np.arange(C) % 33)[:, C - 66:], f(np.arange(C - 66, C) % 33))
