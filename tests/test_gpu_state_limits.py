"""Networks that no state is made for."""
import numpy as np
import pytest

from synth import network as sn
from tests.test_gpu_edges import B, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,taken", [(14000, True), (15000, False)])
@pytest.mark.parametrize("opts", [{}, {"precision": "mixed"}, {"record_steps": 16}])
def test_reactions_beyond_the_refresh_table(torch, B, n_r, taken, opts):  # noqa: F811
    """The refresh holds two derivatives per reaction in shared memory (16 bytes of
    227 KB each), so about 14,300 reactions are the limit, also where they have
    one reactant each and the persistent kernel's tables would fit."""
    n_s = 100
    rng = np.random.default_rng(3)
    none = -np.ones(n_r, int)
    a = np.arange(n_r) % n_s
    d = sn.NetDesc(names=[f"s{i}" for i in range(n_s)], comp=np.zeros((n_s, 1), np.int32),
                   reactants=np.stack([a, none], axis=1).astype(np.int32),
                   products=np.stack([(a + rng.integers(1, n_s, n_r)) % n_s, none, none, none], axis=1).astype(np.int32),
                   rclass=np.full(n_r, sn.COSMIC_RAY, np.int8), alpha=np.ones(n_r), beta=np.zeros(n_r),
                   gamma=np.zeros(n_r))
    net = B.Network(d, 0)
    if taken:
        B.State(net, 4, **opts).close()
    else:
        with pytest.raises(B.StoichError):
            B.State(net, 4, **opts)
