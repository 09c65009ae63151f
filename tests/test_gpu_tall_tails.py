"""The persistent integrator on networks whose tail has more 32-row blocks than
a CTA has warps, or whose sparse head has more rows than a CTA has threads: the
substitution then works on the further blocks in place and takes the head in
several passes.

Tolerances: the oracle runs the same method at rtol 1e-6.  A wrong factor or
substitution is repaired by further Newton iterations, so it shows in the
counters first: no convergence failures beyond the oracle's, and Newton
iterations within a tenth of its number (a decision that rounding turns costs one
or two).  Where a step is chosen differently the solutions part by their global
errors, a few units of the tolerance over these 30 to 100 steps: 10 units.
"""
import numpy as np
import pytest

from oracle import bdf as ob
from oracle import network as on
from synth import network as sn
from tests.test_gpu_edges import B, dev, torch, workload  # noqa: F401

pytestmark = pytest.mark.gpu


def sparse(n_s, n_r, reach):
    """n_r random reactions a + b -> c + d; all species within `reach` of the
    first one where reach > 0."""
    rng = np.random.default_rng(n_s)
    a = rng.integers(0, n_s, n_r)
    pick = lambda: (a + rng.integers(-reach, reach + 1, n_r)) % n_s if reach else rng.integers(0, n_s, n_r)
    reac = np.stack([a, pick()], axis=1).astype(np.int32)
    prod = np.stack([pick(), pick(), -np.ones(n_r, int), -np.ones(n_r, int)], axis=1).astype(np.int32)
    return sn.NetDesc(names=[f"s{i}" for i in range(n_s)], comp=np.zeros((n_s, 1), np.int32), reactants=reac,
                      products=prod, rclass=np.zeros(n_r, np.int8), alpha=np.ones(n_r), beta=np.zeros(n_r),
                      gamma=np.zeros(n_r))


def case(kind, n_s, n_r, C):
    if kind == "synth":
        return *workload(n_s, n_r, C), 1e3
    d = sparse(n_s, n_r, 3 if kind == "chain" else 0)
    rng = np.random.default_rng(7)
    return d, 10.0 ** rng.uniform(-3.0, 2.0, (n_r, C)), 10.0 ** rng.uniform(-4.0, 0.0, (n_s, C)), 0.01


# blocks of tail / rows of head: 13 / 122, 16 / 195, 13 / about 510, 10 / about
# 400 (a second pass of 384 threads), 1 / about 590 (of four warps where the
# cells are many)
@pytest.mark.parametrize("kind,n_s,n_r,C,precision", [
    ("synth", 510, 6800, 3, "mixed"), ("synth", 510, 6800, 3, "tf32"),
    ("synth", 700, 7000, 3, "mixed"), ("synth", 700, 7000, 3, "tf32"),
    ("sparse", 900, 1000, 3, "mixed"), ("sparse", 900, 1000, 3, "tf32"),
    ("sparse", 740, 830, 3, "fp64"), ("sparse", 740, 830, 3, "mixed"), ("sparse", 740, 830, 3, "tf32"),
    ("chain", 600, 1200, 3, "fp64"), ("chain", 600, 1200, 311, "fp64"), ("chain", 600, 1200, 311, "mixed")])
def test_integration_matches_oracle(torch, B, kind, n_s, n_r, C, precision):  # noqa: F811
    d, k, y0, t_end = case(kind, n_s, n_r, C)
    net = B.Network(d, 0)
    head = net.info()["lu_head"]
    assert (n_s - head > 12 * 32) if n_s - head > 350 else head > 384
    ld = B.pad_ld(C)
    st = B.State(net, C, precision=precision)
    yd, stats = dev(torch, y0, ld), B.stats_tensor(C, "cuda")
    assert st.integrate(dev(torch, k, ld), yd, t_end, C, stats) == B.SM_OK
    torch.cuda.synchronize()
    assert st.timing()[0] < 200      # the persistent kernel's launches
    y, s = yd.cpu().numpy()[:, :C], B.stats_to_numpy(stats)
    S = on.stoichiometry(d)
    for c in (0, C - 1):
        r = ob.integrate_cell(d, k[:, c], y0[:, c], t_end, ob.BDFOptions(), S)
        assert s["conv_fails"][c] <= r.conv_fails
        assert abs(int(s["newton_iters"][c]) - r.newton_iters) <= 0.1 * r.newton_iters + 2
        assert np.all(np.abs(y[:, c] - r.y) <= 1e-5 * np.abs(r.y) + 1e-15)
