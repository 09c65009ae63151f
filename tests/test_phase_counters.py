"""The phase counters of the two integrator kernels."""
import os
import subprocess
import sys

import numpy as np
import pytest

import bench
from paper_2312_04998_gb300 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_table_takes_the_kernel_that_ran():
    s = {k: np.array([3, 5]) for k in ("steps", "rejects", "conv_fails", "newton_iters", "jac_evals")}
    refresh, cell = np.zeros(16), np.zeros(16)
    with pytest.raises(RuntimeError):       # nothing counted is an error, not a table of zeros
        bench.phase_table(B, refresh, cell, s)
    cell[:11] = 24.0
    t = bench.phase_table(B, refresh, cell, s)
    assert [p[0] for p in t["phases"]] == B.CELL_PHASE_NAMES
    assert [p[1] for p in t["phases"]] == [1.0, 1.0, 3.0, 3.0, 3.0, 1.0, 3.0, 3.0, 3.0, 3.0, 3.0]
    refresh[:11], refresh[15] = 10.0, 5.0
    t = bench.phase_table(B, refresh, cell, s)
    assert [p[0] for p in t["phases"]] == B.PHASE_NAMES and t["refreshed_cells"] == 5
    assert t["total_cycles_per_cell"] == 22.0


RUN = """
import numpy as np, torch
from oracle import kinetics as ok
from synth import cells as sc, network as sn
from paper_2312_04998_gb300 import build, binding as B
build.build(phase_clocks=True)
B.use_phase_build()
d = sn.generate(2312, 32, 180)
C = 40
k = ok.rate_coefficients(d, *sc.conditions(4998, C, (10.0, 300.0), (1e2, 1e6), (0.0, 10.0)))
dev = lambda a: torch.nn.functional.pad(torch.tensor(a, dtype=torch.float64), (0, B.pad_ld(C) - C)).cuda()
net = B.Network(d, 0)
for cap in (C, 9000):
    B.phase_cycles(0, reset=True)
    B.cell_phase_cycles(0, reset=True)
    st, stats = B.State(net, cap), B.stats_tensor(C, "cuda")
    assert st.integrate(dev(k), dev(sc.atomic_start(d, C)), 1e10, C, stats) == B.SM_OK
    torch.cuda.synchronize()
    r, c, n = B.phase_cycles(0), B.cell_phase_cycles(0), int(B.stats_to_numpy(stats)["jac_evals"].sum())
    if cap == C:
        # (a tail of one block has no panel updates, nor the refresh U blocks)
        assert not r.any() and np.all(c[[0, 1, 2, 3, 4, 5, 6, 7, 8, 10]] > 0), (r, c)
    else:
        assert not c.any() and r[15] == n and np.all(r[:7] > 0) and r[10] > 0, (r, c, n)
print("counted")
"""


@pytest.mark.gpu
def test_each_kernel_counts_its_own_phases():
    p = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, capture_output=True, text=True)
    assert p.returncode == 0 and "counted" in p.stdout, p.stderr[-2000:]
