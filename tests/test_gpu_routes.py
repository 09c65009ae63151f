"""Which kernels a state's capacity selects (see class_path_from)."""
import numpy as np
import pytest

from oracle import kinetics as ok
from synth import cells as sc
from synth import network as sn
from synth import thermal as sth
from tests.test_gpu_edges import B, dev, torch  # noqa: F401

pytestmark = pytest.mark.gpu

SMALL, PADDED, FULL, THREE = (32, 180), (64, 500), (90, 850), (120, 1200)


@pytest.mark.parametrize("size,precision,kind,by_class_from", [
    (SMALL, "mixed", "plain", 4608), (SMALL, "tf32", "recorded", 6144), (SMALL, "mixed", "temperature", 6144),
    (SMALL, "fp64", "plain", 6144), (SMALL, "fp64", "recorded", 12288), (SMALL, "fp64", "temperature", 12288),
    (PADDED, "mixed", "plain", 7168), (PADDED, "mixed", "temperature", 12288), (PADDED, "fp64", "recorded", 12288),
    (FULL, "mixed", "recorded", 16384), (FULL, "fp64", "temperature", None),
    (THREE, "tf32", "plain", 24576), (THREE, "mixed", "temperature", None), (THREE, "fp64", "temperature", 65536)])
def test_kernels_by_capacity(torch, B, size, precision, kind, by_class_from):  # noqa: F811
    """One launch per kernel class is a dozen launches an attempt, the persistent
    kernel many attempts a launch; two cells tell."""
    C = 2
    d = sn.generate(2312, *size)
    T, nH, Av = sc.conditions(4998, C, (10.0, 300.0), (1e2, 1e6), (0.0, 10.0))
    k, y0 = ok.rate_coefficients(d, T, nH, Av), sc.atomic_start(d, C)
    opts = {"precision": precision, **({"record_steps": 16} if kind == "recorded" else {})}
    if kind == "temperature":
        d = sth.with_temperature(d)
        th = sth.thermal_params(d)
        y0 = sth.thermal_start(d, y0, T)
    net = B.Network(d, 0)
    if kind == "temperature":
        net.set_thermal(th)
    ld = B.pad_ld(C)
    vec = lambda a: torch.tensor(np.asarray(a, dtype=float), device="cuda")
    for capacity, by_class in ((by_class_from - 1, False), (by_class_from, True)) if by_class_from else ((70000, False),):
        st = B.State(net, capacity, **opts)
        if kind == "temperature":
            st.set_cells(vec(nH), vec(Av), None, C)
        assert st.integrate(None if kind == "temperature" else dev(torch, k, ld), dev(torch, y0, ld), 1e4, C) == B.SM_OK
        assert (st.timing()[0] > 100) is by_class, (capacity, st.timing()[0])
        st.close()
