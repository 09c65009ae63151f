"""Kernels at the sizes where their tiles, slices and dispatch rules change.

Tolerances:
* the integrator's cells do not depend on the batch that they are part of (CTA
  shape, number of CTAs, turns): exact equality.  Against the oracle both sides
  run the same BDF method at rtol 1e-6; over the few steps here their step
  sequences agree, so the difference is what rounding leaves, bounded by the
  integration tolerance.
* k': |x| 2^-53 per rounding of the exponent x = ln k' (at most four of them on
  either side) plus 8 units in the last place for the factors; results below the
  normal range are compared to 1e-300.
* f and J: 1e-12 of the sum of their terms' magnitudes, as for the other sizes.
* the adjoint's arithmetic does not depend on how many CTAs share a cell: exact
  equality between a pass of few cells and one of many.
"""
import copy

import numpy as np
import pytest

from oracle import bdf as ob
from oracle import kinetics as ok
from oracle import network as on
from synth import cells as sc
from synth import network as sn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as _t
    assert _t.cuda.is_available(), "these tests need a CUDA GPU"
    return _t


@pytest.fixture(scope="module")
def B(torch):
    from paper_2312_04998_gb300 import build
    build.build()
    from paper_2312_04998_gb300 import binding
    return binding


def dev(torch, a, ld):
    h = np.zeros((a.shape[0], ld))
    h[:, : a.shape[1]] = a
    return torch.tensor(h, dtype=torch.float64, device="cuda")


def workload(n_s, n_r, C):
    d = sn.generate(2312, n_s, n_r)
    T, nH, Av = sc.conditions(4998, C, (10.0, 300.0), (1e2, 1e6), (0.0, 10.0))
    return d, ok.rate_coefficients(d, T, nH, Av), sc.loguniform_abundances(d, 4998, C)


def integrate(torch, B, d, k, y0, t_end, **opts):
    C = y0.shape[1]
    ld = B.pad_ld(C)
    st = B.State(B.Network(d, 0), C, **opts)
    yd, stats = dev(torch, y0, ld), B.stats_tensor(C, "cuda")
    code = st.integrate(dev(torch, k, ld), yd, t_end, C, stats)
    torch.cuda.synchronize()
    assert code == B.SM_OK, B.stats_to_numpy(stats)["status"]
    return yd.cpu().numpy()[:, :C]


# tails of less than a block, of a few blocks (four-warp CTAs when cells are
# many), and of more blocks than those take
@pytest.mark.parametrize("size", [(32, 180), (45, 300), (70, 560), (120, 1200), (180, 1900)])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "tf32"])
def test_integrator_batches(torch, B, size, precision):
    C = 311   # more than there are SMs
    d, k, y0 = workload(*size, C)
    t_end = 1e3
    y = integrate(torch, B, d, k, y0, t_end, precision=precision)
    few = [0, 7, 31, 32, 310]
    alone = integrate(torch, B, d, k[:, few], y0[:, few], t_end, precision=precision)
    assert np.array_equal(alone, y[:, few])
    ref = ob.integrate_cell(d, k[:, 7], y0[:, 7], t_end, ob.BDFOptions(), on.stoichiometry(d)).y
    assert np.all(np.abs(y[:, 7] - ref) <= 1e-6 * np.abs(ref) + 1e-16)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_integrator_paths_agree(torch, B, precision):
    """A batch that goes through one launch per kernel class, and some of its
    cells through the persistent kernel: the same sums in the same order."""
    C = 6150
    d, k, y0 = workload(32, 180, 64)
    k, y0 = np.tile(k, (1, 97))[:, :C], np.tile(y0, (1, 97))[:, :C]
    few = [0, 5, 63]
    many = integrate(torch, B, d, k, y0, 1e3, precision=precision)
    alone = integrate(torch, B, d, k[:, few], y0[:, few], 1e3, precision=precision)
    assert np.array_equal(alone, many[:, few])
    assert np.array_equal(many[:, 64 * 95 + 5], many[:, 5])


def test_rates_outside_the_ordinary_range(torch, B):
    """Zero exponents, underflow and overflow, coefficients and conditions that
    the fixed-point form does not take."""
    d = copy.deepcopy(sn.generate(2312, 32, 180))
    two = np.nonzero(np.asarray(d.rclass) == 0)[0]
    d.beta[two[0]] = d.gamma[two[0]] = 0.0
    d.gamma[two[1]] = 9.0e3      # below the normal range at 10 K
    d.gamma[two[2]] = 2.0e5      # 0 at 10 K
    d.gamma[two[3]] = -5.0e3
    d.alpha[two[4]] = 1e-60
    d.alpha[two[5]] = 1e45
    d.alpha[two[6]] = 1e-36
    C = 33
    T = np.linspace(10.0, 3000.0, C)
    nH = 10.0 ** np.linspace(-38.0, 38.0, C)
    Av = np.linspace(0.0, 400.0, C)
    chi = 10.0 ** np.linspace(-40.0, 5.0, C)
    chi[3] = 0.0
    ld = B.pad_ld(C)
    kd = torch.zeros((d.n_r, ld), dtype=torch.float64, device="cuda")
    tt = lambda a: torch.tensor(a, dtype=torch.float64, device="cuda")
    net = B.Network(d, 0)
    net.rates_eval_chi(tt(T), tt(nH), tt(Av), tt(chi), kd, C)
    net.sync()
    got = kd.cpu().numpy()[:, :C]
    with np.errstate(all="ignore"):
        ref = ok.rate_coefficients(d, T, nH, Av, chi=chi)
    x = (np.abs(np.log(np.abs(d.alpha)))[:, None] + np.abs(d.beta)[:, None] * np.abs(np.log(T / 300.0))[None, :]
         + np.abs(d.gamma)[:, None] * np.maximum(1.0 / T, Av)[None, :])
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    tol = (8.0 * x + 16.0) * 2.0 ** -53
    assert np.all(np.abs(got - ref)[fin] <= (tol * np.abs(ref))[fin] + 1e-300)


@pytest.mark.parametrize("size", [(16, 40), (64, 500)])
@pytest.mark.parametrize("C", [1, 31, 33, 65])
@pytest.mark.parametrize("fmt", [("crs", "none", 1, 1), ("crs", "rcm", 1, 1), ("sell", "nnz", 8, 64)])
def test_rhs_and_jacobian_edges(torch, B, size, C, fmt):
    d, k, y = workload(*size, C)
    ld = B.pad_ld(C)
    net = B.Network(d, 0)
    net.set_format(*fmt)
    kd, yd = dev(torch, k, ld), dev(torch, y, ld)
    f = torch.full((d.n_s, ld), -7.0, dtype=torch.float64, device="cuda")
    net.rhs_eval(kd, yd, f, C)
    ptr, col = net.export(B.X_JPAT_PTR), net.export(B.X_JPAT_COL)
    J = torch.full((len(col), ld), -7.0, dtype=torch.float64, device="cuda")
    net.jac_eval(kd, yd, J, C)
    net.sync()
    f, J = f.cpu().numpy(), J.cpu().numpy()
    assert np.all(f[:, C:] == -7.0) and np.all(J[:, C:] == -7.0)
    assert np.all(np.abs(f[:, :C] - ok.rhs(d, k, y)) <= 1e-12 * ok.rhs_scale(d, k, y) + 1e-300)
    S, rows = on.stoichiometry(d), np.repeat(np.arange(d.n_s), np.diff(ptr))
    for c in {0, C - 1}:
        ref, scale = ok.jacobian(d, k[:, c], y[:, c], S), ok.jacobian_scale(d, k[:, c], y[:, c], S)
        assert np.all(np.abs(J[:, c] - ref[rows, col]) <= 1e-12 * scale[rows, col] + 1e-300)


@pytest.mark.parametrize("size", [(32, 180), (180, 1900)])
def test_adjoint_cells_share_ctas(torch, B, size):
    """A pass of 3 cells (several CTAs a cell) and one of 190 (one each)."""
    C, targets = 190, 5
    d, k, y0 = workload(*size, C)
    net = B.Network(d, 0)

    def run(cells):
        n, ld = len(cells), B.pad_ld(len(cells))
        st = B.State(net, n, precision="fp64", record_steps=128)
        kd, yd = dev(torch, k[:, cells], ld), dev(torch, y0[:, cells], ld)
        assert st.integrate(kd, yd, 1e2, n, B.stats_tensor(n, "cuda")) == B.SM_OK
        cot = torch.zeros((targets, d.n_s, ld), dtype=torch.float64, device="cuda")
        cot[:, :, :n] = torch.tensor(np.random.default_rng(5).random((targets, d.n_s, C))[:, :, cells], device="cuda")
        grad = torch.zeros((targets, d.n_r, ld), dtype=torch.float64, device="cuda")
        g0 = torch.zeros_like(cot)
        assert st.adjoint(kd, cot, grad, grad_y0=g0) == B.SM_OK
        torch.cuda.synchronize()
        return grad.cpu().numpy()[:, :, :n], g0.cpu().numpy()[:, :, :n]

    few = [0, 77, 189]
    a, b = run(few), run(list(range(C)))
    assert np.all(np.isfinite(a[0])) and np.any(a[0] != 0.0)
    assert np.array_equal(a[0], b[0][:, :, few]) and np.array_equal(a[1], b[1][:, :, few])
