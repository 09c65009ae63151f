"""The integrator's launch-per-class kernels, on the cases of the integrator's
own tests.

A state of large capacity is integrated by one launch per kernel class (see
sm_state_create), whatever the number of cells of the call; the tests of
test_gpu_integrate.py and test_gpu_thermal.py make states as small as their
batches, which one persistent kernel integrates.  Here the same tests, with
their inputs and tolerances, get states whose capacity puts them on the
launch-per-class path: its gather shapes, graphs, compaction, checkpoints, split
Newton rounds, reduced precisions and coupled-temperature kernels.  The number
of launches shows which path ran.
"""
import pytest

from tests import test_gpu_integrate as ti
from tests import test_gpu_thermal as tt
from tests.test_gpu_integrate import B, moderate_case, small_case, strat_case, torch  # noqa: F401

pytestmark = pytest.mark.gpu

# capacity beyond the batch from which a network's states take this path
CAPACITY = {32: 12288, 33: 12288, 470: 24576}


class ClassPath:
    """The binding, with states of a capacity that takes the class path."""

    def __init__(self, B):
        self._B, self._states = B, []

    def __getattr__(self, name):
        return getattr(self._B, name)

    def State(self, net, C, **opts):
        st = self._B.State(net, CAPACITY[net.n_s] + C, **opts)
        self._states.append(st)
        return st

    def finish(self):
        launches = [st.timing()[0] for st in self._states]
        for st in self._states:
            st.close()
        # (the persistent kernel: a handful of launches)
        assert max(launches) > 200, launches


@pytest.fixture()
def P(B):  # noqa: F811
    p = ClassPath(B)
    yield p
    p.finish()


ALL = pytest.mark.parametrize("precision", ["fp64", "mixed", "tf32"])
TWO = pytest.mark.parametrize("precision", ["fp64", "mixed"])
REDUCED = pytest.mark.parametrize("precision", ["mixed", "tf32"])


@ALL
def test_small_network(torch, P, small_case, precision):  # noqa: F811
    ti.test_small_network_matches_oracle(torch, P, small_case, precision)


@REDUCED
def test_large_network(torch, P, strat_case, precision):  # noqa: F811
    """Eleven blocks of tail: the trailing updates in FP32 and on the tensor cores."""
    ti.test_large_network_matches_oracle(torch, P, strat_case, precision)


@ALL
def test_conservation(torch, P, small_case, moderate_case, precision):  # noqa: F811
    ti.test_conservation_gpu(torch, P, small_case, moderate_case, "stiff", precision)


def test_nan_cell(torch, P):  # noqa: F811
    ti.test_nan_cell_is_isolated(torch, P)


def test_graph_of_a_reused_state(torch, P):  # noqa: F811
    ti.test_state_reuse_with_new_end_time(torch, P)


@TWO
def test_compaction(torch, P, precision):  # noqa: F811
    ti.test_compaction_is_bit_identical(torch, P, precision)


@TWO
def test_split_newton_rounds(torch, P, precision):  # noqa: F811
    ti.test_split_newton_rounds_are_bit_identical(torch, P, precision)


@ALL
@pytest.mark.parametrize("with_factors", [True, False])
def test_save_load_resume(torch, P, with_factors, precision):  # noqa: F811
    ti.test_state_save_load_resume(torch, P, with_factors, precision)


@ALL
def test_step_replay(torch, P, precision):  # noqa: F811
    ti.test_step_replay_matches_oracle(torch, P, precision)


@pytest.mark.parametrize("order", ["none", "nnz", "rcm"])
@pytest.mark.parametrize("kc", [8, 16, 32])
def test_gather_shapes(torch, P, moderate_case, order, kc):  # noqa: F811
    ti.test_integrator_gather_shapes(torch, P, moderate_case, order, kc)


@ALL
def test_coupled_temperature(torch, P, precision):  # noqa: F811
    tt.test_small_network_matches_oracle(torch, P, precision)


@TWO
def test_coupled_temperature_closed_form(torch, P, precision):  # noqa: F811
    tt.test_grain_coupling_closed_form(torch, P, precision)


@TWO
def test_coupled_temperature_steps(torch, P, precision):  # noqa: F811
    tt.test_step_replay_matches_oracle(torch, P, precision)
