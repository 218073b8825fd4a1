"""The limits of a persistent 1D run.  Blocks that run out of polls at the grid
barrier: an error status, no half-taken step counted, no further run from the
barrier's short count, and a context that is usable again once its state is set.
Blocks that do not all fit: the same steps, to the same bits, as graph replays."""
import numpy as np
import pytest

import paper_2108_12742_gb300 as eno
from paper_2108_12742_gb300 import inputs

pytestmark = pytest.mark.gpu

TIMEOUT, EINVAL = 5, 1
N = 2000


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_12742_gb300 import build
    build.build()


def _solver(precision):
    return eno.Solver((N,), (-5.0,), (5.0,), system=eno.EULER, order=5, precision=precision,
                      bc=eno.TRANSMISSIVE)


@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
def test_barrier_polls_run_out_as_a_timeout_status(precision):
    U = inputs.titarev_toro(N)
    with _solver(precision) as s:
        assert s.launches_per_step() == 0  # the persistent run
        s.init_state(U)
        s.advance_steps(5, 0.5)
        good = s.get_state()
        s.init_state(U)
        s.set_run_poll_limit(0)
        # (more steps than one launch takes: the launches after the one that gave up)
        with pytest.raises(eno.EnoaoError) as e:
            s.advance_steps(10000, 0.5)
        assert e.value.status == TIMEOUT and "timed out" in str(e.value)
        # block 0 had begun the first step, which no block finished
        assert s.stats().steps == 0 and s.stats().t == 0.0
        # the error stays, with any poll limit, until the state is set
        s.set_run_poll_limit(-1)
        for run in (lambda: s.advance_steps(2, 0.5), lambda: s.advance(1.0, cfl=0.5, max_steps=2)):
            with pytest.raises(eno.EnoaoError) as e:
                run()
            assert e.value.status == TIMEOUT
            assert s.stats().steps == 0 and s.stats().t == 0.0
        s.init_state(U)
        s.advance_steps(5, 0.5)
        assert s.stats().steps == 5
        assert np.array_equal(s.get_state(), good)


@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
def test_blocks_that_do_not_fit_step_as_graphs(precision):
    U = inputs.titarev_toro(N)
    with _solver(precision) as s:
        def runs():
            s.init_state(U)
            s.advance_steps(37, 0.5)
            a = s.get_state()
            s.init_state(U)
            t, k = s.advance(0.05, cfl=0.5)
            assert t == 0.05
            return a, s.get_state(), k
        a, b, k = runs()
        s.set_run_block_limit(1)
        assert s.launches_per_step() == 0  # not known yet
        for _ in range(2):
            a1, b1, k1 = runs()
            assert s.launches_per_step() > 0
            assert np.array_equal(a, a1) and np.array_equal(b, b1) and k == k1
        s.set_run_block_limit(-1)
        assert s.launches_per_step() == 0


def test_limits_reject_bad_values():
    with _solver(eno.FP64) as s:
        for knob in (s.set_run_poll_limit, s.set_run_block_limit):
            with pytest.raises(eno.EnoaoError) as e:
                knob(-2)
            assert e.value.status == EINVAL
