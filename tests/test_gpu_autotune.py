"""The autotuner does not end with a slower tile than the one it began with."""
import numpy as np
import pytest

import paper_2108_12742_gb300 as eno
from paper_2108_12742_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_12742_gb300 import build
    build.build()


def test_autotune_keeps_a_tile_that_beats_its_candidates():
    # white noise, FP64, one line: the work of a sweep is its slowest SM's, and tiles
    # of 15 cells, on twice as many SMs, take much less than the shortest candidate
    # along x (31 cells)
    n = 2000
    rng = np.random.default_rng(0)
    rho, p, u = (b + 0.3 * rng.uniform(-1, 1, (1, 1, n)) for b in (1.0, 1.0, 0.2))
    with eno.Solver((n,), (0.0,), (1.0,), system=eno.EULER, order=7, precision=eno.FP64) as s:
        s.init_state(inputs.conserved(rho, [u], p, 1.4).reshape(3, 1, 1, n))
        s.set_tiles(0, 1, 31)
        candidate = min(s.time_sweep(0, 50) for _ in range(3))
        s.set_tiles(0, 1, 15)
        before = min(s.time_sweep(0, 50) for _ in range(3))
        assert before < 0.9 * candidate  # else this case says nothing
        s.autotune()
        after = min(s.time_sweep(0, 50) for _ in range(3))
        assert after <= 1.05 * before, (s.get_tiles(0), before, after, candidate)
