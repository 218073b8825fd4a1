"""The persistent run of small 1D problems against the same steps taken stage by
stage (one sweep launch per stage): the same bits, at the sizes where its
tiles, blocks and step limits change."""
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


def _solver(system, n, order, precision, bc):
    lo = -1.0 if system == eno.SCALAR_ADVECTION else 0.0
    return eno.Solver((n,), (lo,), (1.0,), system=system, order=order, precision=precision, bc=bc)


# 11: the least; 15/16/17: one tile, the first with two; 2281: tiles of 16 on
# 152 SMs; 246/247: the last scalar problem in one block; 18241: tiles past
# 120 cells (256 threads); 38912/38913: the last persistent one, and one beyond
@pytest.mark.parametrize("system,sizes", [(eno.EULER, (11, 15, 16, 17, 333, 2281, 18241, 38912, 38913)),
                                          (eno.SCALAR_ADVECTION, (11, 121, 246, 247, 513, 18241))])
@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
def test_persistent_run_equals_stages(system, sizes, order, precision):
    for n in sizes:
        bc = eno.PERIODIC if n % 2 else eno.TRANSMISSIVE
        U0 = inputs.euler1d_riemann(n, seed=n) if system == eno.EULER else \
            inputs.advection_random(n, seed=n)
        with _solver(system, n, order, precision, bc) as s:
            s.init_state(U0)
            dts = []
            for _ in range(3):
                s.advance(1e9, cfl=0.5, max_steps=1)
                dts.append(s.stats().dt)
            run = s.get_state()
            assert s.stats().steps == 3
            s.init_state(U0)
            s.advance_steps(3, cfl=0.5)
            at_once = s.get_state()
            s.init_state(U0)
            for dt in dts:
                for k in range(3):
                    s.rk_stage(k, dt)
            stages = s.get_state()
        assert np.array_equal(run, stages), (n, np.abs(run - stages).max())
        assert np.array_equal(run, at_once), n


def test_persistent_run_limits_and_errors():
    n = 64
    with _solver(eno.SCALAR_ADVECTION, n, 5, eno.FP64, eno.PERIODIC) as s:
        U0 = inputs.advection_sine(n)
        s.init_state(U0)
        s.advance_steps(4099)  # more steps than one launch takes
        assert s.stats().steps == 4099
        a = s.get_state()
        s.init_state(U0)
        for k in (4096, 3):
            s.advance_steps(k)
        assert np.array_equal(a, s.get_state())
        s.init_state(U0)
        t, k = s.advance(0.1, cfl=0.5)
        assert t == 0.1 and s.stats().t == 0.1
        assert s.advance(0.1, cfl=0.5)[1] == k  # already there
    with _solver(eno.EULER, 400, 5, eno.FP64, eno.TRANSMISSIVE) as s:
        U = inputs.euler1d_sod(400)
        U[1, ..., :200] = -25.0 * U[0, ..., :200]  # a Mach-25 double rarefaction opens a vacuum
        U[1, ..., 200:] = 25.0 * U[0, ..., 200:]
        U[2] += 0.5 * U[1] ** 2 / U[0]
        s.init_state(U)
        with pytest.raises(eno.EnoaoError) as e:
            s.advance(1.0, cfl=0.5)
        assert e.value.status == 4
        s.init_state(inputs.euler1d_sod(400))
        s.advance(0.01, cfl=0.5)
        assert np.isfinite(s.get_state()).all()
