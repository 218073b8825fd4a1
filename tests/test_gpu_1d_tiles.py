"""Tiles of 1D problems where nothing but the launch of a stage, the fluxes or the
allocation-free step chooses them: the results do not depend on them.  (A run of a
small 1D problem takes tiles of its own; it ends where the device's SMs do.)"""
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


def _case(system, n):
    if system == eno.EULER:
        return inputs.titarev_toro(n), (-5.0,), (5.0,)
    return inputs.composite_wave(n), (-1.0,), (1.0,)


@pytest.mark.parametrize("system", [eno.EULER, eno.SCALAR_ADVECTION])
@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
@pytest.mark.parametrize("n", [11, 63, 64, 200, 2281, 20001])
def test_stages_fluxes_and_steps_do_not_depend_on_1d_tiles(system, order, precision, n):
    import torch
    U, lo, hi = _case(system, n)
    kw = dict(system=system, order=order, precision=precision, bc=eno.PERIODIC)
    dt = 0.1 * (hi[0] - lo[0]) / n
    out = []
    for ts in (0, 8, 15, 63, 120, 255):  # 0: the default tile
        with eno.Solver((n,), lo, hi, **kw) as s:
            s.set_tiles(0, 1, ts)
            s.init_state(U)
            F, idx = s.reconstruct_fluxes(0, want_idx=True)
            for k in range(3):
                s.rk_stage(k, dt)
            out.append((F, idx, s.get_state()))
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
    # the allocation-free step takes tiles by the device's SMs
    a = torch.from_numpy(U).cuda()
    b = torch.empty_like(a)
    eno.step_noalloc(eno.make_config((n,), lo, hi, **kw), a, b, dt)
    assert np.array_equal(b.cpu().numpy(), out[0][2])


@pytest.mark.parametrize("system", [eno.EULER, eno.SCALAR_ADVECTION])
def test_persistent_runs_end_at_256_cells_an_sm(system):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n, persistent in ((15 * sms + 1, True), (256 * sms, True), (256 * sms + 1, False)):
        U, lo, hi = _case(system, n)
        with eno.Solver((n,), lo, hi, system=system, order=5, bc=eno.PERIODIC) as s:
            assert (s.launches_per_step() == 0) == persistent, n
            s.init_state(U)
            s.advance_steps(2, 0.5)
            dt, run = s.stats().dt, s.get_state()
            assert s.stats().steps == 2
            s.set_run_block_limit(1)
            s.init_state(U)
            s.advance_steps(2, 0.5)  # as graph replays
            assert s.launches_per_step() > 0
            assert s.stats().dt == dt and np.array_equal(s.get_state(), run), n
