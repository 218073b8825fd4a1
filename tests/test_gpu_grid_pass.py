"""The grid-wide re-decision pass against the in-sweep re-decisions: both end with
the FP64 choice of every near-tie, so one stage from one state agrees to FP32
rounding.  The pass re-derives the FP32 choice that the sweep made; derived with
other roundings, a tie within them gets its change twice or not at all, and the
cells beside the face are off by the difference of two candidates' values."""
import numpy as np
import pytest

import paper_2108_12742_gb300 as eno
from paper_2108_12742_gb300 import inputs

pytestmark = pytest.mark.gpu

# Either way a cell's increment is some ten FP32 operations (2^-24 each) on four
# terms of the size of the largest increment, on up to three axes: 120 x 2^-24 = 7e-6.
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_12742_gb300 import build
    build.build()


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("shape", [(200000,), (1024, 1024), (60, 60, 60)])
def test_grid_pass_ends_with_the_choices_of_the_sweep(shape, order):
    # white noise: among the choices of so many faces (33 million on the plane)
    # tens are ties to the last bits
    nd = len(shape)
    rng = np.random.default_rng(order)
    full = tuple(reversed(shape + (1,) * (3 - nd)))
    rho, p, *vel = (b + 0.3 * rng.uniform(-1, 1, full) for b in [1.0, 1.0] + [0.2] * nd)
    U = np.ascontiguousarray(inputs.conserved(rho, vel, p, 1.4).reshape((nd + 2,) + full))
    out = []
    for mode in (eno.REDECIDE_GRID, eno.REDECIDE_IN_SWEEP):
        with eno.Solver(shape, (0.0,) * nd, (1.0,) * nd, system=eno.EULER, order=order,
                        precision=eno.FP32_BULK, bc=eno.PERIODIC) as s:
            s.set_redecide(mode)
            s.init_state(U)
            s.rk_stage(0, 0.1 / max(shape))
            out.append(s.get_stage_state(1))
            assert s.stats().fp64_fallbacks > 0
    grid, sweep = out
    off = np.abs(grid - sweep).max(axis=0) / np.abs(sweep - U).max()
    assert off.max() <= TOL, (off.max(), int((off > TOL).sum()))


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("shape", [(320000,), (768, 768), (64, 48, 48)])
def test_grid_pass_on_ties_that_rounding_decides(shape, order):
    # parabolas with noise, each mirrored about its centre cell (every sixteenth along
    # x), in a uniform supersonic flow: on the windows centred there the candidates of
    # four cells to the left and right tie exactly, FP32 rounding alone makes the
    # sweep's choice, and the rounding of |v|^2 reaches the left eigenvectors
    nd = len(shape)
    rng = np.random.default_rng(order)
    full = tuple(reversed(shape + (1,) * (3 - nd)))
    x = np.arange(shape[0])
    seg, j = (x + 8) // 16 % (shape[0] // 16), np.abs((x + 8) % 16 - 8)

    def field(curve):
        return 1.0 + 0.002 * rng.uniform(-1, 1, full[:2] + (shape[0] // 16, 9))[..., seg, j] \
            + curve * j ** 2

    rho, p = field(0.01), field(0.008)
    vel = [np.broadcast_to(v, full) for v in (3.7, -6.1, 2.9)[:nd]]
    U = np.ascontiguousarray(inputs.conserved(rho, vel, p, 1.4).reshape((nd + 2,) + full))
    out = []
    for mode in (eno.REDECIDE_GRID, eno.REDECIDE_IN_SWEEP):
        with eno.Solver(shape, (0.0,) * nd, (1.0,) * nd, system=eno.EULER, order=order,
                        precision=eno.FP32_BULK, bc=eno.PERIODIC) as s:
            s.set_redecide(mode)
            s.init_state(U)
            s.rk_stage(0, 0.02 / max(shape))
            out.append(s.get_stage_state(1))
            assert s.stats().fp64_fallbacks > 1000
    grid, sweep = out
    off = np.abs(grid - sweep).max(axis=0) / np.abs(sweep - U).max()
    assert off.max() <= TOL, (off.max(), int((off > TOL).sum()))


@pytest.mark.parametrize("order", [5, 7])
def test_tiles_of_the_mode_do_not_show_and_callers_tiles_stay(order):
    shape = (800, 400)  # eight tiles an SM and more
    U = inputs.riemann2d(2, *shape)
    out = []
    for own in (None, ((2, 63), (16, 15))):
        with eno.Solver(shape, (-1.0, -1.0), (1.0, 1.0), system=eno.EULER, order=order,
                        precision=eno.FP32_BULK, bc=eno.TRANSMISSIVE) as s:
            before = [s.get_tiles(d) for d in range(2)]
            if own:
                for d, t in enumerate(own):
                    s.set_tiles(d, *t)
            s.set_redecide(eno.REDECIDE_GRID)
            if own:
                assert [s.get_tiles(d) for d in range(2)] == list(own)
            s.init_state(U)
            s.advance_steps(10, 0.5)
            out.append(s.get_state())
            s.set_redecide(eno.REDECIDE_IN_SWEEP)
            assert [s.get_tiles(d) for d in range(2)] == (list(own) if own else before)
    assert np.array_equal(*out)
