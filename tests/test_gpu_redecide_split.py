"""How a tile's near-ties are split over the warps of its block does not show in the
results: tiles with one choice to re-decide up to hundreds, in launches of fewer
and of more tiles than SMs, give the same bits."""
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


def _data(shape, system):
    """Mirrored parabolas with noise (ties at every sixteenth cell along x) and, past the middle,
    cells that alternate between two states (ties everywhere)."""
    nd = len(shape)
    rng = np.random.default_rng(nd)
    full = tuple(reversed(shape + (1,) * (3 - nd)))
    x = np.arange(shape[0])
    seg, j = (x + 8) // 16, np.abs((x + 8) % 16 - 8)

    def field(curve):
        f = 1.0 + 0.002 * rng.uniform(-1, 1, full[:2] + (shape[0] // 16 + 2, 9))[..., seg, j] \
            + curve * j ** 2
        return np.where(x < shape[0] // 2, f, 1.0 + 0.1 * (x % 3 == 0))

    if system == eno.SCALAR_ADVECTION:
        return field(0.01).reshape((1,) + full)
    vel = [np.broadcast_to(v, full) for v in (3.7, -6.1, 2.9)[:nd]]
    return inputs.conserved(field(0.01), vel, field(0.008), 1.4).reshape((nd + 2,) + full)


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("system,shape,tiles", [
    (eno.EULER, (7001,), [((1, t),) for t in (8, 15, 46, 120, 1000)]),
    (eno.SCALAR_ADVECTION, (7001,), [((1, t),) for t in (15, 63, 255, 1000)]),
    (eno.EULER, (400, 60), [((1, 31), (8, 15)), ((4, 24), (16, 31)), ((4, 255), (64, 15))]),
    (eno.SCALAR_ADVECTION, (400, 60), [((1, 31), (8, 15)), ((4, 255), (64, 63))]),
    (eno.EULER, (60, 22, 31), [((1, 15),) + ((8, 8),) * 2, ((4, 63),) + ((32, 15),) * 2])])
@pytest.mark.parametrize("alpha_mode", [eno.ALPHA_PER_STEP, eno.ALPHA_PER_FIELD])
def test_split_of_re_decisions_keeps_the_bits(order, system, shape, tiles, alpha_mode):
    nd = len(shape)
    U = np.ascontiguousarray(_data(shape, system))
    out = []
    for tile in tiles:
        with eno.Solver(shape, (0.0,) * nd, (1.0,) * nd, system=system, order=order,
                        precision=eno.FP32_BULK, bc=eno.PERIODIC, alpha_mode=alpha_mode) as s:
            for d, t in enumerate(tile):
                s.set_tiles(d, *t)
            s.init_state(U)
            res = [s.reconstruct_fluxes(d, want_idx=True) for d in range(nd)]
            for k in range(3):
                s.rk_stage(k, 0.02 / max(shape))
            out.append([a for r in res for a in r] + [s.get_state()])
            assert s.stats().fp64_fallbacks > 0
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.array_equal(a, b)
