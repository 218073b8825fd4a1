"""Tiles at the end of an SM's shared memory: scalar FP64 tiles whose planes alone
fill it are accepted and give the bits of the default tiles; larger ones are
refused."""
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


# (8 x 980 + halo = 7,912 cells of 24 B; 1 x 8192; 64 x 122 + halo = 8,512)
@pytest.mark.parametrize("shape,d,ta,ts", [((9001,), 0, 1, 8192), ((1001, 11), 0, 8, 980),
                                           ((1500, 11), 0, 8, 1000), ((70, 250), 1, 64, 122),
                                           ((40, 11, 270), 2, 32, 245)])
@pytest.mark.parametrize("order", [5, 7])
def test_scalar_fp64_tiles_that_fill_shared_memory(shape, d, ta, ts, order):
    nd = len(shape)
    full = (1,) + (1,) * (3 - nd) + tuple(reversed(shape))
    U = np.random.default_rng(1).uniform(-1, 1, full)
    out = []
    for tiles in (False, True):
        with eno.Solver(shape, (0.0,) * nd, (1.0,) * nd, system=eno.SCALAR_ADVECTION, order=order,
                        precision=eno.FP64, bc=eno.PERIODIC) as s:
            if tiles:
                s.set_tiles(d, ta, ts)
                assert s.get_tiles(d) == (ta, ts)
            s.init_state(U)
            F, idx = s.reconstruct_fluxes(d, want_idx=True)
            s.rk_stage(0, 1e-4)
            out.append((F, idx, s.get_stage_state(1)))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_tiles_past_shared_memory_are_refused():
    with eno.Solver((70, 250), (0.0, 0.0), (1.0, 1.0), system=eno.SCALAR_ADVECTION, order=7,
                    precision=eno.FP64) as s:
        for ta, ts in ((64, 128), (64, 129)):  # 213 KB of planes; 8,256 cells
            with pytest.raises(eno.EnoaoError) as e:
                s.set_tiles(1, ta, ts)
            assert e.value.status == 1
    with eno.Solver((70, 250), (0.0, 0.0), (1.0, 1.0), system=eno.EULER, order=5,
                    precision=eno.FP64) as s:
        with pytest.raises(eno.EnoaoError) as e:
            s.set_tiles(1, 64, 47)
        assert e.value.status == 1
