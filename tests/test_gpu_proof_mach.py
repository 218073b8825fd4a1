"""The FP32 proof of FP64 choices where the left eigenvectors lose most digits: fast
flows at low pressure, in which c^2 = (gamma - 1) (H - |v|^2 / 2) is a small
difference of large numbers.  Every choice is the oracle's.  (Fluxes are not compared:
the oracle back-projects them, which loses Mach^2 roundings of its own.)"""
import numpy as np
import pytest

import oracle
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
    oracle.build()


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("shape", [(301,), (70, 45), (19, 17, 23)])
@pytest.mark.parametrize("mach,amps", [(3.0, (1e-8, 1e-7, 3e-7, 1e-6)),
                                       (30.0, (1e-10, 1e-9, 1e-8, 1e-7)),
                                       (300.0, (1e-11, 1e-10, 1e-9))])
@pytest.mark.parametrize("pressure", [0.7, 1e-3])
def test_choices_at_high_mach_numbers_match_oracle(shape, order, mach, amps, pressure):
    # noise whose indicators run from far below the threshold to above it.  FP64 itself
    # loses |L| |f| / |L f|, about Mach^2, in the projection (the oracle projects fluxes):
    # decisions closer than that many roundings may go either way
    tie = 1e-13 * (1 + mach ** 2)
    # (L f of a shear field vanishes in uniform tangential flow, and the oracle's gap, which
    # is relative to it, says nothing there: at Mach 300 they are left out)
    fields = slice(None) if mach < 100 else [0, 1, len(shape) + 1]
    nd = len(shape)
    full = tuple(reversed(shape + (1,) * (3 - nd)))
    lo, hi = (0.0,) * nd, (1.0,) * nd
    kw = dict(system=eno.EULER, order=order, bc=eno.TRANSMISSIVE)
    P = oracle.make_problem(shape, lo, hi, **kw)
    speed = mach * np.sqrt(1.4 * pressure)
    for amp in amps:
        rng = np.random.default_rng(order)
        noise = lambda: 1.0 + amp * rng.uniform(-1, 1, full)  # noqa: E731
        vel = [speed * w * noise() for w in (1.0, -0.6, 0.3)[:nd]]
        U = inputs.conserved(noise(), vel, pressure * noise(), 1.4).reshape((nd + 2,) + full)
        U = np.ascontiguousarray(U)
        with eno.Solver(shape, lo, hi, precision=eno.FP64, **kw) as s:
            s.init_state(U)
            for d in range(nd):
                _, idx = s.reconstruct_fluxes(d, want_idx=True)
                _, io, gap = oracle.fluxes(P, U, d, want_idx=True)
                differ = idx != io
                assert not (differ & (gap > tie))[fields].any(), (amp, d, int(differ.sum()))
