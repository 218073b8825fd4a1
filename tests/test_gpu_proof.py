"""The shortcuts of the choice -- the proof that a face takes the top candidate,
the FP32 decision of FP64 choices, and lane groups for short face lists --
against the oracle, where they change over: data whose indicators straddle the
threshold, steep and silent stretches, and tiles whose lists are short or long."""
import numpy as np
import pytest

import oracle
import paper_2108_12742_gb300 as eno
from paper_2108_12742_gb300 import inputs

pytestmark = pytest.mark.gpu

TOL64, TIE, TOL32 = 1e-12, 1e-13, 1e-6  # as in the parity tests


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_12742_gb300 import build
    build.build()
    oracle.build()


SHAPES = {"adv1d": (97,), "adv2d": (33, 29), "euler1d": (301,), "euler2d": (70, 45),
          "euler3d": (19, 17, 23)}


def _data(name, amp, seed):
    """A uniform flow (a third of the domain exactly constant) with noise of size amp, a wave and
    a jump: indicators from zero over delta = 1e-5 to the jump's."""
    shape = SHAPES[name]
    rng = np.random.default_rng(seed)
    full = tuple(reversed(shape)) if len(shape) == 3 else (1,) * (3 - len(shape)) + tuple(reversed(shape))
    x = np.broadcast_to((np.arange(shape[0]) + 0.5) / shape[0], full)

    def field(base, jump):
        f = base + amp * rng.uniform(-1, 1, full) + 3 * amp * np.sin(9 * x)
        return np.where(x < 1 / 3, base, f) + jump * (x > 0.8)

    if name.startswith("adv"):
        return field(0.3, 0.5).reshape((1,) + full)
    vel = [field(v, 0.0) for v in (0.4, -0.2, 0.1)[:len(shape)]]
    return inputs.conserved(field(1.0, 0.4), vel, field(0.7, 0.3), 1.4).reshape((-1,) + full)


def _kw(name, order):
    return dict(system=eno.SCALAR_ADVECTION if name.startswith("adv") else eno.EULER, order=order,
                bc=eno.TRANSMISSIVE)


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("amp", [1e-8, 1e-6, 4e-6, 1e-4, 0.05])
def test_choices_and_fluxes_match_oracle(name, order, amp):
    shape = SHAPES[name]
    lo, hi = (0.0,) * len(shape), (1.0,) * len(shape)
    U = np.ascontiguousarray(_data(name, amp, seed=order))
    P = oracle.make_problem(shape, lo, hi, **_kw(name, order))
    for precision in (eno.FP64, eno.FP32_BULK):
        with eno.Solver(shape, lo, hi, precision=precision, **_kw(name, order)) as s:
            s.init_state(U)
            for d in range(len(shape)):
                F, idx = s.reconstruct_fluxes(d, want_idx=True)
                Fo, io, gap = oracle.fluxes(P, U, d, want_idx=True)
                differ = idx != io
                rel = np.abs(F - Fo) / np.abs(Fo).max()
                if precision == eno.FP64:
                    assert not (differ & (gap > TIE)).any(), (d, int(differ.sum()))
                    assert rel[:, ~differ.any(axis=(0, 1))].max() <= TOL64, d
                else:
                    assert 1 - differ.mean() >= 0.999, (d, int(differ.sum()))
                    assert rel.max() <= TOL32, (d, rel.max())


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
def test_short_and_long_lists_give_the_same_bits(order, precision):
    # tiles of 8 to 255 cells: their lists run from one round of lane groups to
    # several rounds of one face per lane
    U = np.ascontiguousarray(_data("euler1d", 4e-6, seed=3))
    outs = []
    for ts in (8, 15, 16, 31, 120, 255):
        with eno.Solver((301,), (0.0,), (1.0,), precision=precision, **_kw("euler1d", order)) as s:
            s.set_tiles(0, 1, ts)
            s.init_state(U)
            outs.append(s.reconstruct_fluxes(0, want_idx=True))
    for F, idx in outs[1:]:
        assert np.array_equal(F, outs[0][0]) and np.array_equal(idx, outs[0][1])


@pytest.mark.parametrize("delta", [0.0, 1e-40, 1e-3])
@pytest.mark.parametrize("precision", [eno.FP64, eno.FP32_BULK])
def test_other_thresholds_match_oracle(delta, precision):
    # a threshold of zero, one below FP32's normal range, and a coarse one
    U = np.ascontiguousarray(_data("euler2d", 4e-6, seed=11))
    shape = SHAPES["euler2d"]
    P = oracle.make_problem(shape, (0.0, 0.0), (1.0, 1.0), delta=delta, **_kw("euler2d", 5))
    with eno.Solver(shape, (0.0, 0.0), (1.0, 1.0), precision=precision, delta=delta,
                    **_kw("euler2d", 5)) as s:
        s.init_state(U)
        for d in range(2):
            F, idx = s.reconstruct_fluxes(d, want_idx=True)
            Fo, io, gap = oracle.fluxes(P, U, d, want_idx=True)
            differ = idx != io
            if precision == eno.FP64:
                assert not (differ & (gap > TIE)).any(), (d, int(differ.sum()))
            rel = np.abs(F - Fo) / np.abs(Fo).max()
            ok = ~differ.any(axis=(0, 1))
            assert rel[:, ok].max() <= (TOL64 if precision == eno.FP64 else TOL32), d
