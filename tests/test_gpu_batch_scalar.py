"""Batched scalar problems, whose faces are selected without the proof in FP32 bulk, against
the same problems one at a time: the same bits, at lengths around the tile's."""
import numpy as np
import pytest

import paper_2108_12742_gb300 as eno

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2108_12742_gb300 import build
    build.build()


@pytest.mark.parametrize("order", [5, 7])
@pytest.mark.parametrize("precision", [eno.FP32_BULK, eno.FP64])
@pytest.mark.parametrize("bc", [eno.PERIODIC, eno.TRANSMISSIVE])
def test_scalar_batch_equals_single_problems(order, precision, bc):
    sizes = [11, 63, 245, 246, 247, 248, 249, 256, 497, 1000]
    rng = np.random.default_rng(order)
    kw = dict(system=eno.SCALAR_ADVECTION, order=order, precision=precision, bc=bc)
    parts = []
    for i, n in enumerate(sizes):  # noise, a sine and steps in turn
        x = (np.arange(n) + 0.5) / n
        parts.append([rng.uniform(-1, 1, n), np.sin(2 * np.pi * x), np.round(2 * x)][i % 3])
    with eno.Batch(sizes, 0.0, 1.0, **kw) as b:
        b.init_state(np.concatenate(parts)[None])
        b.advance_steps(4, 0.5)
        got = b.get_state()[0]
    at = np.concatenate([[0], np.cumsum(sizes)])
    for i, n in enumerate(sizes):
        with eno.Solver((n,), (0.0,), (1.0,), **kw) as s:
            s.init_state(parts[i].reshape(1, 1, 1, n))
            s.advance_steps(4, 0.5)
            assert np.array_equal(s.get_state().ravel(), got[at[i]:at[i + 1]]), n
