"""Learned sizing queues interference steps; whatever needs the state as it stands comes
after them.  The states are small, so that every path is exact: bit for bit."""
import math

import numpy as np
import pytest

from paper_2503_15118_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _states(sqs, widths):
    exact = sqs.State(widths, merge=sqs.MERGE_PLAIN)
    learned = sqs.State(widths, learned=True)
    learned.set_predictor(sqs.Predictor(seed=1))
    return exact, learned


@pytest.mark.parametrize("eps", [1e-14, 0.3])
@pytest.mark.parametrize("wait", [False, True])
def test_prune_after_queued_steps(sqs, eps, wait):
    """Operations queued after a step run after it, and the prune sees both."""
    got = []
    for st in _states(sqs, [3, 4]):
        st.h_gate(0, 0)
        st.ry(0, 1, 0.9, [(0, 0, 1)])
        st.x(1, 2, [(0, 1, 1)])
        n = st.prune(eps, wait=wait)
        st.ry(1, 2, 0.5)
        st.phase([(1, 2, 1)], math.pi / 2)
        m = st.prune(eps, wait=wait)
        got.append((n, m, st.to_dict(), st.peak_nnz()))
    assert got[0] == got[1]


@pytest.mark.parametrize("n_ops", [60, 97, 230])
def test_a_step_run_again_applies_its_operations_once(sqs, n_ops):
    """A predictor that promises a 256-fold shrink undersizes the second merge, which
    is run again at the exact size: also the operations ahead of it that did not fit
    its own launch (96 at most) and ran as passes in place before it."""
    widths = [20, 24]
    state = W.random_state(widths, 120000, seed=2, pair_fraction=0.3, target=(0, 3))
    got = []
    for st in _states(sqs, widths):
        bad = sqs.Predictor(seed=0)
        w = np.zeros(sqs.PRED_PARAMS, np.float32)
        w[-1] = -8.0
        bad.set_params(w)
        st.set_predictor(bad)
        st.import_(*state)
        st.ry(0, 3, 0.7)
        for i in range(n_ops):
            st.apply(("add", i & 1, -1, 3 * i + 1, ((1 - (i & 1), i % 20, 1),)))
        st.ry(0, 5, 0.4)
        for i in range(n_ops):
            st.apply(("sub", 1, -1, 5 * i + 1, ((0, i % 20, 0),)))
        st.ry(1, 7, 0.2)
        got.append((st.export(), st.peak_nnz(), st.stats()["overflow_reruns"]))
    (x, px, _), (y, py, reruns) = got
    assert reruns > 0
    assert all(np.array_equal(p, q) for p, q in zip(x, y)) and px == py
