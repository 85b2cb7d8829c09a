"""Learned sizing queues interference steps; whatever needs the state as it stands comes
after them.  The states are small, so that every path is exact: bit for bit."""
import math

import pytest

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
