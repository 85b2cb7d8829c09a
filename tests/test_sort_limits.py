"""The one-launch sort of small states at its limits: a grid barrier that runs out is an
error of the call, not a wrong order, and larger sorts ask for no scratch of its."""
import time

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


@pytest.mark.parametrize("segmented", [False, True])
@pytest.mark.parametrize("read", ["export", "sparse"])
def test_grid_barrier_runs_out_then_recovers(sqs, segmented, read):
    """CTA 1 of the sort's grid leaves out its arrivals (the testing hook of
    sqs_state_set_wait_test), so every CTA's wait reaches the short limit."""
    widths = [16, 16, 16, 16]
    state = W.random_state(widths, 5 * 2048 + 7, seed=3)
    st = sqs.State(widths, merge=sqs.MERGE_HASH)

    def load():
        st.import_(*state)
        if segmented:
            st.ry(3, 3, 0.83)
            st.flush()

    call = (lambda: st.export()) if read == "export" else (lambda: st.probabilities_sparse(1))
    load()
    want = call()
    load()
    st.sync()
    assert st.lib.sqs_state_set_wait_test(st.h, 64, 1) == sqs.OK
    t0 = time.perf_counter()
    with pytest.raises(sqs.SqsError) as err:
        call()
    assert err.value.status == sqs.ERR_TIMEOUT
    assert time.perf_counter() - t0 < 30.0
    with pytest.raises(sqs.SqsError):
        st.nnz()  # refused until reset
    assert st.lib.sqs_state_set_wait_test(st.h, 0, -1) == sqs.OK
    st.reset()
    load()
    got = call()
    if read == "export" and not segmented:
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
    assert np.array_equal(got[0], want[0])


def test_scratch_of_larger_sorts(sqs, monkeypatch):
    """A sort in passes needs 256 four-byte counters per tile of 2048 branches,
    and what does not grow with the state (under 128 KB with the bucket counters)."""
    n = (1 << 19) + 5
    asked = []
    given = sqs._TorchAllocator.alloc
    monkeypatch.setattr(sqs._TorchAllocator, "alloc",
                        lambda self, ctx, b, s: asked.append(b) or given(self, ctx, b, s))
    st = sqs.State([30, 30])
    lo, hi, a = W.random_state([30, 30], n, seed=9)
    st.import_(lo, hi, a)
    del asked[:]
    got = st.export()
    order = np.argsort(lo)
    assert np.array_equal(got[0], lo[order]) and np.array_equal(got[2], a[order])
    scratch = [b for b in asked if b < 8 * n]
    assert scratch and max(scratch) <= 1024 * ((n + 2047) // 2048) + (128 << 10)
