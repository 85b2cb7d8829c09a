"""The one-launch sort of small states (export, sparse marginals) against
numpy's order and against the pass-by-pass sort (forced by a digit width it
does not have), bit for bit, at the edges of its tiles and of its range."""
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


def _sizes():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    return [1, 31, 2047, 2048, 2049, 6000, 70001, sms * 2048 - 1, sms * 2048, sms * 2048 + 1]


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[20], [16, 16, 16, 16], [20, 32, 32]])
@pytest.mark.parametrize("i", range(10))
def test_export_of_a_loaded_state(sqs, widths, amp32, i):
    n = min(_sizes()[i], 1 << (sum(widths) - 1) if sum(widths) < 40 else 1 << 40)
    lo, hi, a = W.random_state(widths, n, seed=n % 97)
    if amp32:
        a = a.astype(np.complex64).astype(np.complex128)
    st = sqs.State(widths, amp32=amp32)
    st.import_(lo, hi, a)
    glo, ghi, ga = st.export()
    order = np.lexsort((lo, hi))
    assert np.array_equal(glo, lo[order]) and np.array_equal(ghi, hi[order])
    assert np.array_equal(ga, a[order])


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[9, 8], [16, 16, 16, 16], [20, 32, 32]])
@pytest.mark.parametrize("n", [1, 300, 2600, 40000, 150000])
def test_segmented_states(sqs, monkeypatch, widths, amp32, n):
    """After a bucket merge the state is segmented, most segments part full.
    Exports are compared with the pass-by-pass sort; sparse marginals with sums
    over the export (the storage order after a merge, and with it the order of
    a sum of m positive terms, is not fixed: each side is within m 2^-53 of it)."""
    n = min(n, 1 << (sum(widths) - 2) if sum(widths) < 40 else n)
    target = (len(widths) - 1, 3)
    state = W.random_state(widths, n, seed=5, pair_fraction=0.3 if n > 1 else 0.0, target=target)
    got = []
    for bits in (None, "10"):
        if bits:
            monkeypatch.setenv("SQS_SORT_BITS", bits)
        st = sqs.State(widths, amp32=amp32, merge=sqs.MERGE_HASH)
        st.import_(*state)
        st.ry(target[0], target[1], 0.83)
        lo, hi, a = st.export()
        got.append((lo, hi, a))
        p = a.real ** 2 + a.imag ** 2
        off = np.cumsum([0] + widths)
        for r, w in enumerate(widths):
            o = int(off[r])
            v = lo >> np.uint64(o) if o < 64 else hi >> np.uint64(o - 64)
            if o < 64 < o + w:
                v = v | (hi << np.uint64(64 - o))
            want, inv = np.unique(v & np.uint64((1 << w) - 1), return_inverse=True)
            values, probs, norm = st.probabilities_sparse(r)
            assert np.array_equal(values, want)
            np.testing.assert_allclose(probs, np.bincount(inv.reshape(-1), weights=p),
                                       rtol=2 * (lo.shape[0] + 3) * 2.0 ** -53)
    assert got[0][0].shape[0] >= n
    assert all(np.array_equal(x, y) for x, y in zip(*got))
