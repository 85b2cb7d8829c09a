"""The native gate-list walker issues what State.apply() would, and leaves the
rest to it: the same states, the same refusals at the same gate."""
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


KINDS = ("x", "cx", "ccx", "ry", "cry", "phase", "cphase", "h", "ch", "u1q", "cu1q", "diag",
         "adiag", "add", "sub", "swap", "qram", "muladd", "mulc", "divxor")


@pytest.mark.parametrize("widths", [[6, 5, 4, 4], [20, 31, 40, 20]])
@pytest.mark.parametrize("listed", [list, tuple])
def test_walked_and_applied_states_agree(sqs, widths, listed):
    if sqs._walk is None:
        pytest.skip("built without Python's headers")
    rng = np.random.default_rng(3)
    tables = [rng.integers(0, 32, size=40).astype(np.uint16)]
    c = W.random_circuit(widths, 130, seed=4, kinds=KINDS[:12] * (sum(widths) < 30) + KINDS[12:] +
                         ("cx", "ccx", "ry", "cphase"), tables=tables)
    gates = [("h", 0, b, ()) for b in range(4)] + c["gates"]
    # Forms only apply() takes: lists, numpy numbers, an integer angle, two-entry controls.
    gates += [["x", 0, 1, ()], ("h", 0, 1, [[1, 1, 1]]),
              ("ry", 1, 2, 1, ((0, 1),)), ("ry", 1, 1, np.float32(0.5), ()),
              ("qload", (0, 1), 1, 0), ("qunload", 0, 1, 0), ("prune", 0), ("prune", 1e-13)]
    circ = dict(c, gates=listed(gates), eps=1e-14)
    a = sqs.State(widths).run(circ)
    b = sqs.State(widths)
    for g in circ["gates"]:
        b.apply(g, tables)
    assert a.to_dict() == b.to_dict()
    assert a.peak_nnz() == b.peak_nnz()


@pytest.mark.parametrize("bad", [
    ("h", 9, 0, ()), ("h", 0, 0, ((0, 0, 1),)), ("x", 0, 1), ("nothing", 0), ("add", 0, 0, 0, ()),
    ("phase", ((0, 0, 1),), math.inf), ("phase", ((0, 0, 2),), 0.3), ("mulc", 0, 4, ()),
    ("x", 0, 0, tuple((1, b, 1) for b in range(9))), ("qload", 0, 1, 5), ("h", 0, "1", ()),
    ("ry", 0, 0, "x", ()), ("swap", 0, 1, None), ("prune", -1.0), ("h", 2 ** 40, 0, ())])
def test_refusals_are_the_same(sqs, bad):
    """The error, and the state left behind by the gates before it."""
    widths = [5, 12]
    tables = [np.arange(8, dtype=np.uint8)]
    good = [("h", 0, 0, ()), ("h", 0, 3, ()), ("x", 1, 2, ((0, 3, 1),))]
    circ = {"widths": widths, "tables": tables, "gates": good + [bad] + good}
    a, b = sqs.State(widths), sqs.State(widths)
    errors = []
    for st, go in ((a, lambda: a.run(circ)), (b, lambda: [b.apply(g, tables) for g in circ["gates"]])):
        try:
            go()
            errors.append(None)
        except Exception as e:
            errors.append((type(e), str(e)))
    assert errors[0] == errors[1]
    assert a.to_dict() == b.to_dict()


@pytest.mark.parametrize("n", [0, 1, 5000])
@pytest.mark.parametrize("widths", [[14, 3], [40, 40]])
def test_readouts_in_one_call(sqs, n, widths):
    """Sparse marginals and the split export, from no branch to many."""
    st = sqs.State(widths)
    lo, hi, a = W.random_state(widths, n, seed=2) if n else (np.zeros(0, np.uint64),) * 2 + (
        np.zeros(0, complex),)
    st.import_(lo, hi, a)
    x = st.export()
    order = np.lexsort((lo, hi))
    assert np.array_equal(x[0], lo[order]) and np.array_equal(x[1], hi[order])
    assert np.array_equal(x[2], a[order])
    assert all(v.flags["C_CONTIGUOUS"] and v.shape == (n,) for v in x)
    v, p, norm = st.probabilities_sparse(0)
    want = np.unique(lo & np.uint64((1 << widths[0]) - 1))
    assert np.array_equal(v, want) and p.shape == want.shape
    # At most n + 3 roundings of positive terms on either side.
    assert abs(p.sum() - norm) <= 4 * (n + 3) * 2.0 ** -53 * max(norm, 1e-300)
