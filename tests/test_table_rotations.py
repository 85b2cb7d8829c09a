"""Rotations that read their QRAM table themselves, where something else reads or
writes what the load does.

Each circuit is compared, on every path that moves a load past a rotation, with the
operations one by one (SQS_MERGE_PLAIN), bit for bit, and with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2503_15118_gb300 import qlss
from tests.helpers import compare_states

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _check(sqs, widths, gates, tables, amp32):
    circ = {"widths": widths, "eps": 1e-14, "tables": tables, "gates": gates}

    def state(merge=0, learned=False):
        st = sqs.State(widths, amp32=amp32, eps=circ["eps"], merge=merge, learned=learned)
        if learned:
            st.set_predictor(sqs.Predictor(seed=1))
        return st.run(circ).to_dict()

    want = state(sqs.MERGE_PLAIN)
    if not amp32:
        ref = oracle.run_circuit(circ).to_dict()
        assert set(want) == set(ref)
        assert compare_states(want, ref, eps=circ["eps"], atol=1e-12) >= 1 - 1e-12
    for merge, learned in ((0, False), (sqs.FUSE_ALWAYS, False), (sqs.FUSE_OFF, False),
                           (sqs.MERGE_HASH, False), (sqs.MERGE_SORT, False), (0, True)):
        got = state(merge, learned)
        assert set(got) == set(want), (merge, learned)
        assert all(got[k] == want[k] for k in got), (merge, learned)


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("value", [0, 1])
@pytest.mark.parametrize("loaded", ["zero", "mixed"])
@pytest.mark.parametrize("before", ["nothing", "step", "x"])
def test_controls_on_the_loaded_register(sqs, amp32, value, loaded, before):
    """A rotation controlled on a bit of its own angle register sees the loaded
    bit: the register known zero before the load or in a superposition, the load
    right after a held step, after another operation, or first."""
    rng = np.random.default_rng(7)
    widths = [3, 3, 7, 2]  # address, target, angle, other
    table = rng.integers(0, 128, size=8).astype(np.uint8)
    assert 0 < int(((table >> 4) & 1).sum()) < 8
    gates = [("h", 0, b, ()) for b in range(3)]
    if loaded == "mixed":
        gates += [("h", 2, 4, ()), ("ry", 2, 1, 0.7, ())]
    gates += {"nothing": [], "step": [("ry", 1, 1, 0.3, ())], "x": [("x", 3, 0, ((0, 1, 1),))]}[before]
    gates += [("qload", 0, 2, 0), ("ry_reg", 1, 0, 2, qlss.ANGLE_SCALE * 2.0 ** 24, 0.1,
                                   ((2, 4, value),)),
              ("ry_reg", 1, 2, 2, 0.05, 0.0, ((2, 0, 1), (0, 1, value))), ("qunload", 0, 2, 0)]
    _check(sqs, widths, gates, [table], amp32)


WRITES = {
    "x": [("x", 0, 1, ())],
    "cx": [("x", 0, 0, ((3, 1, 1),))],
    "add": [("add", 0, -1, 3, ())],
    "sub": [("sub", 0, 3, 0, ())],
    "swap": [("swap", 0, 4, ())],
    "load": [("qload", 3, 0, 1)],
    "x_other": [("x", 4, 0, ()), ("x", 4, 3, ((3, 0, 1),))],
    "x_ignored": [("x", 0, 3, ())],
}


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("write", sorted(WRITES))
@pytest.mark.parametrize("ctrl", [(), ((4, 2, 1),)])
def test_folds_after_a_write_to_the_address(sqs, amp32, write, ctrl):
    """The target is copy-paired (a Hadamard on a constant bit), so that queued
    operations may wait until after the rotation; those that write its table's
    address may not.  (Address bit 3 is one that no entry depends on.)"""
    rng = np.random.default_rng(11)
    widths = [4, 3, 9, 3, 4]  # address, target, angle, other, other
    t = rng.integers(0, 512, size=8).astype(np.uint16)
    tables = [np.concatenate([t, t]), rng.integers(0, 16, size=8).astype(np.uint8)]
    gates = [("h", 0, b, ()) for b in range(2)] + [("h", 3, b, ()) for b in range(3)]
    gates += [("h", 4, 2, ()), ("ry", 4, 1, 0.4, ()), ("h", 1, 0, ())]
    gates += WRITES[write]
    gates += [("qload", 0, 2, 0), ("ry_reg", 1, 0, 2, 0.013, 0.2, ctrl), ("qunload", 0, 2, 0)]
    _check(sqs, widths, gates, tables, amp32)
