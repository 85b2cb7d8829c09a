"""Long queued runs in place, which work on bit planes, against the oracle and against
the same gates issued in short runs (a flush after every three), bit for bit:
every kind of operation, fields at every offset and across key words, long
predicates, values in between, prunes, odd branch counts, one and two words."""
import numpy as np
import pytest

import oracle
from paper_2503_15118_gb300 import workloads as W
from tests.helpers import compare_states

pytestmark = pytest.mark.gpu

KINDS = ("x", "cx", "ccx", "phase", "cphase", "diag", "adiag", "add", "sub", "swap", "mulc")
VALUES = ("muladd", "divxor", "qram", "mulc")


@pytest.fixture(scope="module")
def sqs():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_15118_gb300 import sqs as S
    S.load()
    return S


def _gates(rng, widths, n, kinds, n_tables):
    qs = [(r, b) for r, w in enumerate(widths) for b in range(w)]
    out = []
    for _ in range(n):
        g = W._draw_gate(rng, kinds, qs, widths, n_tables)
        if rng.random() < 0.25 and g[0] in ("add", "sub", "swap", "mulc"):
            used = {g[1], g[2] if g[0] != "mulc" else g[1]}
            free = [q for q in qs if q[0] not in used]
            if free:  # a controlled arithmetic operation, value 0 or 1
                c = tuple(free[i] + (int(rng.integers(2)),)
                          for i in rng.choice(len(free), size=min(3, len(free)), replace=False))
                g = g[:-1] + (c,)
        if rng.random() < 0.1:  # a predicate over most of the key
            some = [q + (int(rng.integers(2)),) for q in qs[:: int(rng.integers(1, 4))]]
            g = ("phase", tuple(some), 0.31)
        out.append(g)
    return out


@pytest.mark.parametrize("amp32", [False, True])
@pytest.mark.parametrize("widths", [[7, 7, 3], [9, 14, 9], [20, 20, 24], [16, 16, 16, 16],
                                    [30, 5, 30], [31, 33, 31, 33], [64, 13, 13, 20]])
@pytest.mark.parametrize("values", [False, True])
@pytest.mark.parametrize("n", [3, 1003])
def test_long_runs(sqs, widths, amp32, values, n):
    rng = np.random.default_rng(sum(widths) + n)
    table = rng.integers(0, 2 ** 16, size=200).astype(np.uint16)
    kinds = KINDS + (VALUES if values else ())
    gates = _gates(rng, widths, 75, kinds, 1)
    # Diagonal matrices prune, which keeps a run from the planes: only in the
    # second half.
    gates = [g for g in gates[:40] if g[0] != "u1q"] + [("prune", 1e-13)] + gates[40:]
    gates = _gates(rng, widths, 70, tuple(k for k in kinds if "diag" not in k), 1) + gates
    lo, hi, a = W.random_state(widths, n, seed=n)
    if amp32:
        a = a.astype(np.complex64).astype(np.complex128)
    out = []
    for every in (0, 3):
        st = sqs.State(widths, amp32=amp32)
        st.import_(lo, hi, a)
        for i, g in enumerate(gates):
            st.apply(g, [table])
            if every and i % every == every - 1:
                st.flush()
        out.append(st.export())
    (l1, h1, a1), (l2, h2, a2) = out
    assert np.array_equal(l1, l2) and np.array_equal(h1, h2)
    # Phases of one launch are folded into one factor, so amplitudes differ by
    # the roundings of 145 factors at most.
    tol = 2 * 145 * (2.0 ** -24 if amp32 else 2.0 ** -53) * 2
    assert np.max(np.abs(a1 - a2) / np.abs(a2)) <= tol
    if not amp32:
        o = oracle.OracleState(widths, 1e-14)
        o.import_(lo, hi, a)
        for g in gates:
            o.apply(g, [table])
        assert compare_states({(int(h) << 64) | int(l): v for l, h, v in zip(l1, h1, a1)},
                              o.to_dict(), atol=1e-12) > 1 - 1e-12


@pytest.mark.parametrize("widths", [[10, 10], [22, 40, 22]])
def test_runs_inside_every_first_pass(sqs, widths):
    """The run ahead of a merge, an expansion, a fold and an addressed run."""
    rng = np.random.default_rng(8)
    body = lambda: _gates(rng, widths, 30, ("cx", "ccx", "phase", "add", "sub"), 0)  # noqa: E731
    gates = [("h", 0, b, ()) for b in range(9)] + body() + [("h", 1, 2, ())] + body()
    gates += [("ry", 0, 1, 0.4, ())] + body() + [("prune", 1e-15), ("h", 1, 9, ())]
    gates += [("phase", ((0, 0, 1),), 0.2), ("prune", 1e-15), ("h", 1, 9, ())] + body()
    gates += [("ry", 1, b, 0.3, ()) for b in range(4)] + body()
    circ = {"widths": widths, "eps": 1e-14, "tables": [], "gates": gates}
    got = sqs.State(widths).run(circ).to_dict()
    ref = oracle.run_circuit(circ).to_dict()
    assert set(got) == set(ref)
    assert compare_states(got, ref) > 1 - 1e-12
