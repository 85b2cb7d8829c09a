"""The Python binding's own work, on the CPU: what State.run() looks up and refuses."""
import ctypes

import numpy as np
import pytest

from paper_2503_15118_gb300 import sqs as S


@pytest.fixture
def state():
    """A binding object without a device state behind it."""
    st = S.State.__new__(S.State)
    st.lib = S.load()
    st.h = None
    st.widths, st.kw, st._tables = [4, 4], 1, {}
    yield st
    st.h = None  # nothing to destroy


def test_a_closed_state_refuses_a_circuit_as_it_refuses_a_gate(state):
    circ = {"widths": [4, 4], "gates": [("h", 0, 0, ())]}
    with pytest.raises(S.SqsError) as one:
        state.apply(circ["gates"][0])
    with pytest.raises(S.SqsError) as run:
        state.run(circ)
    assert (run.value.status, str(run.value)) == (one.value.status, str(one.value))
    assert state.run({"widths": [4, 4], "gates": []}) is state


@pytest.mark.parametrize("tables_as", [list, tuple])
def test_tables_are_looked_up_once(state, monkeypatch, tables_as):
    """Gates that the native walker leaves to apply() (matrices, the first use of a
    table) do not look every table of the circuit up again."""
    if S._walk is None:
        pytest.skip("built without Python's headers")

    class Counted(dict):
        looked_up = 0

        def get(self, *a):
            self.looked_up += 1
            return dict.get(self, *a)

    state.h = ctypes.c_void_p(1)  # never dereferenced: nothing reaches the library
    state._tables = Counted()
    tables = tables_as([np.arange(4, dtype=np.uint8) for _ in range(40)])
    gates = [("u1q", 0, 0, np.eye(2), ())] * 60 + [("qload", 0, 1, i) for i in range(40)] * 2
    applied, seen = [], []

    class Walker:
        """Leaves matrices and tables it has no handle of."""

        def run(self, handle, gates, i, handles):
            while i < len(gates) and gates[i][0] == "qload" and handles[gates[i][3]] is not None:
                seen.append(handles[gates[i][3]])
                i += 1
            return i, S.OK

    def apply(self, g, tables=()):
        applied.append(g)
        if g[0] == "qload":
            self._tables[id(tables[g[3]])] = (ctypes.c_void_p(100 + g[3]), tables[g[3]])

    monkeypatch.setattr(S, "_walk", Walker())
    monkeypatch.setattr(S.State, "apply", apply)
    state.run({"widths": [4, 4], "tables": tables, "gates": gates})
    assert applied == gates[:100]                        # each table's first use only
    assert seen == [100 + i for i in range(40)]
    assert state._tables.looked_up <= 2 * len(tables)
